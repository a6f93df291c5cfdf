// pt_staged.cuh -- the push as one kernel per RK stage (the "staged" schedule).
//
// The resident push (k_push) keeps every particle in registers for all
// nsteps x 5 stages of a call; its one kernel carries the inverse map, the
// interpolation, the drag, the RK update, the exact face intersection, the
// walk and (optionally) the learned start, so that its register budget and
// instruction footprint are those of the largest path, and a warp in which one
// lane intersects faces stalls the other 31.  The staged schedule splits a
// stage into
//   k_stage_*   every live particle: start guess, inverse map, interpolation,
//               drag, RK update and the FP32 slab test; a particle whose stage
//               segment may touch a face (~0.5 % at the 64^3 workload) is
//               appended to a compacted list instead of being intersected;
//   k_track_*   the listed particles on full warps: tracking through the
//               faces (Secs. 3.2.3, 3.2.4, 2.4) and the walk that checks the new
//               owner (the missed-crossing repair of the resident push, run at
//               once instead of at the next stage's start); in FP32 mode the
//               segments that need an FP64 intersection go on to k_exact_f32;
// and, with the learned start, k_guess_mlp before k_stage_*.  Between stages
// the particle state goes through HBM in element-sorted order: k_gather
// copies it from the caller's arrays into library-owned structure-of-arrays
// buffers (coalesced in the visiting order), k_scatter copies it back.  Every
// arithmetic step is the resident push's own device code, in the same order.
#pragma once
#include "pt_kernels.cuh"
#include "pt_mlp_tc.cuh"

// Resident blocks of 128 per SM asked of k_stage_f32: 4 (128 registers) against
// 3 (168) and 5 (96, which spills): 20.24 / 20.66 / 21.41 ms for two steps of
// 4.2e6 particles with the learned start (NGeo 3, N 5), 4.37 / 4.56 / 4.72 ms at
// NGeo 4, N 6.
#ifndef PT_STAGE_MINB
#define PT_STAGE_MINB 4
#endif
namespace pt {

// list entry: position t in the sorted state; the high bit marks a stage end
// that needs only the walk (reference-space localisation without a wall)
constexpr unsigned kSettleOnly = 0x80000000u;

// Appends t (| flag) for every lane with want != 0; warp-collective (all 32
// lanes must call it).
__device__ __forceinline__ void list_append(unsigned* list, unsigned* count, int64_t t,
                                            unsigned want) {
  const unsigned m = __ballot_sync(0xffffffffu, want != 0u);
  if (!m) return;
  const int lane = threadIdx.x & 31;
  const int leader = __ffs(m) - 1;
  unsigned base = 0u;
  if (lane == leader) base = atomicAdd(count, (unsigned)__popc(m));
  base = __shfl_sync(0xffffffffu, base, leader);
  if (want)
    list[base + __popc(m & ((1u << lane) - 1u))] = (unsigned)t | (want == 2u ? kSettleOnly : 0u);
}

// Per-thread histogram of small counts: four 16-bit bins per word (a thread
// sees far fewer than 65536 particles per launch).
struct Hist8 {
  unsigned long long w[2] = {0ull, 0ull};
  __device__ __forceinline__ void add(int v) {
    const int b = v < 7 ? (v > 0 ? v : 0) : 7;
    w[b >> 2] += 1ull << (16 * (b & 3));
  }
  __device__ __forceinline__ void flush(unsigned long long* stats, int slot, int nbins) const {
    for (int b = 0; b < nbins; ++b)
      count_add(stats, slot + b, (w[b >> 2] >> (16 * (b & 3))) & 0xFFFFull);
  }
};

__device__ __forceinline__ void stage_counters(const StageArgs& a, const PushCounters& c) {
  count_add(a.stats, PT_C_STEPS, c.steps);
  count_add(a.stats, PT_C_IT32, c.it32);
  count_add(a.stats, PT_C_IT64, c.it64);
  count_add(a.stats, PT_C_CROSS, (unsigned long long)c.tc.cross);
  count_add(a.stats, PT_C_HITS, (unsigned long long)c.tc.hits);
  count_add(a.stats, PT_C_SLOW, (unsigned long long)c.tc.slow);
}

// ---------------------------------------------------------------------------
// FP32 mode: position as a double-float offset from the owner's centre
// ---------------------------------------------------------------------------

// Element data requested up front: the element's low coefficient parts and
// rho, rho u are read well after the owner is known, so one bulk prefetch per
// array, issued by the first lane of each run of equal owners in the warp,
// lets those misses overlap the FP32 iterations.
template <int G, int NP>
__device__ __forceinline__ void prefetch_element(const StageArgs& a, int e) {
  constexpr int CS = Mono<G>::CS, N3 = NP * NP * NP;
  const float* xl = a.m.monolo + (size_t)e * 3 * CS;
  const float* U = reinterpret_cast<const float*>(a.U) + (size_t)e * 5 * N3;
  // a bulk prefetch needs a 16-byte aligned start and size: element blocks are
  // 12 CS and 20 NP^3 bytes apart from aligned bases
  // (called by the warp's live lanes only)
  const int lane = threadIdx.x & 31;
  const unsigned live = __activemask();
  const int prev = __shfl_up_sync(live, e, 1);
  if (lane == 0 || !((live >> (lane - 1)) & 1u) || prev != e) {
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;\n" ::"l"(xl), "r"(12 * CS));
    if constexpr ((20 * N3) % 16 == 0)
      asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;\n" ::"l"(U), "r"(16 * N3));
  }
}

// The particle state one FP32 stage reads, loaded at once and before anything
// that depends on it (the status test included), so that its HBM latency is
// paid once per particle rather than once for the status and again for the
// rest.
struct StageIn {
  unsigned st;
  int e;
  float d;
  df xd[3];
  float v[3], kx[3], kv[3], g[3];
};

template <bool MLP>
__device__ __forceinline__ void stage_load(const StageArgs& a, int64_t t, StageIn& in) {
  const int64_t n = a.n;
  const float* vg = reinterpret_cast<const float*>(a.v);
  const float* kxg = reinterpret_cast<const float*>(a.kx);
  const float* kvg = reinterpret_cast<const float*>(a.kv);
  in.st = a.st[t];
  in.e = a.e[t];
  in.d = reinterpret_cast<const float*>(a.d)[t];
#pragma unroll
  for (int r = 0; r < 3; ++r) {
    in.xd[r] = df{a.xh[r * n + t], a.xl[r * n + t]};
    in.v[r] = vg[r * n + t];
    in.kx[r] = a.stage > 0 ? kxg[r * n + t] : 0.f;
    in.kv[r] = a.stage > 0 ? kvg[r * n + t] : 0.f;
    if constexpr (MLP) in.g[r] = a.guess[r * n + t];
  }
}

// Returns 0 (stage end committed), 1 (listed for exact tracking) or 2 (listed
// for the walk only).
// SM: Es points at the element's data (ElemSlot) in shared memory, or is null
// for an element that has no slot.
template <int G, int NP, bool MLP, bool SM = false>
__device__ __forceinline__ unsigned stage_one_f32(const StageArgs& a, int64_t t,
                                                  const StageIn& in, PushCounters& c, Hist8& h32,
                                                  Hist8& h64, const float* Es = nullptr) {
  constexpr int N3 = NP * NP * NP;
  const int64_t n = a.n;
  const int s = a.stage;
  unsigned st = in.st;
  if (st & PT_ST_FROZEN) return 0u;
  const int e = in.e;
  if constexpr (!MLP && !SM) prefetch_element<G, NP>(a, e);
  const float* Mh = a.m.mono + (size_t)e * 3 * Mono<G>::CS;
  const float* Ml = a.m.monolo + (size_t)e * 3 * Mono<G>::CS;
  const float* Ue = reinterpret_cast<const float*>(a.U) + (size_t)e * 5 * N3;
  const float* Ui = Ue;
  if constexpr (SM) {
    if (Es) {
      Mh = Es;
      Ml = Es + 3 * Mono<G>::CS;
      Ui = Es + 6 * Mono<G>::CS;
    }
  }
  float* vg = reinterpret_cast<float*>(a.v);
  float* kxg = reinterpret_cast<float*>(a.kx);
  float* kvg = reinterpret_cast<float*>(a.kv);
  const float d = in.d;
  df xd[3];
  float v[3], kx[3], kv[3];
#pragma unroll
  for (int r = 0; r < 3; ++r) {
    xd[r] = in.xd[r];
    v[r] = in.v[r];
    kx[r] = in.kx[r];
    kv[r] = in.kv[r];
  }
  const float tau = a.k.rho_p32 * d * d / (18.f * a.k.mu32);
  float xf[3] = {xd[0].hi, xd[1].hi, xd[2].hi};
  float guess[3];
  if constexpr (MLP) {
#pragma unroll
    for (int r = 0; r < 3; ++r) guess[r] = in.g[r];
  } else {
    trilinear_guess(a.m, e, xf, guess);
  }
  df zd[3];
  int i32 = 0, i64 = 0;
  float Ji[9];
  bool jok;
  const bool ok = newton_df<G, SM>(a.m, a.k, e, xd, guess, zd, i32, i64, Ji, jok, Mh, Ml);
  c.it32 += i32;
  c.it64 += i64;
  h32.add(i32);
  h64.add(i64);
  if (!ok) {
    a.st[t] = st | PT_ST_NEWTON_FAIL;
    return 0u;
  }
  const float xi[3] = {zd[0].hi + zd[0].lo, zd[1].hi + zd[1].lo, zd[2].hi + zd[2].lo};
  const float mx = tmax3(xi[0], xi[1], xi[2]);
  if (mx > 1.f - fmaxf(1e-5f, a.k.band_ref32)) {  // decide the bands exactly (rare)
    const double z[3] = {df_to_double(zd[0]), df_to_double(zd[1]), df_to_double(zd[2])};
    const double md = tmax3(z[0], z[1], z[2]);
    if (md > 1.0 + a.k.lost_tol) {  // outside: the walk after the last crossing ran already
      a.st[t] = st | PT_ST_LOST;
      return 0u;
    }
    if (md > 1.0 - a.k.band_ref) st |= near_bits(a.m, e, z, a.k.band_ref);
  }
  // interpolation of rho, rho u at xi, drag + gravity
  float l1[NP], l2[NP], l3[NP], Uv[4], acc[3];
  lagr<NP, float>(xi[0], a.k.sn32, a.k.sw32, l1);
  lagr<NP, float>(xi[1], a.k.sn32, a.k.sw32, l2);
  lagr<NP, float>(xi[2], a.k.sn32, a.k.sw32, l3);
  interp4<NP, SM>(Ui, l1, l2, l3, Uv);
  particle_accel_f32<G, NP>(a.m, a.k, Ue, e, zd, Uv, v, d, tau, st, acc);
  const float As = a.k.A32[s], Bs = a.k.B32[s], dt = a.dt32;
  df xe[3];
  float dx[3];
#pragma unroll
  for (int r = 0; r < 3; ++r) {
    kx[r] = As * kx[r] + dt * v[r];
    kv[r] = As * kv[r] + dt * acc[r];
    dx[r] = Bs * kx[r];
    xe[r] = df_add(xd[r], df_from(dx[r]));
    v[r] = v[r] + Bs * kv[r];
  }
  int touch = 0;
  if (!(jok && stays_inside(a.m, e, xi, Ji, dx, a.k.band_x32))) {
    const float bf[3] = {xe[0].hi, xe[1].hi, xe[2].hi};
    touch = slab_touch(a.m, e, xf, bf);
  }
  unsigned list = 0u;
  if (!(touch & (a.k.track == PT_TRACK_REFERENCE ? 2 : 1))) {
    // no face reachable, or (localisation) no wall or open face: with a touch
    // the end point's owner is checked by the walk
#pragma unroll
    for (int r = 0; r < 3; ++r) xd[r] = xe[r];
    if (touch) list = 2u;
  } else {
    float* xeg = reinterpret_cast<float*>(a.xe);
#pragma unroll
    for (int r = 0; r < 3; ++r) {
      xeg[r * n + t] = xe[r].hi;
      xeg[(3 + r) * n + t] = xe[r].lo;
    }
    list = 1u;
  }
#pragma unroll
  for (int r = 0; r < 3; ++r) {
    a.xh[r * n + t] = xd[r].hi;
    a.xl[r * n + t] = xd[r].lo;
    vg[r * n + t] = v[r];
    if (s < 4) {
      kxg[r * n + t] = kx[r];
      kvg[r * n + t] = kv[r];
    }
  }
  a.st[t] = st;
  if (s == 4 && !list) ++c.steps;
  return list;
}

template <int G, int NP, bool MLP>
__global__ void __launch_bounds__(128, PT_STAGE_MINB) k_stage_f32(const __grid_constant__ StageArgs a) {
  if (blockIdx.x == 0 && threadIdx.x == 0) *a.count_next = *a.count2_next = 0u;
  PushCounters c = {0, 0, 0, {0, 0, 0}};
  Hist8 h32, h64;
  const int64_t n = a.n;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  const int64_t nround = (n + stride - 1) / stride * stride;  // uniform trip count per warp
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < nround; t += stride) {
    StageIn in;
    if (t < n) stage_load<MLP>(a, t, in);
    const unsigned want = t < n ? stage_one_f32<G, NP, MLP>(a, t, in, c, h32, h64) : 0u;
    list_append(a.list, a.count, t, want);
  }
  stage_counters(a, c);
  h32.flush(a.stats, PT_C_H32, 8);
  h64.flush(a.stats, PT_C_H64, 8);
}

// Element slots: per warp two copies of an element's data in shared memory --
// map coefficients, high then low parts (3 CS floats each), and rho, rho u
// (4 NP^3) -- for the two owners most of the warp's 32 sorted particles share.
template <int G, int NP>
struct ElemSlot {
  static constexpr int F = 6 * Mono<G>::CS + 4 * NP * NP * NP;  // floats, a multiple of 4
  static constexpr int bytes = 4 * 2 * F * 4;                    // block of 4 warps
  // bulk copies need 16-byte aligned blocks of the state (even NP); four blocks
  // per SM must leave L1 some room
  static constexpr bool ok = NP % 2 == 0 && bytes <= 45056;
};

// bounded wait without reading a clock: a try may suspend the thread
__device__ __forceinline__ bool slot_wait(uint32_t mbar, uint32_t parity) {
#pragma unroll 1
  for (int k = 0; k < (1 << 20); ++k) {
    uint32_t done;
    asm volatile(
        "{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
        "selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(done)
        : "r"(mbar), "r"(parity)
        : "memory");
    if (done) return true;
  }
  return false;
}

// As k_stage_f32, with the element data of each warp's first two owners copied
// to shared memory by bulk copies as soon as the owners are known.  The stage is
// bound by load latency: through L1 every row of the coefficients and of the
// state that the warp touches first is a round trip to L2, some 30 in a row per
// particle; the copies make that one.  A lane whose owner has no slot (a third
// owner, a particle that has crossed since the binning) reads global memory
// through the same generic loads.  us per stage against k_stage_f32: 203 / 240
// (10^6 particles, 30 per element, NGeo 2, N 5), 964 / 1078 (4.2e6, 38 per
// element, NGeo 3, N 5, learned start), 73 / 86 (5e5, 36, NGeo 2, N 3).  With
// fewer particles per element a warp meets more owners than slots (NGeo 2, N 5:
// 425 / 520 at 37.5 per element, 306 / 295 at 18.8, 210 / 183 at 9.4; NGeo 3,
// N 3: 381 / 405, 259 / 231, 168 / 142): used from 24 per element on.
template <int G, int NP, bool MLP>
__global__ void __launch_bounds__(128, PT_STAGE_MINB) k_stage_sm_f32(const __grid_constant__ StageArgs a) {
  if (blockIdx.x == 0 && threadIdx.x == 0) *a.count_next = *a.count2_next = 0u;
  constexpr int CS = Mono<G>::CS, N3 = NP * NP * NP, F = ElemSlot<G, NP>::F;
  extern __shared__ __align__(128) float s_el[];
  __shared__ unsigned long long s_bar[4];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  float* slots = s_el + w * 2 * F;
  const uint32_t mb = smem_u32(s_bar + w);
  if (lane == 0) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(mb) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
  }
  __syncwarp();
  uint32_t phase = 0u;
  bool dead = false;  // a copy did not arrive in time: no more slots for this warp
  PushCounters c = {0, 0, 0, {0, 0, 0}};
  Hist8 h32, h64;
  const int64_t n = a.n;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  const int64_t nround = (n + stride - 1) / stride * stride;
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < nround; t += stride) {
    StageIn in;
    if (t < n) stage_load<MLP>(a, t, in);
    const int e0 = (t < n && !(in.st & PT_ST_FROZEN)) ? in.e : -1;
    // the first owner, and the first that differs from it
    const unsigned m0 = __ballot_sync(0xffffffffu, e0 >= 0);
    const int ea = __shfl_sync(0xffffffffu, e0, m0 ? __ffs(m0) - 1 : 0);
    const unsigned m1 = __ballot_sync(0xffffffffu, e0 >= 0 && e0 != ea);
    const int eb = __shfl_sync(0xffffffffu, e0, m1 ? __ffs(m1) - 1 : 0);
    const int ns = dead || !m0 ? 0 : (m1 ? 2 : 1);
    const float* Es = nullptr;
    if (ns) {
      fence_async_smem();  // the lanes' reads of the slots come before the copies
      __syncwarp();
      if (lane == 0)
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(mb),
                     "r"(ns * F * 4)
                     : "memory");
      __syncwarp();
      if (lane < 3 * ns) {
        const int q = lane >= 3, part = lane - 3 * q;
        const int e = q ? eb : ea;
        const float* src = part == 0   ? a.m.mono + (size_t)e * 3 * CS
                           : part == 1 ? a.m.monolo + (size_t)e * 3 * CS
                                       : reinterpret_cast<const float*>(a.U) + (size_t)e * 5 * N3;
        const float* dst = slots + q * F + 3 * CS * part;
        const uint32_t bytes = part < 2 ? 12 * CS : 16 * N3;
        asm volatile(
            "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, "
            "[%3];\n" ::"r"(smem_u32(dst)),
            "l"(src), "r"(bytes), "r"(mb)
            : "memory");
      }
      const bool done = slot_wait(mb, phase);
      if (__any_sync(0xffffffffu, !done)) {
        if (!slot_wait(mb, phase)) dead = true;
        dead = __any_sync(0xffffffffu, dead);
        if (dead && lane == 0) atomicAdd(a.stats + PT_C_TIMEOUT, 1ull);
      }
      phase ^= 1u;
      if (!dead && e0 >= 0) Es = e0 == ea ? slots : (e0 == eb ? slots + F : nullptr);
    }
    const unsigned want =
        t < n ? stage_one_f32<G, NP, MLP, true>(a, t, in, c, h32, h64, Es) : 0u;
    list_append(a.list, a.count, t, want);
  }
  stage_counters(a, c);
  h32.flush(a.stats, PT_C_H32, 8);
  h64.flush(a.stats, PT_C_H64, 8);
}

// The listed stage segments, first pass: tracking in reference space (track_f32)
// or the walk.  Segments that it does not decide (walls, open and mortar faces,
// ends and edges within the bands) go to a second list for k_exact_f32, so that
// no warp of this pass waits for an FP64 intersection.  Both passes are
// latency-bound (about a thousand segments per stage and 10^6 particles): 64
// threads per block spread them over the SMs.
template <int G>
__global__ void __launch_bounds__(64, 4) k_track_f32(const __grid_constant__ StageArgs a) {
  PushCounters c = {0, 0, 0, {0, 0, 0}};
  Hist8 hcr;
  const int64_t n = a.n;
  const unsigned cnt = *a.count;
  const float* xeg = reinterpret_cast<const float*>(a.xe);
  const unsigned stride = gridDim.x * blockDim.x;
  const unsigned cround = (cnt + 31u) & ~31u;  // whole warps
  if (((blockIdx.x * blockDim.x + threadIdx.x) & ~31u) >= cround) return;
  for (unsigned j = blockIdx.x * blockDim.x + threadIdx.x; j < cround; j += stride) {
    unsigned exact = 0u, t32 = 0u;
    if (j < cnt) {
      const unsigned ent = a.list[j];
      t32 = ent & ~kSettleOnly;
      const int64_t t = t32;
      int e = a.e[t];
      const int e0 = e;
      df xd[3];
#pragma unroll
      for (int r = 0; r < 3; ++r) xd[r] = df{a.xh[r * n + t], a.xl[r * n + t]};
      int cr = 0, j32 = 0, j64 = 0, rc = 0;
      if (!(ent & kSettleOnly)) {
        df xe[3];
#pragma unroll
        for (int r = 0; r < 3; ++r) xe[r] = df{xeg[r * n + t], xeg[(3 + r) * n + t]};
        const int cr0 = c.tc.cross;
        unsigned bits = 0u;
        exact = track_f32<G>(a.m, a.k, e, xd, xe, bits, j32, j64, c.tc) ? 0u : 1u;
        if (!exact) hcr.add(c.tc.cross - cr0);
        if (bits) a.st[t] |= bits;
      } else {
        df zd[3];
        float Ji[9];
        bool jok;
        rc = settle_f32<G>(a.m, a.k, e, xd, zd, false, j32, j64, cr, Ji, jok);
      }
      c.it32 += j32;
      c.it64 += j64;
      if (!exact) {
        c.tc.cross += cr;
#pragma unroll
        for (int r = 0; r < 3; ++r) {
          a.xh[r * n + t] = xd[r].hi;
          a.xl[r * n + t] = xd[r].lo;
        }
        if (e != e0) a.e[t] = e;
        if (rc)
          a.st[t] |= rc == 1 ? PT_ST_NEWTON_FAIL : PT_ST_LOST;
        else if (a.stage == 4)
          ++c.steps;
      }
    }
    list_append(a.list2, a.count2, t32, exact);
  }
  stage_counters(a, c);
  hcr.flush(a.stats, PT_C_HCR, 4);
}

// Second pass: the FP64 intersection of the segments the first pass left, on
// global positions, back to the double-float offset, and the walk.  One FP64
// instruction holds an SM's FP64 unit for the same time whether one lane or 32
// are active and these lanes rarely agree on a path, so the entries are spread
// over all warps of the grid, one per warp while there are that few.
template <int G, bool CLIP>
__global__ void __launch_bounds__(32) k_exact_f32(const __grid_constant__ StageArgs a) {
  PushCounters c = {0, 0, 0, {0, 0, 0}};
  Hist8 hcr;
  const int64_t n = a.n;
  const int s = a.stage;
  const unsigned cnt = *a.count2;
  if (blockIdx.x >= cnt) return;
  float* vg = reinterpret_cast<float*>(a.v);
  float* kxg = reinterpret_cast<float*>(a.kx);
  float* kvg = reinterpret_cast<float*>(a.kv);
  const float* xeg = reinterpret_cast<const float*>(a.xe);
  const unsigned stride = gridDim.x * blockDim.x;
  // entry j of warp w is w + j gridDim
  for (unsigned j = blockIdx.x + gridDim.x * threadIdx.x; j < cnt; j += stride) {
    const int64_t t = a.list2[j];
    unsigned st = a.st[t];
    int e = a.e[t], hits = a.hits[t];
    df xd[3];
    float v[3], kx[3], kv[3];
    double xs[3], xg[3];
    const double* ce = a.m.ce + 3 * (size_t)e;
#pragma unroll
    for (int r = 0; r < 3; ++r) {
      xd[r] = df{a.xh[r * n + t], a.xl[r * n + t]};
      v[r] = vg[r * n + t];
      kx[r] = kxg[r * n + t];  // stale at the last stage of a step: not used after it
      kv[r] = kvg[r * n + t];
      const double cr = __ldg(ce + r);
      xs[r] = cr + df_to_double(xd[r]);
      xg[r] = cr + df_to_double(df{xeg[r * n + t], xeg[(3 + r) * n + t]});
    }
    const int cr0 = c.tc.cross;
    track_slow<G, float, CLIP>(a.m, a.k, e, xs, xg, v, kx, kv, hits, st, c.tc);
    hcr.add(c.tc.cross - cr0);
    const double* cn = a.m.ce + 3 * (size_t)e;
#pragma unroll
    for (int r = 0; r < 3; ++r) xd[r] = df_from_double(xs[r] - __ldg(cn + r));
    if (!(st & PT_ST_FROZEN)) {
      df zd[3];
      float Ji[9];
      bool jok;
      int cr = 0, j32 = 0, j64 = 0;
      const int rc = settle_f32<G>(a.m, a.k, e, xd, zd, false, j32, j64, cr, Ji, jok);
      c.it32 += j32;
      c.it64 += j64;
      c.tc.cross += cr;
      if (rc) st |= rc == 1 ? PT_ST_NEWTON_FAIL : PT_ST_LOST;
    }
#pragma unroll
    for (int r = 0; r < 3; ++r) {
      a.xh[r * n + t] = xd[r].hi;
      a.xl[r * n + t] = xd[r].lo;
      vg[r * n + t] = v[r];
      if (s < 4) {
        kxg[r * n + t] = kx[r];
        kvg[r * n + t] = kv[r];
      }
    }
    a.e[t] = e;
    a.hits[t] = hits;
    a.st[t] = st;
    if (s == 4 && !(st & PT_ST_FROZEN)) ++c.steps;
  }
  __syncwarp();
  stage_counters(a, c);
  hcr.flush(a.stats, PT_C_HCR, 4);
}

// Position of particle t relative to its owner's centre, in FP32: from the
// sorted state (the high part of the double-float offset), or (FROM_X) from
// global FP64 positions a.x.
template <bool FROM_X>
__device__ __forceinline__ void start_pos(const StageArgs& a, int64_t t, int e, float* xf) {
  const int64_t n = a.n;
  if constexpr (FROM_X) {
    const double* ce = a.m.ce + 3 * (size_t)e;
#pragma unroll
    for (int r = 0; r < 3; ++r) xf[r] = (float)(a.x[r * n + t] - __ldg(ce + r));
  } else {
#pragma unroll
    for (int r = 0; r < 3; ++r) xf[r] = a.xh[r * n + t];
  }
}

// Learned start of every live particle at the current position, warp-level
// mma.sync form (the network is warp-collective: every lane takes part, dead
// lanes with live = false).
template <int G, bool FROM_X>
__global__ void __launch_bounds__(128) k_guess_mlp(const __grid_constant__ StageArgs a) {
  PT_MLP_PROLOGUE(true, a.mlp);
  const int64_t n = a.n;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  const int64_t nround = (n + stride - 1) / stride * stride;
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < nround; t += stride) {
    const bool inr = t < n;
    // (a.st is null for pt_mlp_start: every particle with an owner in range)
    const unsigned st = inr ? (a.st ? a.st[t] : 0u) : (unsigned)PT_ST_FROZEN;
    const int e0 = inr ? a.e[t] : 0;
    const bool live = !(st & PT_ST_FROZEN) && e0 >= 0 && e0 < a.m.nelem;
    const int e = live ? e0 : 0;
    float xf[3] = {0.f, 0.f, 0.f};
    if (live) start_pos<FROM_X>(a, t, e, xf);
    float guess[3];
    start_guess_local<G, true>(a.m, a.k, sm, &a.mlp, e, xf, live, guess);
    if (live) {
#pragma unroll
      for (int r = 0; r < 3; ++r) a.guess[r * n + t] = guess[r];
    }
  }
}

// Learned start of every live particle on the tensor cores (tcgen05): one
// tile of 128 particles at a time per CTA, weights in shared memory,
// accumulators in 128 columns of tensor memory.  An MMA that does not complete
// within the wait limit counts in PT_C_TIMEOUT and ends the CTA's work.
template <int G, bool FROM_X>
__global__ void __launch_bounds__(128, 1) k_guess_tc(const __grid_constant__ StageArgs a) {
  extern __shared__ __align__(1024) unsigned char dsm[];
  MlpTcSmem& s = *reinterpret_cast<MlpTcSmem*>(dsm + ((1024u - (smem_u32(dsm) & 1023u)) & 1023u));
  const int tid = threadIdx.x;
  mlp_tc_load(s, a.mlp);
  if (tid == 0) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(smem_u32(&s.mbar)) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
  }
  if (tid < 32) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(
                     smem_u32(&s.tmem)),
                 "r"(kMlpTcCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
  }
  fence_async_smem();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = s.tmem;
  uint32_t phase = 0u;
  const int64_t n = a.n;
  // the status, owner and (staged state) offset of a row, read one tile ahead
  // so that their HBM latency overlaps the previous tile's network
  auto row_in = [&](int64_t t, unsigned& st, int& e0, float* xo) {
    const bool inr = t < n;
    // (a.st is null for pt_mlp_start: every particle with an owner in range)
    st = inr ? (a.st ? a.st[t] : 0u) : (unsigned)PT_ST_FROZEN;
    e0 = inr ? a.e[t] : 0;
    if constexpr (!FROM_X) {
#pragma unroll
      for (int r = 0; r < 3; ++r) xo[r] = inr ? a.xh[r * n + t] : 0.f;
    }
  };
  const int64_t tstride = (int64_t)gridDim.x * 128;
  unsigned st_nx;
  int e_nx;
  float x_nx[3] = {0.f, 0.f, 0.f};
  row_in((int64_t)blockIdx.x * 128 + tid, st_nx, e_nx, x_nx);
  for (int64_t base = (int64_t)blockIdx.x * 128; base < n; base += tstride) {
    const int64_t t = base + tid;
    const unsigned st = st_nx;
    const int e0 = e_nx;
    float xc[3] = {x_nx[0], x_nx[1], x_nx[2]};
    if (base + tstride < n) row_in(t + tstride, st_nx, e_nx, x_nx);
    const bool live = !(st & PT_ST_FROZEN) && e0 >= 0 && e0 < a.m.nelem;
    const int e = live ? e0 : 0;
    float xf[3] = {0.f, 0.f, 0.f}, xi_tri[3], guess[3];
    if constexpr (FROM_X) {
      if (live) start_pos<FROM_X>(a, t, e, xf);
    } else {
#pragma unroll
      for (int r = 0; r < 3; ++r) xf[r] = live ? xc[r] : 0.f;
    }
    trilinear_guess(a.m, e, xf, xi_tri);
    if (!mlp_tc_tile(s, a.mlp, a.m, tmem, e, xi_tri, guess, phase)) {
      if (tid == 0) atomicAdd(a.stats + PT_C_TIMEOUT, 1ull);
      break;
    }
    if (live) {
#pragma unroll
      for (int r = 0; r < 3; ++r) a.guess[r * n + t] = guess[r];
    }
  }
  tc_fence_before();
  __syncthreads();
  if (tid < 32) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem),
                 "r"(kMlpTcCols)
                 : "memory");
  }
}

// ---------------------------------------------------------------------------
// FP64 mode: global FP64 positions
// ---------------------------------------------------------------------------

template <int G, int NP>
__device__ __forceinline__ unsigned stage_one_f64(const StageArgs& a, int64_t t,
                                                  PushCounters& c, Hist8& h64) {
  constexpr int N3 = NP * NP * NP;
  const int64_t n = a.n;
  const int s = a.stage;
  unsigned st = a.st[t];
  if (st & PT_ST_FROZEN) return 0u;
  const int e = a.e[t];
  double* vg = reinterpret_cast<double*>(a.v);
  double* kxg = reinterpret_cast<double*>(a.kx);
  double* kvg = reinterpret_cast<double*>(a.kv);
  const double d = reinterpret_cast<const double*>(a.d)[t];
  double x[3], v[3], kx[3] = {0, 0, 0}, kv[3] = {0, 0, 0};
#pragma unroll
  for (int r = 0; r < 3; ++r) {
    x[r] = a.x[r * n + t];
    v[r] = vg[r * n + t];
    if (s > 0) {
      kx[r] = kxg[r * n + t];
      kv[r] = kvg[r * n + t];
    }
  }
  const double tau = a.k.rho_p * d * d / (18.0 * a.k.mu);
  const double* ce = a.m.ce + 3 * (size_t)e;
  double xl[3] = {x[0] - __ldg(ce), x[1] - __ldg(ce + 1), x[2] - __ldg(ce + 2)};
  const float xf[3] = {(float)xl[0], (float)xl[1], (float)xl[2]};
  float guess[3];
  trilinear_guess(a.m, e, xf, guess);
  double xi[3];
  int i64 = 0;
  const bool ok = newton_f64<G>(a.m, a.k, e, xl, guess, xi, i64);
  c.it64 += i64;
  h64.add(i64);
  if (!ok) {
    a.st[t] = st | PT_ST_NEWTON_FAIL;
    return 0u;
  }
  const double mx = tmax3(xi[0], xi[1], xi[2]);
  if (mx > 1.0 + a.k.lost_tol) {
    a.st[t] = st | PT_ST_LOST;
    return 0u;
  }
  if (mx > 1.0 - a.k.band_ref) st |= near_bits(a.m, e, xi, a.k.band_ref);
  const double* Ue = reinterpret_cast<const double*>(a.U) + (size_t)e * 5 * N3;
  double l1[NP], l2[NP], l3[NP], Uv[4], acc[3];
  lagr<NP, double>(xi[0], a.k.sn, a.k.sw, l1);
  lagr<NP, double>(xi[1], a.k.sn, a.k.sw, l2);
  lagr<NP, double>(xi[2], a.k.sn, a.k.sw, l3);
  interp4<NP>(Ue, l1, l2, l3, Uv);
  particle_accel<G, NP, double>(a.m, a.k, Ue, e, xi, Uv, v, d, tau, st, acc);
  const double As = a.k.A[s], Bs = a.k.B[s], dt = a.dt;
  double xe[3];
  float bf[3];
#pragma unroll
  for (int r = 0; r < 3; ++r) {
    kx[r] = As * kx[r] + dt * v[r];
    kv[r] = As * kv[r] + dt * acc[r];
    const double dx = Bs * kx[r];
    xe[r] = x[r] + dx;
    bf[r] = (float)(xl[r] + dx);
    v[r] = v[r] + Bs * kv[r];
  }
  const int touch = slab_touch(a.m, e, xf, bf);
  unsigned list = 0u;
  if (!(touch & (a.k.track == PT_TRACK_REFERENCE ? 2 : 1))) {
#pragma unroll
    for (int r = 0; r < 3; ++r) x[r] = xe[r];
    if (touch) list = 2u;
  } else {
    double* xeg = reinterpret_cast<double*>(a.xe);
#pragma unroll
    for (int r = 0; r < 3; ++r) xeg[r * n + t] = xe[r];
    list = 1u;
  }
#pragma unroll
  for (int r = 0; r < 3; ++r) {
    a.x[r * n + t] = x[r];
    vg[r * n + t] = v[r];
    if (s < 4) {
      kxg[r * n + t] = kx[r];
      kvg[r * n + t] = kv[r];
    }
  }
  a.st[t] = st;
  if (s == 4 && !list) ++c.steps;
  return list;
}

template <int G, int NP>
__global__ void __launch_bounds__(128, PT_PUSH_MINB_F64) k_stage_f64(const __grid_constant__ StageArgs a) {
  if (blockIdx.x == 0 && threadIdx.x == 0) *a.count_next = *a.count2_next = 0u;
  PushCounters c = {0, 0, 0, {0, 0, 0}};
  Hist8 h64;
  const int64_t n = a.n;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  const int64_t nround = (n + stride - 1) / stride * stride;
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < nround; t += stride) {
    const unsigned want = t < n ? stage_one_f64<G, NP>(a, t, c, h64) : 0u;
    list_append(a.list, a.count, t, want);
  }
  stage_counters(a, c);
  h64.flush(a.stats, PT_C_H64, 8);
}

template <int G, bool CLIP>
__global__ void __launch_bounds__(128) k_track_f64(const __grid_constant__ StageArgs a) {
  PushCounters c = {0, 0, 0, {0, 0, 0}};
  Hist8 hcr;
  const int64_t n = a.n;
  const int s = a.stage;
  const unsigned cnt = *a.count;
  double* vg = reinterpret_cast<double*>(a.v);
  double* kxg = reinterpret_cast<double*>(a.kx);
  double* kvg = reinterpret_cast<double*>(a.kv);
  const double* xeg = reinterpret_cast<const double*>(a.xe);
  const unsigned stride = gridDim.x * blockDim.x;
  const unsigned cround = (cnt + stride - 1) / stride * stride;
  for (unsigned j = blockIdx.x * blockDim.x + threadIdx.x; j < cround; j += stride) {
    if (j >= cnt) continue;
    const unsigned ent = a.list[j];
    const int64_t t = ent & ~kSettleOnly;
    unsigned st = a.st[t];
    int e = a.e[t], hits = a.hits[t];
    double x[3], v[3], kx[3], kv[3];
#pragma unroll
    for (int r = 0; r < 3; ++r) {
      x[r] = a.x[r * n + t];
      v[r] = vg[r * n + t];
      kx[r] = kxg[r * n + t];  // stale at the last stage of a step: not used after it
      kv[r] = kvg[r * n + t];
    }
    if (!(ent & kSettleOnly)) {
      double xe[3] = {xeg[t], xeg[n + t], xeg[2 * n + t]};
      const int cr0 = c.tc.cross;
      track_slow<G, double, CLIP>(a.m, a.k, e, x, xe, v, kx, kv, hits, st, c.tc);
      hcr.add(c.tc.cross - cr0);
    }
    if (!(st & PT_ST_FROZEN)) {
      double xi[3];
      int cr = 0, j64 = 0;
      const int rc = settle64<G>(a.m, a.k, e, x, xi, false, j64, cr);
      c.it64 += j64;
      c.tc.cross += cr;
      if (rc) st |= rc == 1 ? PT_ST_NEWTON_FAIL : PT_ST_LOST;
    }
#pragma unroll
    for (int r = 0; r < 3; ++r) {
      a.x[r * n + t] = x[r];
      vg[r * n + t] = v[r];
      if (s < 4) {
        kxg[r * n + t] = kx[r];
        kvg[r * n + t] = kv[r];
      }
    }
    a.e[t] = e;
    a.hits[t] = hits;
    a.st[t] = st;
    if (s == 4 && !(st & PT_ST_FROZEN)) ++c.steps;
  }
  stage_counters(a, c);
  hcr.flush(a.stats, PT_C_HCR, 4);
}

// ---------------------------------------------------------------------------
// the caller's arrays <-> the sorted state
// ---------------------------------------------------------------------------

// sorted[t] = caller[perm[t]]; an owner out of range freezes a live particle
// (PT_ST_LOST), as in the resident push
template <bool F64>
__global__ void __launch_bounds__(256) k_gather(const __grid_constant__ StageArgs a,
                                                const DevParticles p, const int* __restrict__ perm) {
  using R = typename RealOf<F64>::type;
  const int64_t n = a.n;
  const R* vc = reinterpret_cast<const R*>(p.v);
  const R* dc = reinterpret_cast<const R*>(p.d);
  R* vs = reinterpret_cast<R*>(a.v);
  R* ds = reinterpret_cast<R*>(const_cast<void*>(a.d));
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < n;
       t += (int64_t)gridDim.x * blockDim.x) {
    const int64_t ip = perm[t];
    unsigned st = p.status[ip];
    const int e = p.elem[ip];
    const bool valid = e >= 0 && e < a.m.nelem;
    if (!valid && !(st & PT_ST_FROZEN)) st |= PT_ST_LOST;
    const double* ce = a.m.ce + 3 * (size_t)(valid ? e : 0);
#pragma unroll
    for (int r = 0; r < 3; ++r) {
      const double xr = p.x[r * n + ip];
      if constexpr (F64) {
        a.x[r * n + t] = xr;
      } else {
        const df o = df_from_double(valid ? xr - __ldg(ce + r) : 0.0);
        a.xh[r * n + t] = o.hi;
        a.xl[r * n + t] = o.lo;
      }
      vs[r * n + t] = vc[r * n + ip];
    }
    ds[t] = dc[ip];
    a.e[t] = e;
    a.hits[t] = p.hits[ip];
    a.st[t] = st;
  }
}

// caller[perm[t]] = sorted[t] for every particle that was not frozen on entry
// (a particle whose owner was out of range keeps its position and velocity)
template <bool F64>
__global__ void __launch_bounds__(256) k_scatter_back(const __grid_constant__ StageArgs a,
                                                      DevParticles p, const int* __restrict__ perm) {
  using R = typename RealOf<F64>::type;
  const int64_t n = a.n;
  R* vc = reinterpret_cast<R*>(p.v);
  const R* vs = reinterpret_cast<const R*>(a.v);
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < n;
       t += (int64_t)gridDim.x * blockDim.x) {
    const int64_t ip = perm[t];
    if (p.status[ip] & PT_ST_FROZEN) continue;
    const int e = a.e[t];
    p.status[ip] = a.st[t];
    if (e < 0 || e >= a.m.nelem) continue;
    const double* ce = a.m.ce + 3 * (size_t)e;
#pragma unroll
    for (int r = 0; r < 3; ++r) {
      if constexpr (F64)
        p.x[r * n + ip] = a.x[r * n + t];
      else
        p.x[r * n + ip] = __ldg(ce + r) + df_to_double(df{a.xh[r * n + t], a.xl[r * n + t]});
      vc[r * n + ip] = vs[r * n + t];
    }
    p.elem[ip] = e;
    p.hits[ip] = a.hits[t];
  }
}

}  // namespace pt
