// pt_device.cuh -- device building blocks of the particle push (arXiv 2211.05458):
// Lagrange bases, the inverse map x -> xi (Sec. 3.2.1), interpolation of the
// nodal state (Eq. part_interpolation), drag (Sec. 2.2) and the physical-
// space tracking with face intersection (Secs. 3.2.3, 3.2.4) and the specular
// wall model (Sec. 2.4).  Everything is templated on the number of geometry
// nodes G = NGeo+1 and solution nodes NP = N+1 so loops unroll into registers.
#pragma once
#include <cuda_runtime.h>

#include <cstdint>
#include <type_traits>

#include "pt_df.cuh"
#include "pt_internal.h"
#include "pt_map.cuh"

// FP32 Newton iterations of the FP32 mode stop once the step is below this;
// the final iterations (double-float residuals, last FP32 inverse Jacobian)
// take over and converge linearly with a factor of about the step at which
// that Jacobian was evaluated
#ifndef PT_NEWTON_SWITCH
#define PT_NEWTON_SWITCH 1e-5f
#endif
// 1: screen each touched face in FP32 before its exact FP64 solve
#ifndef PT_FACE_SCREEN
#define PT_FACE_SCREEN 1
#endif
namespace pt {

template <typename T>
__device__ __forceinline__ T tabs(T a) {
  return a < T(0) ? -a : a;
}

template <typename T>
__device__ __forceinline__ T tmax3(T a, T b, T c) {
  return fmax(fmax(tabs(a), tabs(b)), tabs(c));
}

template <typename T>
__device__ __forceinline__ T tfma(T a, T b, T c);
template <>
__device__ __forceinline__ float tfma<float>(float a, float b, float c) {
  return fmaf(a, b, c);
}
template <>
__device__ __forceinline__ double tfma<double>(double a, double b, double c) {
  return fma(a, b, c);
}

// node set of the right precision from the constants
template <typename T>
struct Nodes;
template <>
struct Nodes<float> {
  __device__ static const float* geo(const DevConsts& k) { return k.gn32; }
  __device__ static const float* geow(const DevConsts& k) { return k.gw32; }
  __device__ static const float* sol(const DevConsts& k) { return k.sn32; }
  __device__ static const float* solw(const DevConsts& k) { return k.sw32; }
};
template <>
struct Nodes<double> {
  __device__ static const double* geo(const DevConsts& k) { return k.gn; }
  __device__ static const double* geow(const DevConsts& k) { return k.gw; }
  __device__ static const double* sol(const DevConsts& k) { return k.sn; }
  __device__ static const double* solw(const DevConsts& k) { return k.sw; }
};

// physical constants of the right precision (a conversion from FP64 inside a
// kernel would hold an SM's FP64 unit for 64 cycles per warp)
template <typename T>
struct Phys;
template <>
struct Phys<float> {
  __device__ static float mu(const DevConsts& k) { return k.mu32; }
  __device__ static float rho_p(const DevConsts& k) { return k.rho_p32; }
  __device__ static const float* g(const DevConsts& k) { return k.g32; }
  __device__ static const float* mask(const DevConsts& k) { return k.mask32; }
  __device__ static const float* hl(const DevConsts& k) { return k.hl32; }
};
template <>
struct Phys<double> {
  __device__ static double mu(const DevConsts& k) { return k.mu; }
  __device__ static double rho_p(const DevConsts& k) { return k.rho_p; }
  __device__ static const double* g(const DevConsts& k) { return k.g; }
  __device__ static const double* mask(const DevConsts& k) { return k.mask; }
  __device__ static const double* hl(const DevConsts& k) { return k.hl; }
};

// Lagrange basis in barycentric product form: l_i(x) = w_i prod_{m != i} (x - x_m),
// w_i = 1 / prod_{m != i} (x_i - x_m).  Prefix and suffix products avoid the
// division of the second barycentric form, so the values at the nodes are exact.
template <int NP, typename T>
__device__ __forceinline__ void lagr(T x, const T* nodes, const T* w, T* l) {
  T d[NP];
#pragma unroll
  for (int m = 0; m < NP; ++m) d[m] = x - nodes[m];
  T pre = T(1);
#pragma unroll
  for (int i = 0; i < NP; ++i) {
    l[i] = pre;
    pre *= d[i];
  }
  T suf = T(1);
#pragma unroll
  for (int i = NP - 1; i >= 0; --i) {
    l[i] *= suf * w[i];
    suf *= d[i];
  }
}

// values and first derivatives (dual-number prefix / suffix products)
template <int NP, typename T>
__device__ __forceinline__ void lagr_d(T x, const T* nodes, const T* w, T* l, T* dl) {
  T d[NP], P[NP], dP[NP];
#pragma unroll
  for (int m = 0; m < NP; ++m) d[m] = x - nodes[m];
  T p = T(1), dp = T(0);
#pragma unroll
  for (int i = 0; i < NP; ++i) {
    P[i] = p;
    dP[i] = dp;
    dp = tfma(dp, d[i], p);
    p *= d[i];
  }
  T s = T(1), ds = T(0);
#pragma unroll
  for (int i = NP - 1; i >= 0; --i) {
    l[i] = w[i] * P[i] * s;
    dl[i] = w[i] * tfma(dP[i], s, P[i] * ds);
    ds = tfma(ds, d[i], s);
    s *= d[i];
  }
}

template <typename T>
__device__ __forceinline__ bool inv3(const T* J, T* Ji) {
  T c00 = J[4] * J[8] - J[5] * J[7];
  T c01 = J[5] * J[6] - J[3] * J[8];
  T c02 = J[3] * J[7] - J[4] * J[6];
  T det = J[0] * c00 + J[1] * c01 + J[2] * c02;
  if (!(tabs(det) > T(0))) return false;
  T id = T(1) / det;
  Ji[0] = c00 * id;
  Ji[1] = (J[2] * J[7] - J[1] * J[8]) * id;
  Ji[2] = (J[1] * J[5] - J[2] * J[4]) * id;
  Ji[3] = c01 * id;
  Ji[4] = (J[0] * J[8] - J[2] * J[6]) * id;
  Ji[5] = (J[2] * J[3] - J[0] * J[5]) * id;
  Ji[6] = c02 * id;
  Ji[7] = (J[1] * J[6] - J[0] * J[7]) * id;
  Ji[8] = (J[0] * J[4] - J[1] * J[3]) * id;
  return true;
}

template <typename T>
__device__ __forceinline__ void matvec3(const T* M, const T* v, T* o) {
#pragma unroll
  for (int r = 0; r < 3; ++r) o[r] = M[3 * r] * v[0] + M[3 * r + 1] * v[1] + M[3 * r + 2] * v[2];
}

// ---------------------------------------------------------------------------
// element map chi(xi) = sum_abc X_abc l_a(xi1) l_b(xi2) l_c(xi3) and its inverse
// (FP32 evaluation: pt_map.cuh)
// ---------------------------------------------------------------------------

// trilinear start xi0 = Jc^{-1} (x_loc - xc), from the per-element table
__device__ __forceinline__ void trilinear_guess(const DevMesh& m, int e, const float* xf,
                                                float* xi) {
  const float* t = m.tri + 12 * (size_t)e;
  float r[3] = {xf[0] - __ldg(t), xf[1] - __ldg(t + 1), xf[2] - __ldg(t + 2)};
#pragma unroll
  for (int q = 0; q < 3; ++q)
    xi[q] = __ldg(t + 3 + 3 * q) * r[0] + __ldg(t + 4 + 3 * q) * r[1] + __ldg(t + 5 + 3 * q) * r[2];
}

// FP64: chi and, with WJ, the Jacobian J[r][q] from the FP64 monomial
// coefficients M [3][G^3] (row (b, c) at G (c + G b), powers of xi1 in order), by
// Horner's rule in xi3, xi2 and xi1
template <int G, bool WJ>
__device__ __forceinline__ void map64(const double* __restrict__ M, const double* xi, double* chi,
                                      double* J) {
  constexpr int G3 = G * G * G;
#pragma unroll
  for (int r = 0; r < 3; ++r) {
    const double* Mr = M + r * G3;
    double W[G], Wy[G], Wz[G];
#pragma unroll
    for (int b = G - 1; b >= 0; --b) {
#pragma unroll
      for (int a = 0; a < G; ++a) {
        double V = __ldg(Mr + G * (G - 1 + G * b) + a), D = 0.0;
#pragma unroll
        for (int c = G - 2; c >= 0; --c) {
          if (WJ) D = c == G - 2 ? V : fma(D, xi[2], V);
          V = fma(V, xi[2], __ldg(Mr + G * (c + G * b) + a));
        }
        if (b == G - 1) {
          W[a] = V;
          if (WJ) Wz[a] = D;
        } else {
          if (WJ) {
            Wy[a] = b == G - 2 ? W[a] : fma(Wy[a], xi[1], W[a]);
            Wz[a] = fma(Wz[a], xi[1], D);
          }
          W[a] = fma(W[a], xi[1], V);
        }
      }
    }
    double v = W[G - 1], dx = 0.0, dy = 0.0, dz = 0.0;
    if (WJ) {
      dy = Wy[G - 1];
      dz = Wz[G - 1];
    }
#pragma unroll
    for (int a = G - 2; a >= 0; --a) {
      if (WJ) {
        dx = a == G - 2 ? v : fma(dx, xi[0], v);
        dy = fma(dy, xi[0], Wy[a]);
        dz = fma(dz, xi[0], Wz[a]);
      }
      v = fma(v, xi[0], W[a]);
    }
    chi[r] = v;
    if (WJ) {
      J[3 * r] = dx;
      J[3 * r + 1] = dy;
      J[3 * r + 2] = dz;
    }
  }
}

// Full FP64 Newton: chi(xi) - x = 0, |dxi|_inf < tol (Sec. 3.2.1).
template <int G>
__device__ __forceinline__ bool newton64(const double* M, const double* xl, double* xi,
                                         const DevConsts& k, int maxit, int& it64) {
  #pragma unroll 1
  for (int it = 0; it < maxit; ++it) {
    double chi[3], J[9], Ji[9], r[3], d[3];
    map64<G, true>(M, xi, chi, J);
    if (!inv3(J, Ji)) return false;
#pragma unroll
    for (int q = 0; q < 3; ++q) r[q] = chi[q] - xl[q];
    matvec3(Ji, r, d);
#pragma unroll
    for (int q = 0; q < 3; ++q) xi[q] -= d[q];
    ++it64;
    double md = tmax3(d[0], d[1], d[2]);
    if (md < k.newton_tol) return true;
    if (!(tmax3(xi[0], xi[1], xi[2]) <= 4.0)) return false;
  }
  return false;
}

template <int G>
__device__ __noinline__ bool newton64_cold(const double* M, const double* xl, double* xi,
                                           const DevConsts& k, int maxit, int& it64) {
  return newton64<G>(M, xl, xi, k, maxit, it64);
}

// The inverse map of the FP64 mode.  An FP64 instruction holds an SM's FP64
// unit for 64 cycles per warp, so only what the result's accuracy needs runs in
// FP64: the start is improved by FP32 Newton iterations (to ~1e-7); one full
// FP64 Newton step squares that, and the steps after it (one, as a rule, to
// confirm |dxi| < tol) evaluate the FP64 residual alone and keep the FP64
// inverse Jacobian of that step, whose relative error is the step's size.  The
// fixed point is the FP64 residual's zero, as with full Newton steps, which
// took 3 to 4 evaluations of the FP64 map and Jacobian from the trilinear start.
// Where the FP32 iterations do not settle in six, or the FP64 steps leave the
// range, meet a singular Jacobian or take more than four, full Newton steps run
// from the start that was given: whatever they converge from is found.
template <int G>
__device__ __forceinline__ bool newton_f64(const DevMesh& m, const DevConsts& k, int e,
                                           const double* xl, const float* guess, double* xi,
                                           int& it64) {
  const double* M = m.mono64 + (size_t)e * 3 * G * G * G;
  bool settled = false;
  {
    const float* Mh = m.mono + (size_t)e * 3 * Mono<G>::CS;
    const int tm = G == 2 ? 7 : __ldg(m.tmask + e);
    const float xf[3] = {(float)xl[0], (float)xl[1], (float)xl[2]};
    float z[3] = {guess[0], guess[1], guess[2]};
#pragma unroll 1
    for (int it = 0; it < 6; ++it) {
      float chi[3], J[9], Ji[9], r[3], d[3];
      map_j32<G>(Mh, z, tm, chi, J);
      if (!inv3(J, Ji)) break;
#pragma unroll
      for (int q = 0; q < 3; ++q) r[q] = chi[q] - xf[q];
      matvec3(Ji, r, d);
#pragma unroll
      for (int q = 0; q < 3; ++q) z[q] -= d[q];
      if (!(tmax3(z[0], z[1], z[2]) <= 4.f)) break;
      settled = tmax3(d[0], d[1], d[2]) < PT_NEWTON_SWITCH;
      if (settled) break;
    }
#pragma unroll
    for (int q = 0; q < 3; ++q) xi[q] = z[q];
  }
  double chi[3], J[9], Ji[9], r[3], d[3];
  if (settled) {
    map64<G, true>(M, xi, chi, J);
    settled = inv3(J, Ji);
  }
  if (settled) {
    const int maxit = k.max_newton < 4 ? k.max_newton : 4;
    int it = 0;
#pragma unroll 1
    while (true) {
#pragma unroll
      for (int q = 0; q < 3; ++q) r[q] = chi[q] - xl[q];
      matvec3(Ji, r, d);
#pragma unroll
      for (int q = 0; q < 3; ++q) xi[q] -= d[q];
      ++it64;
      if (tmax3(d[0], d[1], d[2]) < k.newton_tol) return true;
      if (!(tmax3(xi[0], xi[1], xi[2]) <= 4.0) || ++it >= maxit) break;
      map64<G, false>(M, xi, chi, nullptr);
    }
  }
#pragma unroll
  for (int q = 0; q < 3; ++q) xi[q] = guess[q];
  return newton64_cold<G>(M, xl, xi, k, k.max_newton, it64);
}

// Mixed-precision Newton on a double-float local position xd (relative to the
// element centre): FP32 iterations (chi and J in FP32) until the step is below
// 1e-5 (after eight of them 1e-3 will do: in thin elements rounding keeps it above
// 1e-5; sixteen that do not get there count as failed), then double-float residuals with the last FP32 inverse Jacobian until
// the step is below newton_tol.  Returns the double-float xi in zd and, unless
// the (out-of-line) fallback of a full FP64 Newton was taken (jok false), the
// inverse Jacobian of a point within about 1e-3 of xi (1e-5 as a rule) in Ji.
// GEN: the element's coefficients (high, low parts) may be in shared memory,
// at Mh and Ml.
template <int G, bool GEN = false>
__device__ __forceinline__ bool newton_df(const DevMesh& m, const DevConsts& k, int e,
                                          const df* xd, const float* guess, df* zd, int& it32,
                                          int& it64, float* Ji, bool& jok,
                                          const float* Mh = nullptr, const float* Ml = nullptr) {
  if constexpr (!GEN) {
    Mh = m.mono + (size_t)e * 3 * Mono<G>::CS;
    Ml = m.monolo + (size_t)e * 3 * Mono<G>::CS;
  }
  const int tm = G == 2 ? 7 : __ldg(m.tmask + e);
  float z[3] = {guess[0], guess[1], guess[2]};
  bool have = false;
  jok = true;
  #pragma unroll 1
  for (int it = 0;; ++it) {
    float chi[3], J[9], r[3], d[3];
    map_j32<G, GEN>(Mh, z, tm, chi, J);
    if (!inv3(J, Ji)) break;
    have = true;
#pragma unroll
    for (int q = 0; q < 3; ++q) r[q] = chi[q] - xd[q].hi;
    matvec3(Ji, r, d);
#pragma unroll
    for (int q = 0; q < 3; ++q) z[q] -= d[q];
    ++it32;
    if (!(tmax3(z[0], z[1], z[2]) <= 4.f)) {
      have = false;
      break;
    }
    if (tmax3(d[0], d[1], d[2]) < (it < 7 ? PT_NEWTON_SWITCH : 1e-3f)) break;
    if (it == 15) {
      have = false;
      break;
    }
  }
  if (have) {
#pragma unroll
    for (int q = 0; q < 3; ++q) zd[q] = df_from(z[q]);
    const float tol = k.newton_tol32;
    // Each step needs the residual at the current iterate.  The first is the
    // double-float residual at the FP32 iterate z.  After a first step d with
    // |d| <= 4e-7 the next residual is r(z) + [chi(z - d) - chi(z)], and the
    // bracket is -J(z - d/2) d up to terms of third order in d: FP32 gives it
    // to ~1e-7 of a term of size |J d|, far below the tolerance.  Later
    // residuals are double-float again, at the iterate's high part plus J
    // times its low part.
    float rp[3] = {0.f, 0.f, 0.f}, dz[3] = {0.f, 0.f, 0.f};
    bool inc = false;
#pragma unroll 1
    for (int it = 0; it < 6; ++it) {
      float r[3], d[3], zm[3];
#pragma unroll
      for (int q = 0; q < 3; ++q) zm[q] = inc ? fmaf(0.5f, dz[q], z[q]) : zd[q].hi;
      if (!inc) resid_df<G, GEN>(Mh, Ml, zm, tm, xd, rp);
#pragma unroll
      for (int q = 0; q < 3; ++q) r[q] = rp[q];
      if (it > 0) {
        float chi[3], J[9], Jd[3];
        const float by[3] = {inc ? dz[0] : zd[0].lo, inc ? dz[1] : zd[1].lo,
                             inc ? dz[2] : zd[2].lo};
        map_j32<G, GEN>(Mh, zm, tm, chi, J);
        matvec3(J, by, Jd);
#pragma unroll
        for (int q = 0; q < 3; ++q) r[q] += Jd[q];
      }
      matvec3(Ji, r, d);
#pragma unroll
      for (int q = 0; q < 3; ++q) zd[q] = df_sub(zd[q], df_from(d[q]));
      ++it64;
      const float md = tmax3(d[0], d[1], d[2]);
      if (md < tol) return true;
      inc = it == 0 && md <= 4e-7f;
#pragma unroll
      for (int q = 0; q < 3; ++q) {
        rp[q] = r[q];
        dz[q] = -d[q];
      }
    }
  }
  // fallback: full FP64 Newton
  jok = false;
  double xl[3], xi[3];
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    xl[q] = df_to_double(xd[q]);
    xi[q] = have ? df_to_double(zd[q]) : (double)guess[q];
  }
  if (!(tmax3(xi[0], xi[1], xi[2]) <= 4.0)) xi[0] = xi[1] = xi[2] = 0.0;
  const bool ok = newton64_cold<G>(m.mono64 + (size_t)e * 3 * G * G * G, xl, xi, k, k.max_newton, it64);
#pragma unroll
  for (int q = 0; q < 3; ++q) zd[q] = df_from_double(xi[q]);
  return ok;
}

template <int G>
__device__ __forceinline__ bool newton_df(const DevMesh& m, const DevConsts& k, int e,
                                          const df* xd, const float* guess, df* zd, int& it32,
                                          int& it64) {
  float Ji[9];
  bool jok;
  return newton_df<G>(m, k, e, xd, guess, zd, it32, it64, Ji, jok);
}

// As newton_df for a local position in FP64 (xl) and a FP64 result.
template <int G>
__device__ __forceinline__ bool newton_mixed(const DevMesh& m, const DevConsts& k, int e,
                                             const double* xl, const float* guess, double* xi,
                                             int& it32, int& it64) {
  df xd[3], zd[3];
#pragma unroll
  for (int q = 0; q < 3; ++q) xd[q] = df_from_double(xl[q]);
  const bool ok = newton_df<G>(m, k, e, xd, guess, zd, it32, it64);
#pragma unroll
  for (int q = 0; q < 3; ++q) xi[q] = df_to_double(zd[q]);
  return ok;
}

// ---------------------------------------------------------------------------
// interpolation of rho and rho u (Eq. part_interpolation), sum-factorised
// ---------------------------------------------------------------------------

// FP32, sum-factorised, the sum over a row in packed pairs (its even and odd
// nodes, joined at the end).  NP = 6 takes two variables per pass: twice the
// loads in flight, which is what the staged push is short of (weights of a whole
// plane in registers save another 150 instructions per particle, but leave
// room for fewer loads: 312 against 235 us per stage of 10^6 particles).  The
// third-direction basis is shifted through registers by the rolled loop, which
// keeps it out of local memory.
template <int NP, bool GEN = false>
__device__ __forceinline__ void interp4(const float* __restrict__ Ue, const float* l1,
                                        const float* l2, const float* l3, float* out) {
  constexpr int N2 = NP * NP, N3 = N2 * NP, NH = NP / 2;
  if constexpr (NP % 2 == 0) {
    constexpr int VB = NP == 6 ? 2 : 1;  // variables per pass
    f32x2 w1[NH];
#pragma unroll
    for (int i = 0; i < NH; ++i) w1[i] = pk2(l1[2 * i], l1[2 * i + 1]);
    float lk[NP], res[4];
#pragma unroll
    for (int c = 0; c < NP; ++c) lk[c] = l3[c];
#pragma unroll
    for (int v = 0; v < 4; ++v) res[v] = 0.f;
#pragma unroll 1
    for (int v = 0; v < 4; v += VB) {
      f32x2 acc[VB];
#pragma unroll
      for (int q = 0; q < VB; ++q) acc[q] = dup2(0.f);
#pragma unroll 1
      for (int kk = 0; kk < NP; ++kk) {
        const f32x2 lz = dup2(lk[0]);
        {  // rotate: after NP iterations the basis is in place again
          const float l0 = lk[0];
#pragma unroll
          for (int c = 0; c + 1 < NP; ++c) lk[c] = lk[c + 1];
          lk[NP - 1] = l0;
        }
        f32x2 u[VB][N2 / 2];
#pragma unroll
        for (int q = 0; q < VB; ++q) {
          const ulonglong2* P =
              reinterpret_cast<const ulonglong2*>(Ue + (v + q) * N3 + kk * N2);
#pragma unroll
          for (int i = 0; i < N2 / 4; ++i) {
            const ulonglong2 x = ldx<GEN>(P + i);
            u[q][2 * i] = x.x;
            u[q][2 * i + 1] = x.y;
          }
        }
#pragma unroll
        for (int q = 0; q < VB; ++q) {
          f32x2 t;
#pragma unroll
          for (int j = 0; j < NP; ++j) {
            f32x2 t1 = mul2(u[q][j * NH], w1[0]);
#pragma unroll
            for (int i = 1; i < NH; ++i) t1 = fma2(u[q][j * NH + i], w1[i], t1);
            t = j ? fma2(t1, dup2(l2[j]), t) : mul2(t1, dup2(l2[0]));
          }
          acc[q] = fma2(t, lz, acc[q]);
        }
      }
      // the results move up the registers (v is a run-time index)
#pragma unroll
      for (int q = 0; q + VB < 4; ++q) res[q] = res[q + VB];
#pragma unroll
      for (int q = 0; q < VB; ++q) {
        float x, y;
        unpk2(acc[q], x, y);
        res[4 - VB + q] = x + y;
      }
    }
#pragma unroll
    for (int v = 0; v < 4; ++v) out[v] = res[v];
  } else {
    float lk[NP], res[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int c = 0; c < NP; ++c) lk[c] = l3[c];
    f32x2 w2[NP];
#pragma unroll
    for (int j = 0; j < NP; ++j) w2[j] = dup2(l2[j]);
    // single values are read (rows of odd length have no alignment): two
    // variables per packed operation instead
#pragma unroll 1
    for (int v = 0; v < 4; v += 2) {
      f32x2 acc = dup2(0.f);
#pragma unroll 1
      for (int kk = 0; kk < NP; ++kk) {
        const f32x2 lz = dup2(lk[0]);
        {
          const float l0 = lk[0];
#pragma unroll
          for (int c = 0; c + 1 < NP; ++c) lk[c] = lk[c + 1];
          lk[NP - 1] = l0;
        }
        const float* P = Ue + v * N3 + kk * N2;
        f32x2 t;
#pragma unroll
        for (int j = 0; j < NP; ++j) {
          f32x2 t1;
#pragma unroll
          for (int i = 0; i < NP; ++i) {
            const f32x2 x = pk2(ldx<GEN>(P + j * NP + i), ldx<GEN>(P + N3 + j * NP + i));
            t1 = i ? fma2(x, dup2(l1[i]), t1) : mul2(x, dup2(l1[0]));
          }
          t = j ? fma2(t1, w2[j], t) : mul2(t1, w2[0]);
        }
        acc = fma2(t, lz, acc);
      }
      res[0] = res[2];
      res[1] = res[3];
      unpk2(acc, res[2], res[3]);
    }
#pragma unroll
    for (int v = 0; v < 4; ++v) out[v] = res[v];
  }
}

// FP64 (bound by the FP64 unit): up to N = 5 the weights l1_i l2_j of a plane are
// formed once for the four variables, a tenth fewer multiply-adds than the sum-
// factorised form, which larger N keep (the plane's weights would take half
// the registers); even rows are read 16 bytes at a time
template <int NP>
__device__ __forceinline__ void interp4(const double* __restrict__ Ue, const double* l1,
                                        const double* l2, const double* l3, double* out) {
  constexpr int N2 = NP * NP, N3 = N2 * NP;
  constexpr bool kW = NP <= 6;
  double w[kW ? N2 : 1];
  if constexpr (kW) {
#pragma unroll
    for (int q = 0; q < N2; ++q) w[q] = l1[q % NP] * l2[q / NP];
  }
#pragma unroll 1
  for (int v = 0; v < 4; ++v) {
    double acc = 0.0;
#pragma unroll 1
    for (int kk = 0; kk < NP; ++kk) {
      const double* P = Ue + v * N3 + kk * N2;
      double t2 = 0.0, t3 = 0.0;
      if constexpr (kW && NP % 2 == 0) {
#pragma unroll
        for (int q = 0; q < N2; q += 2) {
          const double2 u = __ldg(reinterpret_cast<const double2*>(P + q));
          t2 = fma(u.x, w[q], t2);
          t3 = fma(u.y, w[q + 1], t3);
        }
        t2 += t3;
      } else if constexpr (kW) {
#pragma unroll
        for (int q = 0; q < N2; ++q) {
          if (q & 1)
            t3 = fma(__ldg(P + q), w[q], t3);
          else
            t2 = fma(__ldg(P + q), w[q], t2);
        }
        t2 += t3;
      } else {
#pragma unroll
        for (int j = 0; j < NP; ++j) {
          double t1 = 0.0;
          if constexpr (NP % 2 == 0) {
#pragma unroll
            for (int i = 0; i < NP; i += 2) {
              const double2 u = __ldg(reinterpret_cast<const double2*>(P + NP * j + i));
              t1 = fma(u.x, l1[i], t1);
              t1 = fma(u.y, l1[i + 1], t1);
            }
          } else {
#pragma unroll
            for (int i = 0; i < NP; ++i) t1 = fma(__ldg(P + NP * j + i), l1[i], t1);
          }
          t2 = fma(t1, l2[j], t2);
        }
      }
      acc = fma(t2, l3[kk], acc);
    }
    out[v] = acc;
  }
}

// power in the working precision
__device__ __forceinline__ float tpow(float a, float b) { return powf(a, b); }
__device__ __forceinline__ double tpow(double a, double b) { return pow(a, b); }

// drag factor f_D (Sec. 2.2): 1 (Stokes), 1 + 0.15 Re_p^0.687 (Schiller-
// Naumann) or 1 + A Re^B + (Re/24) C / (1 + D/Re) (Haider-Levenspiel, A..D in
// k.hl); called for laws 1 and 2
template <typename T>
__device__ __forceinline__ T drag_factor(const DevConsts& k, T re) {
  if (k.drag_law == 1) return T(1) + T(0.15) * tpow(re, T(0.687));
  if (!(re > T(0))) return T(1);
  const T* h = Phys<T>::hl(k);
  return T(1) + h[0] * tpow(re, h[1]) + re / T(24) * h[2] / (T(1) + h[3] / re);
}

// ---------------------------------------------------------------------------
// tracking (Secs. 3.2.3-3.2.4, 2.4)
// ---------------------------------------------------------------------------

// Node (mm, kk) of local face f is base + mm sm + kk sk (mm along the face's
// first in-plane direction, kk along its second).
template <int G>
__device__ __forceinline__ void face_strides(int f, int& base, int& sm, int& sk) {
  const int fixed = (f & 1) ? G - 1 : 0;
  const int dir = f >> 1;
  base = fixed * (dir == 0 ? 1 : dir == 1 ? G : G * G);
  sm = dir == 0 ? G : 1;
  sk = dir == 2 ? G : G * G;
}

// curved face p(s,t) and its tangents from the element's Lagrange nodes
template <int G>
__device__ __forceinline__ void face_eval(const double* X64, int f, double s, double t,
                                          const DevConsts& k, double* p, double* ps,
                                          double* pt) {
  double ls[G], ds[G], lt[G], dt[G];
  lagr_d<G, double>(s, k.gn, k.gw, ls, ds);
  lagr_d<G, double>(t, k.gn, k.gw, lt, dt);
#pragma unroll
  for (int r = 0; r < 3; ++r) p[r] = ps[r] = pt[r] = 0.0;
  int base, sm, sk;
  face_strides<G>(f, base, sm, sk);
#pragma unroll
  for (int kk = 0; kk < G; ++kk)
#pragma unroll
    for (int mm = 0; mm < G; ++mm) {
      const double* P = X64 + 3 * (base + mm * sm + kk * sk);
      double w = ls[mm] * lt[kk], wsv = ds[mm] * lt[kk], wtv = ls[mm] * dt[kk];
#pragma unroll
      for (int r = 0; r < 3; ++r) {
        double xv = __ldg(P + r);
        p[r] = fma(xv, w, p[r]);
        ps[r] = fma(xv, wsv, ps[r]);
        pt[r] = fma(xv, wtv, pt[r]);
      }
    }
}

__device__ __forceinline__ void cross3d(const double* a, const double* b, double* c) {
  c[0] = a[1] * b[2] - a[2] * b[1];
  c[1] = a[2] * b[0] - a[0] * b[2];
  c[2] = a[0] * b[1] - a[1] * b[0];
}
__device__ __forceinline__ double dot3d(const double* a, const double* b) {
  return a[0] * b[0] + a[1] * b[1] + a[2] * b[2];
}

// Roots of the ray (origin xs, unit direction td, frame n1, n2) with the
// bilinear patch p(s,t) = a st + b s + c t + d: the two plane equations
// n_k.(p - xs) = 0 are eliminated to one quadratic (Ramsey et al. 2004).
// Writes up to 2 (s, t, alpha) triples; returns their number.
__device__ __forceinline__ int bilinear_roots(const double* B, const double* xs, const double* td,
                                              const double* n1, const double* n2, double* rs,
                                              double* rt, double* ra) {
  const double* a = B;
  const double* b = B + 3;
  const double* c = B + 6;
  double dd[3] = {B[9] - xs[0], B[10] - xs[1], B[11] - xs[2]};
  double A1 = dot3d(n1, a), B1 = dot3d(n1, b), C1 = dot3d(n1, c), D1 = dot3d(n1, dd);
  double A2 = dot3d(n2, a), B2 = dot3d(n2, b), C2 = dot3d(n2, c), D2 = dot3d(n2, dd);
  double scl = fabs(A1) + fabs(B1) + fabs(C1) + fabs(D1) + fabs(A2) + fabs(B2) + fabs(C2) +
               fabs(D2);
  if (!(scl > 0.0)) return 0;
  int nr = 0;
  #pragma unroll 1
  for (int pass = 0; pass < 2 && nr == 0; ++pass) {
    // pass 0 eliminates t (quadratic in s), pass 1 eliminates s (quadratic in t)
    double P1 = pass ? C1 : B1, Q1 = pass ? B1 : C1, P2 = pass ? C2 : B2, Q2 = pass ? B2 : C2;
    double q2 = P1 * A2 - P2 * A1;
    double q1 = P1 * Q2 + D1 * A2 - P2 * Q1 - D2 * A1;
    double q0 = D1 * Q2 - D2 * Q1;
    double r[2];
    int k = 0;
    if (fabs(q2) <= 1e-14 * scl * scl) {
      if (fabs(q1) > 0.0) r[k++] = -q0 / q1;
    } else {
      double disc = q1 * q1 - 4.0 * q2 * q0;
      if (disc >= 0.0) {
        double sq = sqrt(disc);
        double qq = -0.5 * (q1 + (q1 >= 0.0 ? sq : -sq));
        if (qq != 0.0) {
          r[k++] = qq / q2;
          r[k++] = q0 / qq;
        } else {
          r[k++] = 0.0;
        }
      }
    }
    #pragma unroll 1
    for (int i = 0; i < k; ++i) {
      double u = r[i];
      double den1 = A1 * u + Q1, den2 = A2 * u + Q2, w;
      if (fabs(den1) >= fabs(den2)) {
        if (fabs(den1) <= 1e-14 * scl) continue;
        w = -(P1 * u + D1) / den1;
      } else {
        if (fabs(den2) <= 1e-14 * scl) continue;
        w = -(P2 * u + D2) / den2;
      }
      double s = pass ? w : u, t = pass ? u : w;
      double pp[3];
#pragma unroll
      for (int q = 0; q < 3; ++q) pp[q] = a[q] * s * t + b[q] * s + c[q] * t + B[9 + q] - xs[q];
      rs[nr] = s;
      rt[nr] = t;
      ra[nr] = dot3d(td, pp);
      nr++;
    }
  }
  return nr;
}

// FP32 version of bilinear_roots used to screen faces before the exact FP64
// solve; sets ill when a root is ill-conditioned in FP32 (near-tangent ray,
// vanishing denominator), in which case the caller must not trust it.
__device__ __forceinline__ int bilinear_roots_f32(const float* B, const float* xs, const float* td,
                                                  const float* n1, const float* n2, float* rs,
                                                  float* rt, float* ra, bool& ill) {
  const float* a = B;
  const float* b = B + 3;
  const float* c = B + 6;
  const float dd[3] = {B[9] - xs[0], B[10] - xs[1], B[11] - xs[2]};
  auto dot = [](const float* u, const float* w) { return u[0] * w[0] + u[1] * w[1] + u[2] * w[2]; };
  const float A1 = dot(n1, a), B1 = dot(n1, b), C1 = dot(n1, c), D1 = dot(n1, dd);
  const float A2 = dot(n2, a), B2 = dot(n2, b), C2 = dot(n2, c), D2 = dot(n2, dd);
  const float scl = fabsf(A1) + fabsf(B1) + fabsf(C1) + fabsf(D1) + fabsf(A2) + fabsf(B2) +
                    fabsf(C2) + fabsf(D2);
  if (!(scl > 0.f)) {
    ill = true;
    return 0;
  }
  const float q2 = B1 * A2 - B2 * A1;
  const float q1 = B1 * C2 + D1 * A2 - B2 * C1 - D2 * A1;
  const float q0 = D1 * C2 - D2 * C1;
  float r[2];
  int k = 0;
  if (fabsf(q2) <= 1e-4f * scl * scl) {
    if (fabsf(q1) <= 1e-3f * scl * scl) {
      ill = true;
      return 0;
    }
    r[k++] = -q0 / q1;
  } else {
    const float disc = q1 * q1 - 4.f * q2 * q0;
    if (fabsf(disc) <= 1e-3f * q1 * q1 + 1e-6f * scl * scl * scl * scl) ill = true;
    if (disc >= 0.f) {
      const float sq = sqrtf(disc);
      const float qq = -0.5f * (q1 + (q1 >= 0.f ? sq : -sq));
      if (qq != 0.f) {
        r[k++] = qq / q2;
        r[k++] = q0 / qq;
      } else {
        ill = true;
      }
    }
  }
  int nr = 0;
  for (int i = 0; i < k; ++i) {
    const float u = r[i];
    const float den1 = A1 * u + C1, den2 = A2 * u + C2;
    const bool use1 = fabsf(den1) >= fabsf(den2);
    const float den = use1 ? den1 : den2;
    if (fabsf(den) <= 1e-3f * scl) {
      ill = true;
      continue;
    }
    const float w = -((use1 ? B1 : B2) * u + (use1 ? D1 : D2)) / den;
    float pp[3];
#pragma unroll
    for (int q = 0; q < 3; ++q) pp[q] = a[q] * u * w + b[q] * u + c[q] * w + dd[q];
    rs[nr] = u;
    rt[nr] = w;
    ra[nr] = dot(td, pp);
    nr++;
  }
  return nr;
}

// FP32 Newton on F(s,t,alpha) = p(s,t) - xs - alpha td for a curved face, from
// the element's FP32 nodes (coordinate-major); false if it does not settle.
template <int G>
__device__ __forceinline__ bool curved_newton_f32(const float* __restrict__ X32, int f,
                                                  const float* xs, const float* td,
                                                  const DevConsts& k, float& s, float& t,
                                                  float& al) {
  constexpr int G3 = G * G * G;
  #pragma unroll 1
  for (int it = 0; it < 12; ++it) {
    float ls[G], ds[G], lt[G], dt[G];
    lagr_d<G, float>(s, k.gn32, k.gw32, ls, ds);
    lagr_d<G, float>(t, k.gn32, k.gw32, lt, dt);
    float p[3] = {0, 0, 0}, ps[3] = {0, 0, 0}, pt[3] = {0, 0, 0};
    int base, sm, sk;
    face_strides<G>(f, base, sm, sk);
#pragma unroll
    for (int kk = 0; kk < G; ++kk)
#pragma unroll
      for (int mm = 0; mm < G; ++mm) {
        const int q = base + mm * sm + kk * sk;
        const float w = ls[mm] * lt[kk], wsv = ds[mm] * lt[kk], wtv = ls[mm] * dt[kk];
#pragma unroll
        for (int r = 0; r < 3; ++r) {
          const float xv = __ldg(X32 + r * G3 + q);
          p[r] = fmaf(xv, w, p[r]);
          ps[r] = fmaf(xv, wsv, ps[r]);
          pt[r] = fmaf(xv, wtv, pt[r]);
        }
      }
    float F[3], J[9], Ji[9], dl[3];
#pragma unroll
    for (int r = 0; r < 3; ++r) {
      F[r] = p[r] - xs[r] - al * td[r];
      J[3 * r] = ps[r];
      J[3 * r + 1] = pt[r];
      J[3 * r + 2] = -td[r];
    }
    if (!inv3(J, Ji)) return false;
    matvec3(Ji, F, dl);
    s -= dl[0];
    t -= dl[1];
    al -= dl[2];
    if (fabsf(dl[0]) < 1e-5f && fabsf(dl[1]) < 1e-5f) return true;
    if (!(fabsf(s) < 3.f && fabsf(t) < 3.f)) return false;
  }
  return false;
}

// curved face point p(s,t) alone (FP64), sum-factorised
template <int G>
__device__ __forceinline__ void face_point(const double* X64, int f, double s, double t,
                                           const DevConsts& k, double* p) {
  double ls[G], lt[G];
  lagr<G, double>(s, k.gn, k.gw, ls);
  lagr<G, double>(t, k.gn, k.gw, lt);
  int base, sm, sk;
  face_strides<G>(f, base, sm, sk);
  p[0] = p[1] = p[2] = 0.0;
#pragma unroll
  for (int kk = 0; kk < G; ++kk) {
    double q[3] = {0.0, 0.0, 0.0};
#pragma unroll
    for (int mm = 0; mm < G; ++mm) {
      const double* P = X64 + 3 * (base + mm * sm + kk * sk);
#pragma unroll
      for (int r = 0; r < 3; ++r) q[r] = fma(__ldg(P + r), ls[mm], q[r]);
    }
#pragma unroll
    for (int r = 0; r < 3; ++r) p[r] = fma(q[r], lt[kk], p[r]);
  }
}

// Newton on F(s,t,alpha) = p(s,t) - xs - alpha td for a curved face, started
// from a bilinear root: FP32 iterations on the FP32 nodes until the step is
// below 1e-5, then FP64 residuals with the last FP32 inverse Jacobian (each
// such step gains about six digits) until the step is below 1e-14; a full
// FP64 Newton if either stage does not settle.  Returns true on convergence.
template <int G>
__device__ __forceinline__ bool curved_refine(const double* X64, const float* __restrict__ X32,
                                              int f, const double* xs, const double* td,
                                              const DevConsts& k, double& s, double& t,
                                              double& al, double L) {
  constexpr int G3 = G * G * G;
  {
    float sf = (float)s, tf = (float)t, af = (float)al;
    const float xsf[3] = {(float)xs[0], (float)xs[1], (float)xs[2]};
    const float tdf[3] = {(float)td[0], (float)td[1], (float)td[2]};
    const float atol = 1e-5f * ((float)L + 1.f);
    int base, sm, sk;
    face_strides<G>(f, base, sm, sk);
    float Ji[9];
    bool ok32 = false;
#pragma unroll 1
    for (int it = 0; it < 12; ++it) {
      float ls[G], ds[G], lt[G], dt[G];
      lagr_d<G, float>(sf, k.gn32, k.gw32, ls, ds);
      lagr_d<G, float>(tf, k.gn32, k.gw32, lt, dt);
      float p[3] = {0, 0, 0}, ps[3] = {0, 0, 0}, pt[3] = {0, 0, 0};
#pragma unroll
      for (int kk = 0; kk < G; ++kk)
#pragma unroll
        for (int mm = 0; mm < G; ++mm) {
          const int q = base + mm * sm + kk * sk;
          const float w = ls[mm] * lt[kk], wsv = ds[mm] * lt[kk], wtv = ls[mm] * dt[kk];
#pragma unroll
          for (int r = 0; r < 3; ++r) {
            const float xv = __ldg(X32 + r * G3 + q);
            p[r] = fmaf(xv, w, p[r]);
            ps[r] = fmaf(xv, wsv, ps[r]);
            pt[r] = fmaf(xv, wtv, pt[r]);
          }
        }
      float F[3], J[9], dl[3];
#pragma unroll
      for (int r = 0; r < 3; ++r) {
        F[r] = p[r] - xsf[r] - af * tdf[r];
        J[3 * r] = ps[r];
        J[3 * r + 1] = pt[r];
        J[3 * r + 2] = -tdf[r];
      }
      if (!inv3(J, Ji)) break;
      matvec3(Ji, F, dl);
      sf -= dl[0];
      tf -= dl[1];
      af -= dl[2];
      if (fabsf(dl[0]) < 1e-5f && fabsf(dl[1]) < 1e-5f && fabsf(dl[2]) < atol) {
        ok32 = true;
        break;
      }
      if (!(fabsf(sf) < 3.f && fabsf(tf) < 3.f)) break;
    }
    if (ok32) {
      double sd = sf, tq = tf, ad = af;
#pragma unroll 1
      for (int it = 0; it < 4; ++it) {
        double p[3];
        face_point<G>(X64, f, sd, tq, k, p);
        float Fr[3], dl[3];
#pragma unroll
        for (int r = 0; r < 3; ++r) Fr[r] = (float)(p[r] - xs[r] - ad * td[r]);
        matvec3(Ji, Fr, dl);
        sd -= dl[0];
        tq -= dl[1];
        ad -= dl[2];
        if (fabs(dl[0]) < 1e-14 && fabs(dl[1]) < 1e-14 && fabs(dl[2]) < 1e-14 * (L + 1.0)) {
          s = sd;
          t = tq;
          al = ad;
          return true;
        }
      }
    }
  }
#pragma unroll 1
  for (int it = 0; it < 20; ++it) {
    double p[3], ps[3], pt[3], F[3], J[9], Ji[9], dl[3];
    face_eval<G>(X64, f, s, t, k, p, ps, pt);
#pragma unroll
    for (int r = 0; r < 3; ++r) {
      F[r] = p[r] - xs[r] - al * td[r];
      J[3 * r] = ps[r];
      J[3 * r + 1] = pt[r];
      J[3 * r + 2] = -td[r];
    }
    if (!inv3(J, Ji)) return false;
    matvec3(Ji, F, dl);
    s -= dl[0];
    t -= dl[1];
    al -= dl[2];
    if (fabs(dl[0]) < 1e-14 && fabs(dl[1]) < 1e-14 && fabs(dl[2]) < 1e-14 * (L + 1.0))
      return true;
    if (!(fabs(s) < 3.0 && fabs(t) < 3.0)) return false;
  }
  return false;
}

// ---------------------------------------------------------------------------
// Bezier clipping (Sec. 3.2.4; Nishita, Sederberg & Kakimoto 1990)
// ---------------------------------------------------------------------------

// x-range where the convex hull of the points (x_i, y_i) meets y = 0: the hull
// meets the axis exactly where some segment between two of its points does.
__device__ __forceinline__ bool hull_axis(const double* x, const double* y, int n, double& lo,
                                          double& hi) {
  lo = 1e300;
  hi = -1e300;
  for (int i = 0; i < n; ++i) {
    if (y[i] == 0.0) {
      lo = fmin(lo, x[i]);
      hi = fmax(hi, x[i]);
    }
    for (int j = i + 1; j < n; ++j)
      if ((y[i] < 0.0 && y[j] > 0.0) || (y[i] > 0.0 && y[j] < 0.0)) {
        const double xc = x[i] + (x[j] - x[i]) * (y[i] / (y[i] - y[j]));
        lo = fmin(lo, xc);
        hi = fmax(hi, xc);
      }
  }
  return lo <= hi;
}

// Control values of a tensor Bernstein polynomial restricted to [a, b] in its
// first (dir 0) or second (dir 1) parameter, by two de Casteljau splits.
template <int G>
__device__ __forceinline__ void bz_restrict(double (&D)[G][G], int dir, double a, double b) {
  for (int l = 0; l < G; ++l) {
    double c[G];
    for (int i = 0; i < G; ++i) c[i] = dir == 0 ? D[i][l] : D[l][i];
    // [0, b]: the left control points of the split at b
    double w[G], left[G];
    for (int i = 0; i < G; ++i) w[i] = c[i];
    for (int r = 0; r < G; ++r) {
      left[r] = w[0];
      for (int i = 0; i + 1 < G - r; ++i) w[i] = (1.0 - b) * w[i] + b * w[i + 1];
    }
    // [a/b, 1] of that: the right control points of the split at a/b
    const double t = b > 0.0 ? a / b : 0.0;
    for (int i = 0; i < G; ++i) w[i] = left[i];
    for (int r = 0; r < G; ++r) {
      c[G - 1 - r] = w[G - 1 - r];
      for (int i = 0; i + 1 < G - r; ++i) w[i] = (1.0 - t) * w[i] + t * w[i + 1];
    }
    for (int i = 0; i < G; ++i) {
      if (dir == 0)
        D[i][l] = c[i];
      else
        D[l][i] = c[i];
    }
  }
}

// Interval of the first (dir 0) or second (dir 1) parameter in [0, 1] outside
// which the Bernstein polynomial with control values D has no zero.
template <int G>
__device__ __forceinline__ bool bz_clip(const double (&D)[G][G], int dir, double& lo,
                                        double& hi) {
  double x[2 * G], y[2 * G];
  for (int i = 0; i < G; ++i) {
    double mn = 1e300, mx = -1e300;
    for (int l = 0; l < G; ++l) {
      const double v = dir == 0 ? D[i][l] : D[l][i];
      mn = fmin(mn, v);
      mx = fmax(mx, v);
    }
    x[2 * i] = x[2 * i + 1] = G > 1 ? (double)i / (G - 1) : 0.0;
    y[2 * i] = mn;
    y[2 * i + 1] = mx;
  }
  if (!hull_axis(x, y, 2 * G, lo, hi)) return false;
  lo = fmax(0.0, lo - 1e-12);
  hi = fmin(1.0, hi + 1e-12);
  return lo <= hi;
}

// All crossings of the line xs + alpha td (frame n1, n2 normal to td) with a
// curved face, by Bezier clipping: the face's control net is projected on the
// two planes through the line, and the parameter domain is cut to where the
// convex hulls of both projections can vanish, in s and in t; a domain whose
// area does not at least halve is split in two, and pending domains wait on a
// stack of parameter boxes (their nets are restricted again from the face's).
// A domain below 1e-9 gives a candidate, refined by curved_refine (kept as it
// is if the refinement does not settle).  Writes up to maxr (s, t, alpha) with
// s, t in [-1, 1]; returns their number.
template <int G>
__device__ __noinline__ int bezier_clip_roots(const double* X64, const float* X32, int f,
                                              const double* xs, const double* td,
                                              const double* n1, const double* n2,
                                              const DevConsts& k, double L, double* rs,
                                              double* rt, double* ra, int maxr) {
  constexpr int kStack = 24;
  double full[2][G][G];
  int base, sm, sk;
  face_strides<G>(f, base, sm, sk);
  for (int i = 0; i < G; ++i)
    for (int j = 0; j < G; ++j) {
      double c[3] = {0.0, 0.0, 0.0};
      for (int mm = 0; mm < G; ++mm)
        for (int kk = 0; kk < G; ++kk) {
          const double w = k.gbz[i * G + mm] * k.gbz[j * G + kk];
          const double* P = X64 + 3 * (base + mm * sm + kk * sk);
          for (int r = 0; r < 3; ++r) c[r] = fma(w, __ldg(P + r), c[r]);
        }
      const double q[3] = {c[0] - xs[0], c[1] - xs[1], c[2] - xs[2]};
      full[0][i][j] = n1[0] * q[0] + n1[1] * q[1] + n1[2] * q[2];
      full[1][i][j] = n2[0] * q[0] + n2[1] * q[1] + n2[2] * q[2];
    }
  double box[kStack][4];
  box[0][0] = 0.0;
  box[0][1] = 1.0;
  box[0][2] = 0.0;
  box[0][3] = 1.0;
  int top = 1, nr = 0;
#pragma unroll 1
  for (int visit = 0; visit < 600 && top > 0; ++visit) {
    --top;
    double u0 = box[top][0], u1 = box[top][1], v0 = box[top][2], v1 = box[top][3];
    double D[2][G][G];
    for (int w = 0; w < 2; ++w) {
      for (int i = 0; i < G; ++i)
        for (int j = 0; j < G; ++j) D[w][i][j] = full[w][i][j];
      bz_restrict<G>(D[w], 0, u0, u1);
      bz_restrict<G>(D[w], 1, v0, v1);
    }
    bool split = true;
#pragma unroll 1
    for (int it = 0; it < 16; ++it) {
      double ulo = 0.0, uhi = 1.0, vlo = 0.0, vhi = 1.0;
      bool hit = true;
      for (int w = 0; w < 2 && hit; ++w) {
        double a, b;
        hit = bz_clip<G>(D[w], 0, a, b);
        ulo = fmax(ulo, a);
        uhi = fmin(uhi, b);
        hit = hit && ulo <= uhi;
      }
      for (int w = 0; w < 2 && hit; ++w) {
        double a, b;
        hit = bz_clip<G>(D[w], 1, a, b);
        vlo = fmax(vlo, a);
        vhi = fmin(vhi, b);
        hit = hit && vlo <= vhi;
      }
      if (!hit) {
        split = false;
        break;
      }
      const double wu = u1 - u0, wv = v1 - v0;
      for (int w = 0; w < 2; ++w) {
        bz_restrict<G>(D[w], 0, ulo, uhi);
        bz_restrict<G>(D[w], 1, vlo, vhi);
      }
      u1 = u0 + wu * uhi;
      u0 = u0 + wu * ulo;
      v1 = v0 + wv * vhi;
      v0 = v0 + wv * vlo;
      if (u1 - u0 < 1e-9 && v1 - v0 < 1e-9) {
        double s = u0 + u1 - 1.0, t = v0 + v1 - 1.0;  // 2 * midpoint - 1
        double p[3];
        face_point<G>(X64, f, s, t, k, p);
        double al = td[0] * (p[0] - xs[0]) + td[1] * (p[1] - xs[1]) + td[2] * (p[2] - xs[2]);
        double s2 = s, t2 = t, al2 = al;
        if (curved_refine<G>(X64, X32, f, xs, td, k, s2, t2, al2, L) &&
            fabs(s2 - s) < 1e-6 && fabs(t2 - t) < 1e-6) {
          s = s2;
          t = t2;
          al = al2;
        }
        bool dup = false;
        for (int q = 0; q < nr; ++q)
          if (fabs(rs[q] - s) < 1e-9 && fabs(rt[q] - t) < 1e-9) dup = true;
        if (!dup && nr < maxr) {
          rs[nr] = s;
          rt[nr] = t;
          ra[nr] = al;
          ++nr;
        }
        split = false;
        break;
      }
      if ((uhi - ulo) * (vhi - vlo) > 0.5) break;  // little progress: split
    }
    if (split && top + 2 <= kStack) {
      // halve the longer side of the current box
      double b0[4] = {u0, u1, v0, v1}, b1[4] = {u0, u1, v0, v1};
      if (u1 - u0 >= v1 - v0) {
        b0[1] = b1[0] = 0.5 * (u0 + u1);
      } else {
        b0[3] = b1[2] = 0.5 * (v0 + v1);
      }
      for (int q = 0; q < 4; ++q) {
        box[top][q] = b1[q];
        box[top + 1][q] = b0[q];
      }
      top += 2;
    }
  }
  return nr;
}

template <typename R>
__device__ __forceinline__ void reflect3(R* a, const double* n) {
  double s = 2.0 * ((double)a[0] * n[0] + (double)a[1] * n[1] + (double)a[2] * n[2]);
#pragma unroll
  for (int r = 0; r < 3; ++r) a[r] = (R)((double)a[r] - s * n[r]);
}

struct TrackCounters {
  int cross, hits, slow;
};

// Conservative FP32 test: which kind of face of element e can the segment a -> b
// (element-local coordinates, extended by the band) touch: bit 0 some face (or a
// long segment), bit 1 a wall or open face (or a long segment).  Slab of face f:
// lo <= n.(P - ce) <= hi for every point of the face, margins (band plus
// 4e-6 of the element radius, which covers the FP32 rounding of a and b while
// they stay within 8 radii) included; longer segments take the exact path.  Slab
// word 7 flags the wall and open faces.
__device__ __forceinline__ int slab_touch(const DevMesh& m, int e, const float* a,
                                          const float* b) {
  const float4* S = reinterpret_cast<const float4*>(m.slab + 48 * (size_t)e);
  const float rlim = 8.f * __ldg(m.slab + 48 * (size_t)e + 5);
  int t = (fmaxf(fmaxf(fabsf(b[0]), fabsf(b[1])), fabsf(b[2])) <= rlim) ? 0 : 3;
#pragma unroll
  for (int f = 0; f < 6; ++f) {
    float4 s0 = __ldg(S + 2 * f), s1 = __ldg(S + 2 * f + 1);
    float pa = s0.x * a[0] + s0.y * a[1] + s0.z * a[2];
    float pb = s0.x * b[0] + s0.y * b[1] + s0.z * b[2];
    if ((fmaxf(pa, pb) >= s0.w) && (fminf(pa, pb) <= s1.x)) t |= s1.w != 0.f ? 3 : 1;
  }
  return t;
}

// Big side of a mortar (Sec. 3.2.3): the crossing found on the big face is
// searched again on the small faces matched to it -- their own tables and
// geometry, the same ray (a root finder that reports every crossing needs no
// inverted ray) -- and the small face whose accepted crossing lies closest to
// the big face's one (lowest index on ties) becomes the entry face.  If none
// reports it (a rounding-size gap at the small faces' shared edges), the small
// face whose part of the big face holds the big face's crossing parameters
// (bs, bt) is taken.  Out of line: mortar crossings are rare.
template <int G, bool CLIP>
__device__ __noinline__ void mortar_enter(const DevMesh& m, const DevConsts& k, int row, double bs,
                                          double bt, const double* xs, const double* td,
                                          const double* n1, const double* n2, double L, double a0,
                                          double best, int& e, int& fin, double& anew,
                                          unsigned& st) {
  const int* mt = m.mort + 9 * (size_t)row;
  const int type = __ldg(mt);
  const int ns = type == PT_MORTAR_FOUR ? 4 : 2;
  int kb = -1;
  double db = 1e300, ka = best, km = 1.0;
#pragma unroll 1
  for (int q = 0; q < ns; ++q) {
    const int es = __ldg(mt + 1 + q), fs = __ldg(mt + 5 + q);
    const double* ce = m.ce + 3 * (size_t)es;
    const double xl[3] = {xs[0] - __ldg(ce), xs[1] - __ldg(ce + 1), xs[2] - __ldg(ce + 2)};
    const double* X64 = m.xg64 + (size_t)es * 3 * G * G * G;
    const float* X32 = m.xg32 + (size_t)es * 3 * G * G * G;
    const int kind = finfo_kind(__ldg(m.finfo + 6 * (size_t)es + fs));
    constexpr int MR = CLIP ? 4 : 2;
    double rs[MR], rt[MR], ra[MR];
    int nr;
    if (CLIP && kind == PT_FACE_CURVED) {
      nr = bezier_clip_roots<G>(X64, X32, fs, xl, td, n1, n2, k, L, rs, rt, ra, MR);
    } else {
      const double* Bf = m.bil + 72 * (size_t)es + 12 * fs;
      double Bl[12];
#pragma unroll
      for (int i = 0; i < 12; ++i) Bl[i] = __ldg(Bf + i);
      nr = bilinear_roots(Bl, xl, td, n1, n2, rs, rt, ra);
      if (kind == PT_FACE_CURVED) {
        int kk = 0;
#pragma unroll 1
        for (int i = 0; i < nr; ++i) {
          double s = rs[i], t = rt[i], al = ra[i];
          if (!(fabs(s) < 2.0 && fabs(t) < 2.0)) continue;
          if (curved_refine<G>(X64, X32, fs, xl, td, k, s, t, al, L)) {
            rs[kk] = s;
            rt[kk] = t;
            ra[kk] = al;
            kk++;
          }
        }
        nr = kk;
      }
    }
#pragma unroll 1
    for (int i = 0; i < nr; ++i) {
      const double mm = fmax(fabs(rs[i]), fabs(rt[i]));
      if (mm > 1.0 + k.band_ref) continue;
      if (ra[i] < a0 - k.band_x || ra[i] > L + k.band_x) continue;
      const double dd = fabs(ra[i] - best);
      if (dd < db) {
        db = dd;
        kb = q;
        ka = ra[i];
        km = mm;
      }
    }
  }
  if (kb < 0) {
    const int is = bs > 0.0, it = bt > 0.0;
    kb = type == PT_MORTAR_FOUR ? is + 2 * it : (type == PT_MORTAR_S ? is : it);
    ka = best;
    km = 1.0;
  }
  if (fabs(km - 1.0) < k.band_ref) st |= PT_ST_NEAR_FACE;
  e = __ldg(mt + 1 + kb);
  fin = __ldg(mt + 5 + kb);
  anew = ka;
}

// Bound on how far xi(x + dx) can be from xi(x) + D, D = Ji dx, along the
// straight segment dx: with the second derivatives of chi_r bounded by S_r and
// K_d = sum_j |Ji_dj| S_j / 2, |xi - xi_lin|_d <= 2 K_d |D|^2 while K |D| <= 1/8
// (else the bound is not used: returns false).  |D| is taken larger by what the
// path is extended by the distance band_x at its ends and by 1e-3, how far from xi
// Ji may have been evaluated (newton_df).  S_r = grow DevMesh::curv, which holds
// for |xi| <= 1.1; the caller says by grow how far the path goes beyond (1 if it
// does not).  D_d is a sum of products that may cancel (a displacement along the
// long side of a thin element that is not aligned with the axes), so its FP32
// rounding scales with sum_j |Ji_dj| |dx_j|: 2e-6 of that, some 30 roundings, for
// the Jacobian's Horner sums, its inverse and the product.  bend is the largest of
// the curvature parts and roundings, marg[d] their sum plus band_x in reference
// units plus 1e-5 for the FP32 rounding of xi.
__device__ __forceinline__ bool xi_margin(const DevMesh& m, int e, const float* Ji,
                                          const float* dx, const float* D, float bx, float grow,
                                          float* marg, float& bend) {
  const float4 S = __ldg(reinterpret_cast<const float4*>(m.curv) + e);
  float b[3];
#pragma unroll
  for (int d = 0; d < 3; ++d)
    b[d] = (fabsf(Ji[3 * d]) + fabsf(Ji[3 * d + 1]) + fabsf(Ji[3 * d + 2])) * bx;
  const float a = tmax3(D[0], D[1], D[2]) + tmax3(b[0], b[1], b[2]) + 1e-3f, a2 = grow * a * a;
  const float c[3] = {fmaf(2e-6f, fabsf(dx[0]), S.x * a2), fmaf(2e-6f, fabsf(dx[1]), S.y * a2),
                      fmaf(2e-6f, fabsf(dx[2]), S.z * a2)};
  bend = 0.f;
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    const float q =
        fabsf(Ji[3 * d]) * c[0] + fabsf(Ji[3 * d + 1]) * c[1] + fabsf(Ji[3 * d + 2]) * c[2];
    bend = fmaxf(bend, q);
    marg[d] = q + b[d] + 1e-5f;
  }
  return bend <= 0.25f * a;
}

// True only if the stage segment from xi (inside element e) along dx cannot come
// within the bands of any face: its linearised path and the bound above stay
// inside.  Ji: the inverse Jacobian at xi.  Much sharper than the faces' slabs,
// which are as thick as a face is curved (0.85 % of the 32^3 channel's segments
// touch a slab, 0.12 % cross a face), and it needs 16 bytes of the element
// instead of 192.
__device__ __forceinline__ bool stays_inside(const DevMesh& m, int e, const float* xi,
                                             const float* Ji, const float* dx, float bx) {
  float D[3], marg[3], bend;
  matvec3(Ji, dx, D);
  bool in = xi_margin(m, e, Ji, dx, D, bx, 1.f, marg, bend);
#pragma unroll
  for (int d = 0; d < 3; ++d)
    in = in && fmaxf(fabsf(xi[d]), fabsf(xi[d] + D[d])) <= 1.f - marg[d];
  return in;
}

// One Newton step d on F(s, t, alpha) = chi(s, t on face f) - (x + alpha td) = 0
// from the Jacobian in FP32 and the double-float residual of the inverse map
// (error ~1e-14 of the element); x a double-float offset, td the unit
// direction.  cosr: the cosine between the ray and the face normal there; lat:
// the largest change of s or t per unit of length of the right-hand side.
// False if the Jacobian is singular.
template <int G>
__device__ __forceinline__ bool face_step(const DevMesh& m, int e, int tm, int f, const df* x,
                                          const float* td, float s, float t, float al, float* d,
                                          float& cosr, float& lat) {
  const float* Mh = m.mono + (size_t)e * 3 * Mono<G>::CS;
  const int q = f >> 1;
  const float w = (f & 1) ? 1.f : -1.f;
  // xi_q = -1 or +1, s and t along the two other directions in order
  const float xi[3] = {q == 0 ? w : s, q == 1 ? w : (q == 0 ? s : t), q == 2 ? w : t};
  float chi[3], J[9], A[9], Ai[9], F[3];
  map_j32<G>(Mh, xi, tm, chi, J);
  df xa[3];
#pragma unroll
  for (int r = 0; r < 3; ++r) {
    A[3 * r] = q == 0 ? J[3 * r + 1] : J[3 * r];
    A[3 * r + 1] = q == 2 ? J[3 * r + 1] : J[3 * r + 2];
    A[3 * r + 2] = -td[r];
    df p;
    two_prod(al, td[r], p.hi, p.lo);
    xa[r] = df_add(x[r], p);
  }
  if (!inv3(A, Ai)) return false;
  resid_df<G>(Mh, m.monolo + (size_t)e * 3 * Mono<G>::CS, xi, tm, xa, F);
  // row 3 of Ai is -n / (n . td), n the face normal p_s x p_t
  cosr = 1.f / sqrtf(Ai[6] * Ai[6] + Ai[7] * Ai[7] + Ai[8] * Ai[8]);
  lat = fmaxf(fabsf(Ai[0]) + fabsf(Ai[1]) + fabsf(Ai[2]),
              fabsf(Ai[3]) + fabsf(Ai[4]) + fabsf(Ai[5]));
  matvec3(Ai, F, d);
  return true;
}

// FP32 pass of the tracking (FP32 mode): the stage segment xd -> xe (double-
// float offsets from the centre of element e) in reference space.  In the
// current element the end point's xi is found by the inverse map, and the
// segment's path is xi - (1 - tau) D up to the bound of xi_margin.  Only faces
// that the path can come to within the bands are intersected: the linear path
// gives the start, two Newton steps with the double-float residual follow.  The
// direction, the length and alpha itself are single FP32 numbers, so the crossing
// is good to a few roundings (6e-8) of the length L, whatever the residual is:
// acceptance and the near-face bands are decided with the margins tb on alpha,
// 1e-6 (L + band_x) plus 1e-8 of the element over the cosine to the face, and ms
// on s and t, 2e-6 plus 1e-6 (L + band_x) in reference units; an end that is not
// inside by a rounding is not decided here either.  (With 1e-8 of L, 3 % of the
// ends up to 1e-7 beyond a wall were taken as inside at L from 0.2 elements on.)
// The smallest accepted alpha wins; an internal or
// periodic face leads to the next element, the position is the segment's end.
// A wall, open or mortar face that is hit, a path nearly parallel to a face it
// may reach, a quantity within the margin of its threshold and two crossings
// within the margin return false with nothing changed, and track_slow
// intersects the faces in FP64.
template <int G>
__device__ __forceinline__ bool track_f32(const DevMesh& m, const DevConsts& k, int& e_io, df* xd,
                                          const df* xe, unsigned& st, int& it32, int& it64,
                                          TrackCounters& tc) {
  int e = e_io, cross = 0, fin = -1;
  unsigned bits = 0u;
  float dx[3], td[3], a0 = 0.f, a0tb = 0.f;
  df x[3] = {xe[0], xe[1], xe[2]};      // the segment's ends in the current element's frame
  df x0[3] = {xd[0], xd[1], xd[2]};
  double xg[3] = {0.0, 0.0, 0.0}, xs[3] = {0.0, 0.0, 0.0};  // global, once it has crossed
#pragma unroll
  for (int r = 0; r < 3; ++r) dx[r] = (xe[r].hi - xd[r].hi) + (xe[r].lo - xd[r].lo);
  const float L = sqrtf(dx[0] * dx[0] + dx[1] * dx[1] + dx[2] * dx[2]);
  if (!(L > 0.f)) return false;
#pragma unroll
  for (int r = 0; r < 3; ++r) td[r] = dx[r] / L;
  const float bx = k.band_x32, br = k.band_ref32, ext = 1.f + 2.f * bx / L;
#pragma unroll 1
  while (true) {
    const float xf[3] = {x[0].hi, x[1].hi, x[2].hi};
    const int tm = G == 2 ? 7 : __ldg(m.tmask + e);
    float g[3], Ji[9], D[3], marg[3], bend;
    df zd[3];
    trilinear_guess(m, e, xf, g);
    bool jok;
    if (!newton_df<G>(m, k, e, x, g, zd, it32, it64, Ji, jok) || !jok) return false;
    matvec3(Ji, dx, D);
    // The segment leaves the element, so the path may reach far beyond the range
    // that the curvature bound holds for: from its end back to where it came in,
    // and 0.1 to the sides, which the margins may not exceed.  There a second
    // derivative's terms of total degree n <= 3 (G - 1) are at most (z / 1.1)^(n - 2) /
    // 1.1^2 times the bound's.
    const float back = 1.f - a0 / L;
    float zr = 0.f;
#pragma unroll
    for (int d = 0; d < 3; ++d)
      zr = fmaxf(zr, fmaxf(fabsf(zd[d].hi), fabsf(zd[d].hi - back * D[d])));
    const float zq1 = (zr + 0.1f) * (1.f / 1.1f);
    float grow = 1.f / 1.21f;
#pragma unroll
    for (int p = 0; p < 3 * G - 5; ++p) grow *= zq1;
    if (!xi_margin(m, e, Ji, dx, D, bx, fmaxf(grow, 1.f), marg, bend)) return false;
    if (!(tmax3(marg[0], marg[1], marg[2]) <= 0.1f)) return false;
    unsigned faces = 0u;
    bool in = true;
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      const float z1 = zd[d].hi, z0 = z1 - D[d];
      if (fmaxf(z0, z1) > 1.f - marg[d]) faces |= 2u << (2 * d);
      if (fminf(z0, z1) < -1.f + marg[d]) faces |= 1u << (2 * d);
      in = in && fabsf(z1) < 1.f;
    }
    if (fin >= 0) faces &= ~(1u << fin);
    int pf = -1;
    float pal = 0.f, ptb = 0.f;
#pragma unroll 1
    while (faces) {
      const int f = __ffs(faces) - 1, q = f >> 1;
      faces &= faces - 1u;
      const float w = (f & 1) ? 1.f : -1.f;
      const float Dq = q == 0 ? D[0] : (q == 1 ? D[1] : D[2]);
      const float zq = q == 0 ? zd[0].hi : (q == 1 ? zd[1].hi : zd[2].hi);
      // the path (and band_x beyond its ends) is monotone across the face, so
      // that it meets the face once: slope Dq against the bend of the bound
      if (!(fabsf(Dq) > fmaxf(2.f * ext * bend, 1e-2f * tmax3(D[0], D[1], D[2])))) return false;
      const float u = (zq - w) / Dq;  // 1 - tau at the face
      if (!(fabsf(u) < 4.f * ext)) continue;
      float s = q == 0 ? zd[1].hi - u * D[1] : zd[0].hi - u * D[0];
      float t = q == 2 ? zd[1].hi - u * D[1] : zd[2].hi - u * D[2];
      float al = L - u * L, d[3], cosr = 0.f, lat = 0.f;
#pragma unroll 1
      for (int it = 0; it < 2; ++it) {
        if (!face_step<G>(m, e, tm, f, x0, td, s, t, al, d, cosr, lat)) return false;
        s -= d[0];
        t -= d[1];
        al -= d[2];
      }
      if (!(cosr > 1e-3f) || !(fabsf(d[0]) < 1e-5f && fabsf(d[1]) < 1e-5f && fabsf(d[2]) < 1e-4f * (L + bx)))
        return false;
      const float Rmax = __ldg(m.slab + 48 * (size_t)e + 5);
      const float el = 1e-6f * (L + bx), mm = fmaxf(fabsf(s), fabsf(t));
      const float ms = 2e-6f + el * lat, tb = (1e-8f * Rmax + el) / cosr, ta = tb + a0tb;
      const float om = mm - 1.f, da = al - a0, dL = L - al;
      if (om > br + ms || da < -bx - ta || dL < -bx - tb) continue;
      if (fabsf(om) <= ms || fabsf(fabsf(om) - br) <= ms || fabsf(da) <= ta ||
          fabsf(dL) <= tb || fabsf(fabsf(da) - bx) <= ta || fabsf(fabsf(dL) - bx) <= tb)
        return false;
      const int bc = finfo_bc(__ldg(m.finfo + 6 * (size_t)e + f));
      if (fabsf(om) < br || fabsf(da) < bx || fabsf(dL) < bx)
        bits |= PT_ST_NEAR_FACE |
                ((bc == PT_BC_WALL || bc == PT_BC_OPEN) ? (unsigned)PT_ST_NEAR_WALL : 0u);
      if (om < 0.f && da > 0.f && dL > 0.f) {
        if (!(bc == PT_BC_INTERNAL || bc == PT_BC_PERIODIC)) return false;
        if (pf >= 0 && fabsf(al - pal) <= tb + ptb) return false;
        if (pf < 0 || al < pal) {
          pf = f;
          pal = al;
          ptb = tb;
        }
      }
    }
    if (pf < 0) {
      if (!in) return false;
      break;
    }
    if (cross + 1 >= k.max_cross || cross >= 8) return false;
    if (!cross) {
      const double* ce = m.ce + 3 * (size_t)e;
#pragma unroll
      for (int r = 0; r < 3; ++r) {
        const double cr = __ldg(ce + r);
        xs[r] = cr + df_to_double(xd[r]);
        xg[r] = cr + df_to_double(xe[r]);
      }
    }
    const int info = __ldg(m.finfo + 6 * (size_t)e + pf);
    if (finfo_bc(info) == PT_BC_PERIODIC) {
      const double* sh = m.shift + 18 * (size_t)e + 3 * pf;
#pragma unroll
      for (int r = 0; r < 3; ++r) {
        xs[r] += __ldg(sh + r);
        xg[r] += __ldg(sh + r);
      }
    }
    fin = finfo_nf(info);
    e = __ldg(m.fnbr + 6 * (size_t)e + pf);
    a0 = pal;
    a0tb = ptb;
    const double* cn = m.ce + 3 * (size_t)e;
#pragma unroll
    for (int r = 0; r < 3; ++r) {
      const double cr = __ldg(cn + r);
      x[r] = df_from_double(xg[r] - cr);
      x0[r] = df_from_double(xs[r] - cr);
    }
    ++cross;
  }
#pragma unroll
  for (int r = 0; r < 3; ++r) xd[r] = x[r];
  e_io = e;
  st |= bits;
  tc.cross += cross;
  ++tc.slow;
  return true;
}

// Tracks the stage segment x -> xe through the mesh.  The ray
// x(alpha) = xs + alpha td, alpha in (a0, L] (Eq. parttrajectory) is tested
// against every face of the current element except the entry face; the
// smallest accepted alpha wins (lowest face index on ties).  Internal face:
// continue in the neighbour on the same ray.  Periodic: same, translated.
// Wall: restart at the hit point with the remaining length, mirroring the
// direction, v, kx and kv by I - 2 n n^T (Sec. 2.4).  Open: stop there.
// CLIP: curved faces by Bezier clipping (a separate instantiation, so that the
// default path carries none of its code)
template <int G, typename R, bool CLIP>
__device__ __noinline__ void track_slow(const DevMesh& m, const DevConsts& k, int& e, double* x,
                                        double* xe, R* v, R* kx, R* kv, int& hits, unsigned& st,
                                        TrackCounters& tc) {
  tc.slow++;
  double xs[3] = {x[0], x[1], x[2]};
  double td[3] = {xe[0] - xs[0], xe[1] - xs[1], xe[2] - xs[2]};
  double L = sqrt(dot3d(td, td));
  if (!(L > 0.0)) {
#pragma unroll
    for (int r = 0; r < 3; ++r) x[r] = xe[r];
    return;
  }
  {
    const double iL = 1.0 / L;
#pragma unroll
    for (int r = 0; r < 3; ++r) td[r] *= iL;
  }
  float tdf[3] = {(float)td[0], (float)td[1], (float)td[2]};
  float Lf = (float)L;
  float n1f[3], n2f[3];
  double n1[3], n2[3];
  {
    double ax[3] = {0, 0, 0};
    int im = 0;
    if (fabs(td[1]) < fabs(td[im])) im = 1;
    if (fabs(td[2]) < fabs(td[im])) im = 2;
    ax[im] = 1.0;
    cross3d(td, ax, n1);
    const double inn = 1.0 / sqrt(dot3d(n1, n1));
#pragma unroll
    for (int r = 0; r < 3; ++r) n1[r] *= inn;
    cross3d(td, n1, n2);
#pragma unroll
    for (int r = 0; r < 3; ++r) {
      n1f[r] = (float)n1[r];
      n2f[r] = (float)n2[r];
    }
  }
  double a0 = 0.0;
  int fin = -1;
  int ncr;
  for (ncr = 0; ncr < k.max_cross; ++ncr) {
    const double* ce = m.ce + 3 * (size_t)e;
    double xl[3] = {xs[0] - __ldg(ce), xs[1] - __ldg(ce + 1), xs[2] - __ldg(ce + 2)};
    const double* X64 = m.xg64 + (size_t)e * 3 * G * G * G;
    const float xlf[3] = {(float)xl[0], (float)xl[1], (float)xl[2]};
    double best = 1e300, bs = 0.0, bt = 0.0;
    int bf = -1;
#pragma unroll 1
    for (int f = 0; f < 6; ++f) {
      if (f == fin) continue;
      // slab prefilter (FP32, conservative: the margins cover its rounding)
      const float* sl = m.slab + 48 * (size_t)e + 8 * f;
      const float cosf_ = __ldg(sl) * tdf[0] + __ldg(sl + 1) * tdf[1] + __ldg(sl + 2) * tdf[2];
      const float pa = __ldg(sl) * xlf[0] + __ldg(sl + 1) * xlf[1] + __ldg(sl + 2) * xlf[2];
      const float pb = pa + Lf * cosf_;
      if (fmaxf(pa, pb) < __ldg(sl + 3) || fminf(pa, pb) > __ldg(sl + 4)) continue;
      const int info = __ldg(m.finfo + 6 * (size_t)e + f);
      const int kind = finfo_kind(info);
      // FP32 screen: skip the exact solve when every FP32 root is clearly
      // outside the segment or the face (margins ~100x the FP32 error)
      float fs[2], ft[2], fa[2];
      bool ill = fabsf(cosf_) < 1e-2f;
      if (PT_FACE_SCREEN) {
        const float* Bf32 = m.bil32 + 72 * (size_t)e + 12 * f;
        float B32[12];
#pragma unroll
        for (int q = 0; q < 12; ++q) B32[q] = __ldg(Bf32 + q);
        const int n32 = bilinear_roots_f32(B32, xlf, tdf, n1f, n2f, fs, ft, fa, ill);
        const float ta = 1e-4f * (__ldg(sl + 5) + Lf) / fmaxf(fabsf(cosf_), 1e-2f) +
                         4.f * (float)k.band_x;
        const float a0f = (float)a0;
        bool any = ill;
        #pragma unroll 1
        for (int i = 0; i < n32 && !ill; ++i) {
          if (kind == PT_FACE_CURVED &&
              !curved_newton_f32<G>(m.xg32 + (size_t)e * 3 * G * G * G, f, xlf, tdf, k, fs[i],
                                    ft[i], fa[i])) {
            any = true;
            break;
          }
          const float mm = fmaxf(fabsf(fs[i]), fabsf(ft[i]));
          if (!(fa[i] < a0f - ta || fa[i] > Lf + ta || mm > 1.f + 1e-3f)) any = true;
        }
        if (!any) continue;
      }
      const double* Bf = m.bil + 72 * (size_t)e + 12 * f;
      double Bl[12];
#pragma unroll
      for (int q = 0; q < 12; ++q) Bl[q] = __ldg(Bf + q);
      constexpr int MR = CLIP ? 4 : 2;
      double rs[MR], rt[MR], ra[MR];
      int nr = 0;
      const bool clip_all = CLIP && kind == PT_FACE_CURVED;
      if constexpr (CLIP) {
        if (clip_all)
          nr = bezier_clip_roots<G>(X64, m.xg32 + (size_t)e * 3 * G * G * G, f, xl, td, n1, n2,
                                    k, L, rs, rt, ra, MR);
        else
          nr = bilinear_roots(Bl, xl, td, n1, n2, rs, rt, ra);
      } else {
        nr = bilinear_roots(Bl, xl, td, n1, n2, rs, rt, ra);
      }
      if (kind == PT_FACE_CURVED && !clip_all) {
        // the curved face lies within dev of its bilinear patch: a bilinear
        // crossing far beyond the segment cannot refine into one inside it
        const double dev = (double)__ldg(sl + 6);
        const double reach = 4.0 * dev / fmax((double)fabsf(cosf_), 0.05) + 2.0 * k.band_x;
        int kk = 0;
        #pragma unroll 1
        for (int i = 0; i < nr; ++i) {
          double s = rs[i], t = rt[i], al = ra[i];
          if (!(fabs(s) < 2.0 && fabs(t) < 2.0)) continue;
          if (al > L + reach || al < a0 - reach) continue;
          if (curved_refine<G>(X64, m.xg32 + (size_t)e * 3 * G * G * G, f, xl, td, k, s, t,
                               al, L)) {
            bool dup = false;
            for (int j = 0; j < kk; ++j)
              if (fabs(rs[j] - s) < 1e-10 && fabs(rt[j] - t) < 1e-10) dup = true;
            if (!dup) {
              rs[kk] = s;
              rt[kk] = t;
              ra[kk] = al;
              kk++;
            }
          }
        }
        nr = kk;
      }
      #pragma unroll 1
      for (int i = 0; i < nr; ++i) {
        double al = ra[i], s = rs[i], t = rt[i];
        double mm = fmax(fabs(s), fabs(t));
        if (mm > 1.0 + k.band_ref) continue;
        if (al < a0 - k.band_x || al > L + k.band_x) continue;
        if (fabs(mm - 1.0) < k.band_ref || fabs(al - a0) < k.band_x ||
            fabs(L - al) < k.band_x) {
          const int bcf = finfo_bc(info);
          st |= PT_ST_NEAR_FACE |
                ((bcf == PT_BC_WALL || bcf == PT_BC_OPEN) ? (unsigned)PT_ST_NEAR_WALL : 0u);
        }
        if (mm <= 1.0 && al > a0 && al <= L && al < best) {
          best = al;
          bf = f;
          bs = s;
          bt = t;
        }
      }
    }
    if (bf < 0) break;
    const int info = __ldg(m.finfo + 6 * (size_t)e + bf);
    const int bc = finfo_bc(info);
    if (bc == PT_BC_MORTAR) {
      mortar_enter<G, CLIP>(m, k, __ldg(m.fnbr + 6 * (size_t)e + bf), bs, bt, xs, td, n1, n2, L,
                            a0, best, e, fin, a0, st);
      tc.cross++;
    } else if (bc == PT_BC_INTERNAL || bc == PT_BC_PERIODIC) {
      if (bc == PT_BC_PERIODIC) {
        const double* sh = m.shift + 18 * (size_t)e + 3 * bf;
#pragma unroll
        for (int r = 0; r < 3; ++r) {
          xs[r] += __ldg(sh + r);
          xe[r] += __ldg(sh + r);
        }
      }
      fin = finfo_nf(info);
      e = __ldg(m.fnbr + 6 * (size_t)e + bf);
      a0 = best;
      tc.cross++;
    } else if (bc == PT_BC_WALL) {
      double ps[3], pt[3], nrm[3];
      const int kind = finfo_kind(info);
      if (kind == PT_FACE_CURVED) {
        double p[3];
        face_eval<G>(X64, bf, bs, bt, k, p, ps, pt);
      } else {
        const double* Bf = m.bil + 72 * (size_t)e + 12 * bf;
#pragma unroll
        for (int r = 0; r < 3; ++r) {
          ps[r] = __ldg(Bf + r) * bt + __ldg(Bf + 3 + r);
          pt[r] = __ldg(Bf + r) * bs + __ldg(Bf + 6 + r);
        }
      }
      cross3d(ps, pt, nrm);
      const double inn = 1.0 / sqrt(dot3d(nrm, nrm));
#pragma unroll
      for (int r = 0; r < 3; ++r) nrm[r] *= inn;
      double xh[3];
#pragma unroll
      for (int r = 0; r < 3; ++r) xh[r] = xs[r] + best * td[r];
      double Lr = L - best;
      double sdt = 2.0 * dot3d(td, nrm);
#pragma unroll
      for (int r = 0; r < 3; ++r) td[r] -= sdt * nrm[r];
      reflect3(v, nrm);
      reflect3(kx, nrm);
      reflect3(kv, nrm);
#pragma unroll
      for (int r = 0; r < 3; ++r) {
        xs[r] = xh[r];
        xe[r] = xs[r] + Lr * td[r];
      }
      L = Lr;
      a0 = 0.0;
      fin = bf;
      hits++;
      tc.hits++;
      // the frame follows the new direction
      double ax[3] = {0, 0, 0};
      int im = 0;
      if (fabs(td[1]) < fabs(td[im])) im = 1;
      if (fabs(td[2]) < fabs(td[im])) im = 2;
      ax[im] = 1.0;
      cross3d(td, ax, n1);
      const double in1 = 1.0 / sqrt(dot3d(n1, n1));
#pragma unroll
      for (int r = 0; r < 3; ++r) n1[r] *= in1;
      cross3d(td, n1, n2);
      // and so do the FP32 copies that the slab test and the screen use
#pragma unroll
      for (int r = 0; r < 3; ++r) {
        tdf[r] = (float)td[r];
        n1f[r] = (float)n1[r];
        n2f[r] = (float)n2[r];
      }
      Lf = (float)L;
      if (!(L > 0.0)) break;
    } else {
#pragma unroll
      for (int r = 0; r < 3; ++r) x[r] = xs[r] + best * td[r];
      st |= PT_ST_OPEN;
      return;
    }
  }
  if (ncr >= k.max_cross) st |= PT_ST_CROSS_CAP;
#pragma unroll
  for (int r = 0; r < 3; ++r) x[r] = xe[r];
}

}  // namespace pt
