// pt_map.cuh -- the element map chi(xi) of the FP32 mode and its inverse
// (Sec. 3.2.1, Eq. dgsem_curvedfaces).
//
// The map of each coordinate is kept as a polynomial in monomials,
//   chi_r = sum_{b,c,a} M_r[b][c][a] xi1^a xi2^b xi3^c,
// converted once from the geometry nodes (k_mono).  Horner's rule needs no
// basis functions, so a point evaluation is G^3 multiply-adds with nothing but
// the point itself in registers; the Lagrange form spent more on the bases in
// double-float (~450 instructions) than on anything else.  Two neighbouring
// powers of xi1 are evaluated per instruction (packed FP32).  The
// conversion can make coefficients larger than the nodes by a factor of 2, 4.5 or
// 10.7 per direction at degree 2, 3 or 4 (its largest row sum), but the elements of
// a smooth mesh have coefficients that fall off with the degree, and the form
// costs no accuracy (conversion in FP64, coefficients split in a high and a low
// FP32 part): error of xi over 10^6 points of the 32^3 channel against 64 bits at
// NGeo 1 / 2 / 3 / 4: 6.8e-15 / 9.1e-15 / 3.2e-14 / 2.4e-14 of xi's norm (3.7e-14 at
// NGeo 3 with the Lagrange form in double-float), at most 6.0e-14 / 8.1e-14 / 1.0e-13 /
// 1.4e-13.  The stage kernel went from 7640 to 3200 instructions
// per warp and stage and from 0.45 to 0.255 ns per particle and stage (10^6
// particles, 32^3, NGeo 2, N 5); point location from 931 to 582 us for 10^6.
#pragma once
#include "pt_df.cuh"
#include "pt_f32x2.cuh"
#include "pt_internal.h"

namespace pt {

// Layout of one coordinate's coefficients: rows of AP floats (xi1 powers,
// padded with zeros to a multiple of 2, or to 4 where 16-byte loads serve it),
// row (b, c) at AP (c + G b), the block CS floats long (a multiple of 4).  A
// coordinate that is trilinear in xi (DevMesh::tmask) holds its 8 coefficients
// in the first 8 floats instead, index a + 2 b + 4 c.
template <int G>
struct Mono {
  static constexpr int AP = G == 3 ? 4 : (G == 5 ? 6 : G);
  static constexpr int NQ = AP / 2;  // packed pairs per row
  static constexpr int CS = (G * G * AP + 3) & ~3;
};

// Read-only load: non-coherent from global memory, or (GEN) generic, for data
// that may sit in shared memory.
template <bool GEN, typename V>
__device__ __forceinline__ V ldx(const V* p) {
  if constexpr (GEN)
    return *p;
  else
    return __ldg(p);
}

// one row as packed pairs
template <int G, bool GEN>
__device__ __forceinline__ void mono_row(const float* __restrict__ p, f32x2* q) {
  if constexpr (Mono<G>::AP == 4) {
    const ulonglong2 w = ldx<GEN>(reinterpret_cast<const ulonglong2*>(p));
    q[0] = w.x;
    q[1] = w.y;
  } else {
#pragma unroll
    for (int i = 0; i < Mono<G>::NQ; ++i) q[i] = ldx<GEN>(reinterpret_cast<const f32x2*>(p) + i);
  }
}

// chi_r and its three derivatives of a trilinear coordinate
template <bool GEN>
__device__ __forceinline__ void mono_tri32(const float* __restrict__ M, const float* xi, float& chi,
                                           float* J) {
  const ulonglong2 q0 = ldx<GEN>(reinterpret_cast<const ulonglong2*>(M));
  const ulonglong2 q1 = ldx<GEN>(reinterpret_cast<const ulonglong2*>(M) + 1);
  const f32x2 z = dup2(xi[2]), y = dup2(xi[1]);
  const f32x2 s0 = fma2(z, q1.x, q0.x), s1 = fma2(z, q1.y, q0.y);  // b = 0, 1
  float u0, u1, v0, v1, w0, w1;
  unpk2(fma2(y, s1, s0), u0, u1);
  unpk2(s1, v0, v1);
  unpk2(fma2(y, q1.y, q1.x), w0, w1);
  chi = fmaf(xi[0], u1, u0);
  J[0] = u1;
  J[1] = fmaf(xi[0], v1, v0);
  J[2] = fmaf(xi[0], w1, w0);
}

// the same for a curved coordinate: Horner in xi3, then xi2 (packed over the
// powers of xi1), then xi1, each with its derivative
template <int G, bool GEN>
__device__ __forceinline__ void mono_curved32(const float* __restrict__ M, const float* xi,
                                              float& chi, float* J) {
  constexpr int AP = Mono<G>::AP, NQ = Mono<G>::NQ;
  const f32x2 z = dup2(xi[2]), y = dup2(xi[1]);
  f32x2 W[NQ], Wy[NQ], Wz[NQ];
#pragma unroll
  for (int b = G - 1; b >= 0; --b) {
    f32x2 row[G][NQ];
#pragma unroll
    for (int c = 0; c < G; ++c) mono_row<G, GEN>(M + AP * (c + G * b), row[c]);
#pragma unroll
    for (int p = 0; p < NQ; ++p) {
      f32x2 V = fma2(row[G - 1][p], z, row[G - 2][p]), D = row[G - 1][p];
#pragma unroll
      for (int c = G - 3; c >= 0; --c) {
        D = fma2(D, z, V);
        V = fma2(V, z, row[c][p]);
      }
      if (b == G - 1) {
        W[p] = V;
        Wz[p] = D;
      } else {
        Wy[p] = b == G - 2 ? W[p] : fma2(Wy[p], y, W[p]);
        W[p] = fma2(W[p], y, V);
        Wz[p] = fma2(Wz[p], y, D);
      }
    }
  }
  float w[AP], wy[AP], wz[AP];
#pragma unroll
  for (int p = 0; p < NQ; ++p) {
    unpk2(W[p], w[2 * p], w[2 * p + 1]);
    unpk2(Wy[p], wy[2 * p], wy[2 * p + 1]);
    unpk2(Wz[p], wz[2 * p], wz[2 * p + 1]);
  }
  float v = w[G - 1], dx = 0.f, dy = wy[G - 1], dz = wz[G - 1];
#pragma unroll
  for (int a = G - 2; a >= 0; --a) {
    dx = a == G - 2 ? v : fmaf(dx, xi[0], v);
    v = fmaf(v, xi[0], w[a]);
    dy = fmaf(dy, xi[0], wy[a]);
    dz = fmaf(dz, xi[0], wz[a]);
  }
  chi = v;
  J[0] = dx;
  J[1] = dy;
  J[2] = dz;
}

// chi and Jacobian J[r][q] = d chi_r / d xi_q in FP32; M: the element's
// coefficients (high parts), tm: its trilinear coordinates
template <int G, bool GEN = false>
__device__ __forceinline__ void map_j32(const float* __restrict__ M, const float* xi, int tm,
                                        float* chi, float* J) {
#pragma unroll
  for (int r = 0; r < 3; ++r) {
    const float* Mr = M + r * Mono<G>::CS;
    if (G == 2 || ((tm >> r) & 1))
      mono_tri32<GEN>(Mr, xi, chi[r], J + 3 * r);
    else if constexpr (G > 2)
      mono_curved32<G, GEN>(Mr, xi, chi[r], J + 3 * r);
  }
}

// One step of the compensated Horner rule (Graillat, Langlois & Louvet 2009):
// (s, e) <- (s, e) z + (h, l), s the FP32 value and e the running compensation,
// from the exact error of the product (TwoProduct) and of the sum (TwoSum);
// zn = -z.  z is one FP32 number, so the rounding of e (about 6e-8 of s's
// rounding) is all that is lost: the value is good to ~2^-47.
__device__ __forceinline__ void comp_step(f32x2& s, f32x2& e, f32x2 z, f32x2 zn, f32x2 h, f32x2 l) {
  const f32x2 q = mul2(s, zn);      // -(s z)
  const f32x2 pe = fma2(s, z, q);   // s z = -q + pe
  const f32x2 t = sub2(h, q);
  const f32x2 bb = sub2(t, h);
  const f32x2 te = sub2(sub2(h, sub2(t, bb)), add2(q, bb));
  e = fma2(e, z, add2(add2(pe, te), l));
  s = t;
}
__device__ __forceinline__ void comp_step(float& s, float& e, float z, float h, float l) {
  const float p = __fmul_rn(s, z);
  const float pe = __fmaf_rn(s, z, -p);
  float t, te;
  two_sum(h, p, t, te);
  e = __fmaf_rn(e, z, __fadd_rn(__fadd_rn(pe, te), l));
  s = t;
}

// chi_r(xi) of one coordinate as s + e, xi three FP32 numbers
template <bool GEN>
__device__ __forceinline__ void comp_tri(const float* __restrict__ Mh, const float* __restrict__ Ml,
                                         const float* xi, float& s, float& e) {
  const ulonglong2 h0 = ldx<GEN>(reinterpret_cast<const ulonglong2*>(Mh));
  const ulonglong2 h1 = ldx<GEN>(reinterpret_cast<const ulonglong2*>(Mh) + 1);
  const ulonglong2 l0 = ldx<GEN>(reinterpret_cast<const ulonglong2*>(Ml));
  const ulonglong2 l1 = ldx<GEN>(reinterpret_cast<const ulonglong2*>(Ml) + 1);
  const f32x2 z = dup2(xi[2]), zn = dup2(-xi[2]), y = dup2(xi[1]), yn = dup2(-xi[1]);
  f32x2 s0 = h1.x, e0 = l1.x, s1 = h1.y, e1 = l1.y;
  comp_step(s0, e0, z, zn, h0.x, l0.x);
  comp_step(s1, e1, z, zn, h0.y, l0.y);
  comp_step(s1, e1, y, yn, s0, e0);
  float a0, a1, b0, b1;
  unpk2(s1, a0, a1);
  unpk2(e1, b0, b1);
  comp_step(a1, b1, xi[0], a0, b0);
  s = a1;
  e = b1;
}

template <int G, bool GEN>
__device__ __forceinline__ void comp_curved(const float* __restrict__ Mh,
                                            const float* __restrict__ Ml, const float* xi,
                                            float& so, float& eo) {
  constexpr int AP = Mono<G>::AP, NQ = Mono<G>::NQ;
  const f32x2 z = dup2(xi[2]), zn = dup2(-xi[2]), y = dup2(xi[1]), yn = dup2(-xi[1]);
  f32x2 S[NQ], E[NQ];
#pragma unroll
  for (int b = G - 1; b >= 0; --b) {
    f32x2 s[NQ], e[NQ];
    mono_row<G, GEN>(Mh + AP * (G - 1 + G * b), s);
    mono_row<G, GEN>(Ml + AP * (G - 1 + G * b), e);
#pragma unroll
    for (int c = G - 2; c >= 0; --c) {
      f32x2 h[NQ], l[NQ];
      mono_row<G, GEN>(Mh + AP * (c + G * b), h);
      mono_row<G, GEN>(Ml + AP * (c + G * b), l);
#pragma unroll
      for (int p = 0; p < NQ; ++p) comp_step(s[p], e[p], z, zn, h[p], l[p]);
    }
#pragma unroll
    for (int p = 0; p < NQ; ++p) {
      if (b == G - 1) {
        S[p] = s[p];
        E[p] = e[p];
      } else {
        comp_step(S[p], E[p], y, yn, s[p], e[p]);
      }
    }
  }
  float w[AP], f[AP];
#pragma unroll
  for (int p = 0; p < NQ; ++p) {
    unpk2(S[p], w[2 * p], w[2 * p + 1]);
    unpk2(E[p], f[2 * p], f[2 * p + 1]);
  }
  so = w[G - 1];
  eo = f[G - 1];
#pragma unroll
  for (int a = G - 2; a >= 0; --a) comp_step(so, eo, xi[0], w[a], f[a]);
}

// Residual chi(xi) - x at an FP32 point xi, x a double-float; the difference
// of the high parts is exact where they agree to a factor of two, which is
// where the residual's accuracy counts.
template <int G, bool GEN = false>
__device__ __forceinline__ void resid_df(const float* __restrict__ Mh, const float* __restrict__ Ml,
                                         const float* xi, int tm, const df* x, float* r) {
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    const float* h = Mh + q * Mono<G>::CS;
    const float* l = Ml + q * Mono<G>::CS;
    float s = 0.f, e = 0.f;
    if (G == 2 || ((tm >> q) & 1))
      comp_tri<GEN>(h, l, xi, s, e);
    else if constexpr (G > 2)
      comp_curved<G, GEN>(h, l, xi, s, e);
    r[q] = __fadd_rn(__fsub_rn(s, x[q].hi), __fsub_rn(e, x[q].lo));
  }
}

}  // namespace pt
