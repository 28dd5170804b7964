// lgt_anchor.cuh -- the anchored polishing sweeps (overrelaxation; the same scheme by
// stochastic relaxation: lgt_anchor_sr.cuh).
//
// After promotion the field U' (FP64) is already close to the gauge-fixed
// field.  The anchored polish keeps U' fixed and relaxes the gauge
// transformation G(x) = 1 + D(x) alone.  With every other G fixed, the local
// maximisation at x sees
//     K(x) = G(x) M(x),   M(x) = sum_mu U'_mu(x) G(x+mu)^+ + U'_mu(x-mu)^+ G(x-mu)^+,
// which is exactly the K(x) that the relaxation sweep of Sec. 3 would gather
// from the transformed links G U' G^+; the update G(x) <- g(x) G(x) is the
// update U_mu(x) <- g U_mu(x), U_mu(x-mu) <- U_mu(x-mu) g^+ of those links.  So
// these are the paper's sweeps with the transformation kept apart from the
// links, which allows each term to be stored at the precision it needs:
//   * M = K0 + C with the constant K0(x) = sum_mu U'_mu(x) + U'_mu(x-mu)^+,
//     formed once in FP64 and kept as its Hermitian part (FP32) and its
//     anti-Hermitian part A0 (FP32 pairs), and the small
//     C(x) = sum_mu U'_mu(x) D(x+mu)^+ + U'_mu(x-mu)^+ D(x-mu)^+, which FP32
//     resolves to |D| 2^-24 from FP32 copies of U' and the high parts of D;
//   * K = M + D(x) M with the small product in FP32, its roundings kept at the size of
//     the sum C + D M, not of the terms that cancel in it (anchor_K);
//   * the rotation angles in FP32.  What must be resolved near the maximum is the
//     anti-Hermitian part of K (theta and the vector part of every subgroup's
//     quaternion are differences of its entries), so it is carried apart as the
//     small number it is, from A0 through the subgroup steps, its 9 reals with their
//     roundings (two_sum), where holding all of K in pairs spent a pair addition (11
//     operations) on each of 18 entries at every stage; the Hermitian part
//     gives the quaternion's scalar part, which FP32 rounds anyway.  Against an
//     all-FP64 polish of the same field the sweeps end 0.86 times as far off as with
//     all of K in pairs (rms over 40 fields of 8^3 x 6 to 34^4, both gauges, 6 to 20
//     sweeps; A in plain FP32 with the terms of T rounded at their own size: 1.29
//     times) and take 67 us per 32^4 half-sweep against 83 (plain FP32: 64);
//   * each SU(2) element in FP32 near-identity form (unit to ~|r|^2 2^-24) and
//     delta = g - 1 in FP32 from the small quantities (error ~|delta| 2^-24);
//   * D <- D + delta + delta D accumulated as an FP32 pair, so G stays unitary
//     to ~1e-10 over a polish (what its rounding per update sums to), far below
//     the ~1e-7 violations that theta < 1e-14 resolves; the field is formed as
//     G U' G^+ in FP64 with G orthonormalised in FP64, an exact gauge transform
//     of the input whatever G's rounding.
// Per site update the sweep reads K0 (112 B), 8 FP32 links (384 B), the high
// parts of 8 neighbours' D (384 B, each neighbour's read by 8 sites, so 48 B
// of compulsory traffic) and its own D (96 B), and writes its own D (96 B):
// 736 B of compulsory traffic; no link is written.
#pragma once

#include "lgt_device.cuh"
#include "lgt_pair.cuh"

namespace lgt {

// Row 2 of G = 1 + D from rows 0 and 1 (G in SU(3)): G_2 = conj(G_0 x G_1)
// with G_0 = e_0 + D_0 and G_1 = e_1 + D_1, hence
//   D_2 = conj(e_0 x D_1 + D_0 x e_1 + D_0 x D_1)
//       = conj((-D_02, -D_12, D_00 + D_11) + D_0 x D_1),
// formed from the small entries only (error relative to |D|).
__device__ __forceinline__ void small_row2(float d[18]) {
#pragma unroll
  for (int k = 0; k < 3; k++) {
    const int a = (k + 1) % 3, b = (k + 2) % 3;
    const float lre = k == 0 ? -d[LGT_RE(0, 2)] : (k == 1 ? -d[LGT_RE(1, 2)] : d[LGT_RE(0, 0)] + d[LGT_RE(1, 1)]);
    const float lim = k == 0 ? d[LGT_IM(0, 2)] : (k == 1 ? d[LGT_IM(1, 2)] : -d[LGT_IM(0, 0)] - d[LGT_IM(1, 1)]);
    float re = d[LGT_RE(0, a)] * d[LGT_RE(1, b)];
    float im = -d[LGT_RE(0, a)] * d[LGT_IM(1, b)];
    re = fmaf(-d[LGT_IM(0, a)], d[LGT_IM(1, b)], re);
    im = fmaf(-d[LGT_IM(0, a)], d[LGT_RE(1, b)], im);
    re = fmaf(-d[LGT_RE(0, b)], d[LGT_RE(1, a)], re);
    im = fmaf(d[LGT_RE(0, b)], d[LGT_IM(1, a)], im);
    re = fmaf(d[LGT_IM(0, b)], d[LGT_IM(1, a)], re);
    im = fmaf(d[LGT_IM(0, b)], d[LGT_RE(1, a)], im);
    d[LGT_RE(2, k)] = lre + re;
    d[LGT_IM(2, k)] = lim + im;
  }
}

// The same in pair arithmetic (D need not be small: a context may be promoted
// far from convergence).
__device__ __forceinline__ void small_row2_pair(f2 d[18]) {
  f2 cre[3], cim[3];
#pragma unroll
  for (int k = 0; k < 3; k++) {
    const int k1 = (k + 1) % 3, k2 = (k + 2) % 3;
    const f2 ar1 = d[LGT_RE(0, k1)], ai1 = d[LGT_IM(0, k1)], ar2 = d[LGT_RE(0, k2)], ai2 = d[LGT_IM(0, k2)];
    const f2 br1 = d[LGT_RE(1, k1)], bi1 = d[LGT_IM(1, k1)], br2 = d[LGT_RE(1, k2)], bi2 = d[LGT_IM(1, k2)];
    // a_k1 b_k2 - a_k2 b_k1
    cre[k] = pair_dot4(ar1, br2, pair_neg(ai1), bi2, pair_neg(ar2), br1, ai2, bi1);
    cim[k] = pair_dot4(ar1, bi2, ai1, br2, pair_neg(ar2), bi1, pair_neg(ai2), br1);
  }
  const f2 lre[3] = {pair_neg(d[LGT_RE(0, 2)]), pair_neg(d[LGT_RE(1, 2)]), pair_add(d[LGT_RE(0, 0)], d[LGT_RE(1, 1)])};
  const f2 lim[3] = {pair_neg(d[LGT_IM(0, 2)]), pair_neg(d[LGT_IM(1, 2)]), pair_add(d[LGT_IM(0, 0)], d[LGT_IM(1, 1)])};
#pragma unroll
  for (int k = 0; k < 3; k++) {
    d[LGT_RE(2, k)] = pair_add(lre[k], cre[k]);
    d[LGT_IM(2, k)] = pair_neg(pair_add(lim[k], cim[k]));
  }
}

// D = G - 1: rows 0 and 1 as FP32 pairs; the high parts in one array and the
// low parts in a second, each laid out as the G of the bulk phase (chunk k of
// parity p at (p * 3 + k) * vh + i), so a neighbour's term reads 48 B.
struct DIO {
  static __device__ __forceinline__ size_t lo_offset(int vh) { return (size_t)6 * vh; }
  static __device__ __forceinline__ void load_pair(const void *base, int vh, int p, int i, f2 d[18]) {
    const float4 *h4 = reinterpret_cast<const float4 *>(base) + (size_t)(p * 3) * vh + i;
    const float4 *l4 = h4 + lo_offset(vh);
#pragma unroll
    for (int k = 0; k < 3; k++) {
      const float4 h = __ldg(h4 + (size_t)k * vh), l = __ldg(l4 + (size_t)k * vh);
      d[4 * k] = {h.x, l.x};
      d[4 * k + 1] = {h.y, l.y};
      d[4 * k + 2] = {h.z, l.z};
      d[4 * k + 3] = {h.w, l.w};
    }
    small_row2_pair(d);
  }
  static __device__ __forceinline__ void store_pair(void *base, int vh, int p, int i, const f2 d[18]) {
    float4 *h4 = reinterpret_cast<float4 *>(base) + (size_t)(p * 3) * vh + i;
    float4 *l4 = h4 + lo_offset(vh);
#pragma unroll
    for (int k = 0; k < 3; k++) {
      h4[(size_t)k * vh] = make_float4(d[4 * k].hi, d[4 * k + 1].hi, d[4 * k + 2].hi, d[4 * k + 3].hi);
      l4[(size_t)k * vh] = make_float4(d[4 * k].lo, d[4 * k + 1].lo, d[4 * k + 2].lo, d[4 * k + 3].lo);
    }
  }
};

// K0(x) as its Hermitian part H (FP32) and its anti-Hermitian part A (FP32 pairs),
// 28 floats in 7 float4 chunks (chunk c of parity p at (p * 7 + c) * vh + i):
//   0: H_00 H_11 H_22 (less anchor_diag) and Im A_00     1: Im A_11 Im A_22 H_01    2: H_02 H_12
//   3: A_01 A_02                      4: A_12, low Im A_00 Im A_11
//   5: low Im A_22, low A_01, low Re A_02   6: low Im A_02, low A_12, tau
// A is the traceless part: Im tr K0, which is not small, drops out of theta and of
// every rotation; tau = Im tr K0 / 3 is kept for the products with K0.
struct AnchorK0 {
  float h[3];     // H_aa - anchor_diag
  float ho[6];    // H_01, H_02, H_12 (re, im)
  float ad[3];    // Im A_aa
  float ao[6];    // A_01, A_02, A_12 (re, im)
  float adl[3], aol[6];  // low parts
  float tau;             // Im tr K0 / 3
};
// H_aa is stored less this constant, near which it lies on a field near its maximum
// (8 or 6 links of Re tr U / 3 ~ 0.8 to 0.95): 2 bits or more for its rounding.
__host__ __device__ constexpr float anchor_diag(int gauge) { return gauge == GAUGE_COULOMB ? 5.0f : 6.5f; }
struct K0IO {
  // EARLY: before the wait for the launch before (relaxed at GPU scope, as ld_early)
  template <bool EARLY>
  static __device__ __forceinline__ void load(const void *base, int vh, int p, int i, AnchorK0 &k) {
    const float4 *b = reinterpret_cast<const float4 *>(base) + (size_t)(p * 7) * vh + i;
    float4 v[7];
#pragma unroll
    for (int c = 0; c < 7; c++) {
      if constexpr (EARLY)
        asm volatile("ld.relaxed.gpu.global.L1::no_allocate.v4.f32 {%0,%1,%2,%3}, [%4];"
                     : "=f"(v[c].x), "=f"(v[c].y), "=f"(v[c].z), "=f"(v[c].w)
                     : "l"(b + (size_t)c * vh)
                     : "memory");
      else v[c] = __ldcs(b + (size_t)c * vh);
    }
    k.h[0] = v[0].x, k.h[1] = v[0].y, k.h[2] = v[0].z, k.ad[0] = v[0].w;
    k.ad[1] = v[1].x, k.ad[2] = v[1].y, k.ho[0] = v[1].z, k.ho[1] = v[1].w;
    k.ho[2] = v[2].x, k.ho[3] = v[2].y, k.ho[4] = v[2].z, k.ho[5] = v[2].w;
    k.ao[0] = v[3].x, k.ao[1] = v[3].y, k.ao[2] = v[3].z, k.ao[3] = v[3].w;
    k.ao[4] = v[4].x, k.ao[5] = v[4].y, k.adl[0] = v[4].z, k.adl[1] = v[4].w;
    k.adl[2] = v[5].x, k.aol[0] = v[5].y, k.aol[1] = v[5].z, k.aol[2] = v[5].w;
    k.aol[3] = v[6].x, k.aol[4] = v[6].y, k.aol[5] = v[6].z, k.tau = v[6].w;
  }
  // from K0 in FP64
  static __device__ __forceinline__ void store(void *base, int vh, int p, int i, const double K[18], float h0) {
    float4 *b = reinterpret_cast<float4 *>(base) + (size_t)(p * 7) * vh + i;
    float f[28];
    auto pair = [&](int hi, int lo, double v) {
      f[hi] = __double2float_rn(v);
      f[lo] = __double2float_rn(v - (double)f[hi]);
    };
    const int ad[3] = {3, 4, 5}, adl[3] = {18, 19, 20};
    const double tau = (K[LGT_IM(0, 0)] + K[LGT_IM(1, 1)] + K[LGT_IM(2, 2)]) * (1.0 / 3.0);
#pragma unroll
    for (int a = 0; a < 3; a++) {
      f[a] = __double2float_rn(K[LGT_RE(a, a)] - (double)h0);
      pair(ad[a], adl[a], K[LGT_IM(a, a)] - tau);
    }
#pragma unroll
    for (int n = 0; n < 3; n++) {  // (0,1), (0,2), (1,2)
      const int a = n == 2 ? 1 : 0, c = n == 0 ? 1 : 2;
      f[6 + 2 * n] = __double2float_rn(0.5 * (K[LGT_RE(a, c)] + K[LGT_RE(c, a)]));
      f[7 + 2 * n] = __double2float_rn(0.5 * (K[LGT_IM(a, c)] - K[LGT_IM(c, a)]));
      pair(12 + 2 * n, 21 + 2 * n, 0.5 * (K[LGT_RE(a, c)] - K[LGT_RE(c, a)]));
      pair(13 + 2 * n, 22 + 2 * n, 0.5 * (K[LGT_IM(a, c)] + K[LGT_IM(c, a)]));
    }
    f[27] = __double2float_rn(tau);
#pragma unroll
    for (int c = 0; c < 7; c++) b[(size_t)c * vh] = make_float4(f[4 * c], f[4 * c + 1], f[4 * c + 2], f[4 * c + 3]);
  }
};

// c += a b^+
__device__ __forceinline__ void acc_mul_dag(const float a[18], const float b[18], float c[18]) {
#pragma unroll
  for (int i = 0; i < 3; i++)
#pragma unroll
    for (int j = 0; j < 3; j++) {
      float re = 0.0f, im = 0.0f;
#pragma unroll
      for (int k = 0; k < 3; k++) {  // a_ik conj(b_jk)
        re = k ? fmaf(a[LGT_RE(i, k)], b[LGT_RE(j, k)], re) : a[LGT_RE(i, k)] * b[LGT_RE(j, k)];
        im = k ? fmaf(a[LGT_IM(i, k)], b[LGT_RE(j, k)], im) : a[LGT_IM(i, k)] * b[LGT_RE(j, k)];
        re = fmaf(a[LGT_IM(i, k)], b[LGT_IM(j, k)], re);
        im = fmaf(-a[LGT_RE(i, k)], b[LGT_IM(j, k)], im);
      }
      c[LGT_RE(i, j)] += re;
      c[LGT_IM(i, j)] += im;
    }
}

// c += a^+ b^+ = (b a)^+
__device__ __forceinline__ void acc_dag_mul_dag(const float a[18], const float b[18], float c[18]) {
#pragma unroll
  for (int i = 0; i < 3; i++)
#pragma unroll
    for (int j = 0; j < 3; j++) {
      float re = 0.0f, im = 0.0f;
#pragma unroll
      for (int k = 0; k < 3; k++) {  // b_jk a_ki
        re = k ? fmaf(b[LGT_RE(j, k)], a[LGT_RE(k, i)], re) : b[LGT_RE(j, k)] * a[LGT_RE(k, i)];
        im = k ? fmaf(b[LGT_RE(j, k)], a[LGT_IM(k, i)], im) : b[LGT_RE(j, k)] * a[LGT_IM(k, i)];
        re = fmaf(-b[LGT_IM(j, k)], a[LGT_IM(k, i)], re);
        im = fmaf(b[LGT_IM(j, k)], a[LGT_RE(k, i)], im);
      }
      c[LGT_RE(i, j)] += re;
      c[LGT_IM(i, j)] -= im;
    }
}

// x <- x + t, the rounding kept in x.lo (not renormalised: x is hi + lo)
__device__ __forceinline__ void small_add(f2 &x, float t) {
  const f2 s = two_sum(x.hi, t);
  x = {s.hi, __fadd_rn(x.lo, s.lo)};
}
// x - y in one float
__device__ __forceinline__ float small_diff(f2 x, f2 y) {
  const f2 s = two_sum(x.hi, -y.hi);
  return __fadd_rn(s.hi, __fadd_rn(s.lo, __fsub_rn(x.lo, y.lo)));
}

// K(x) = M + D M of the anchored polish, M = K0 + C: all of it as floats (W), and
// its anti-Hermitian part apart (see above).
struct AnchorK {
  float W[18];
  float wd[3];      // Re W_aa - anchor_diag
  f2 ad[3], ao[6];  // Im A_aa (less tau); A_01, A_02, A_12
};
// h0: anchor_diag
__device__ __forceinline__ void anchor_K(const AnchorK0 &k0, float h0, const float C[18], const float dh[18], AnchorK &K) {
  // K0 + X as floats: the small parts are summed first, so that each entry takes one
  // rounding at its size
  auto add_k0 = [&](const float X[18], float Y[18]) {
#pragma unroll
    for (int a = 0; a < 3; a++) {
      Y[LGT_RE(a, a)] = h0 + (k0.h[a] + X[LGT_RE(a, a)]);
      Y[LGT_IM(a, a)] = k0.tau + (k0.ad[a] + X[LGT_IM(a, a)]);
    }
#pragma unroll
    for (int n = 0; n < 3; n++) {
      const int a = n == 2 ? 1 : 0, c = n == 0 ? 1 : 2;
      Y[LGT_RE(a, c)] = k0.ho[2 * n] + (k0.ao[2 * n] + X[LGT_RE(a, c)]);
      Y[LGT_IM(a, c)] = k0.ho[2 * n + 1] + (k0.ao[2 * n + 1] + X[LGT_IM(a, c)]);
      Y[LGT_RE(c, a)] = k0.ho[2 * n] + (X[LGT_RE(c, a)] - k0.ao[2 * n]);
      Y[LGT_IM(c, a)] = (k0.ao[2 * n + 1] + X[LGT_IM(c, a)]) - k0.ho[2 * n + 1];
    }
  };
  float M[18], T[18];
  add_k0(C, M);
  // T = C + D M = K - K0.  The large entries of M are its diagonal's real parts, and
  // D times them nearly cancels C where D is smooth: that product is added to C in one
  // rounding of their sum, and the other products, small, are summed apart, with D
  // times what the diagonal's rounding left (low).
  float low[3];
#pragma unroll
  for (int a = 0; a < 3; a++) low[a] = (k0.h[a] + C[LGT_RE(a, a)]) - (M[LGT_RE(a, a)] - h0);
#pragma unroll
  for (int a = 0; a < 3; a++)
#pragma unroll
    for (int c = 0; c < 3; c++) {
      float re = dh[LGT_RE(a, c)] * low[c], im = dh[LGT_IM(a, c)] * low[c];
      re = fmaf(-dh[LGT_IM(a, c)], M[LGT_IM(c, c)], re);
      im = fmaf(dh[LGT_RE(a, c)], M[LGT_IM(c, c)], im);
#pragma unroll
      for (int d = 1; d < 3; d++) {
        const int k = (c + d) % 3;
        re = fmaf(dh[LGT_RE(a, k)], M[LGT_RE(k, c)], re);
        im = fmaf(dh[LGT_RE(a, k)], M[LGT_IM(k, c)], im);
        re = fmaf(-dh[LGT_IM(a, k)], M[LGT_IM(k, c)], re);
        im = fmaf(dh[LGT_IM(a, k)], M[LGT_RE(k, c)], im);
      }
      T[LGT_RE(a, c)] = fmaf(dh[LGT_RE(a, c)], M[LGT_RE(c, c)], C[LGT_RE(a, c)]) + re;
      T[LGT_IM(a, c)] = fmaf(dh[LGT_IM(a, c)], M[LGT_RE(c, c)], C[LGT_IM(a, c)]) + im;
    }
  add_k0(T, K.W);
#pragma unroll
  for (int a = 0; a < 3; a++) K.wd[a] = k0.h[a] + T[LGT_RE(a, a)];
#pragma unroll
  for (int a = 0; a < 3; a++) K.ad[a] = {k0.ad[a], k0.adl[a]}, small_add(K.ad[a], T[LGT_IM(a, a)]);
#pragma unroll
  for (int n = 0; n < 3; n++) {
    const int a = n == 2 ? 1 : 0, c = n == 0 ? 1 : 2;
    K.ao[2 * n] = {k0.ao[2 * n], k0.aol[2 * n]};
    K.ao[2 * n + 1] = {k0.ao[2 * n + 1], k0.aol[2 * n + 1]};
    small_add(K.ao[2 * n], 0.5f * T[LGT_RE(a, c)]), small_add(K.ao[2 * n], -0.5f * T[LGT_RE(c, a)]);
    small_add(K.ao[2 * n + 1], 0.5f * T[LGT_IM(a, c)]), small_add(K.ao[2 * n + 1], 0.5f * T[LGT_IM(c, a)]);
  }
}

// Re tr K and tr[Delta Delta^dagger], Delta the traceless part of (K - K^+)/(2i)
__device__ __forceinline__ void anchor_violation(const AnchorK &K, float &retr, float &delta2) {
  retr = K.W[LGT_RE(0, 0)] + K.W[LGT_RE(1, 1)] + K.W[LGT_RE(2, 2)];
  const float ad[3] = {pair_to_float(K.ad[0]), pair_to_float(K.ad[1]), pair_to_float(K.ad[2])};
  const float tr3 = (ad[0] + ad[1] + ad[2]) * (1.0f / 3.0f);
  float s = 0.0f, t = 0.0f;
#pragma unroll
  for (int a = 0; a < 3; a++) s = fmaf(ad[a] - tr3, ad[a] - tr3, s);
#pragma unroll
  for (int e = 0; e < 6; e++) t = fmaf(pair_to_float(K.ao[e]), pair_to_float(K.ao[e]), t);
  delta2 = fmaf(2.0f, t, s);
}

// Sec. 3 local update for the anchored polish: the quaternions' scalar parts from
// the diagonal, in one rounding of their size, their vector parts from the
// anti-Hermitian part; each subgroup element in FP32 near-identity form (1 + e0, r),
// unit to ~|r|^2 2^-24, i.e. ~1e-15 for the |r| <~ 1e-4 of polishing (only G's
// unitarity depends on it, and G is orthonormalised in FP64 when the field is
// formed).  W <- W + rho W between the subgroups, as far as the later ones see it.
__device__ __forceinline__ void anchor_local_update(AnchorK &K, float h0, RotF rf[3], float omega) {
  float *W = K.W;
  // (0,1)
  RotF r = rf[0] = subgroup_rotation<ALGO_OR>(2.0f * h0 + (K.wd[0] + K.wd[1]), 2.0f * pair_to_float(K.ao[1]), 2.0f * pair_to_float(K.ao[0]),
                                           small_diff(K.ad[0], K.ad[1]), omega, false);
#pragma unroll
  for (int c = 0; c < 3; c++) {
    const float xi = W[LGT_RE(0, c)], yi = W[LGT_IM(0, c)];
    const float xj = W[LGT_RE(1, c)], yj = W[LGT_IM(1, c)];
    const float t0r = r.e0 * xi - r.r3 * yi + r.r2 * xj - r.r1 * yj, t0i = r.e0 * yi + r.r3 * xi + r.r2 * yj + r.r1 * xj;
    W[LGT_RE(0, c)] += t0r;
    W[LGT_IM(0, c)] += t0i;
    if (c == 0) K.wd[0] += t0r, small_add(K.ad[0], t0i);
    if (c == 2) small_add(K.ao[2], 0.5f * t0r), small_add(K.ao[3], 0.5f * t0i);
    if (c > 0) {
      const float t1r = -r.r2 * xi - r.r1 * yi + r.e0 * xj + r.r3 * yj, t1i = -r.r2 * yi + r.r1 * xi + r.e0 * yj - r.r3 * xj;
      if (c == 1) K.wd[1] += t1r, small_add(K.ad[1], t1i);
      else small_add(K.ao[4], 0.5f * t1r), small_add(K.ao[5], 0.5f * t1i);
    }
  }
  // (0,2)
  r = rf[1] = subgroup_rotation<ALGO_OR>(2.0f * h0 + (K.wd[0] + K.wd[2]), 2.0f * pair_to_float(K.ao[3]), 2.0f * pair_to_float(K.ao[2]),
                                      small_diff(K.ad[0], K.ad[2]), omega, false);
#pragma unroll
  for (int c = 1; c < 3; c++) {
    const float xi = W[LGT_RE(0, c)], yi = W[LGT_IM(0, c)];
    const float xj = W[LGT_RE(2, c)], yj = W[LGT_IM(2, c)];
    const float tr = -r.r2 * xi - r.r1 * yi + r.e0 * xj + r.r3 * yj, ti = -r.r2 * yi + r.r1 * xi + r.e0 * yj - r.r3 * xj;
    if (c == 1) small_add(K.ao[4], -0.5f * tr), small_add(K.ao[5], 0.5f * ti);  // A_12 -= conj(t_21) / 2
    else K.wd[2] += tr, small_add(K.ad[2], ti);
  }
  // (1,2)
  rf[2] = subgroup_rotation<ALGO_OR>(2.0f * h0 + (K.wd[1] + K.wd[2]), 2.0f * pair_to_float(K.ao[5]), 2.0f * pair_to_float(K.ao[4]),
                                  small_diff(K.ad[1], K.ad[2]), omega, false);
}

// delta = g - 1 for g = R2 R1 R0 from FP32 near-identity elements, written with
// the small quantities only (the structure of pair_delta, in FP32): error
// ~|delta| 2^-24.
__device__ __forceinline__ void float_delta(const RotF rf[3], float d[18]) {
  // deviation blocks of element s: a = e0 + i r3, B = r2 + i r1, C = -r2 + i r1, d = e0 - i r3
  float ar[3], ai[3], br[3], bi[3], cr[3], ci[3], dr[3], di[3];
#pragma unroll
  for (int s = 0; s < 3; s++) {
    ar[s] = rf[s].e0, ai[s] = rf[s].r3;
    br[s] = rf[s].r2, bi[s] = rf[s].r1;
    cr[s] = -rf[s].r2, ci[s] = rf[s].r1;
    dr[s] = rf[s].e0, di[s] = -rf[s].r3;
  }
  auto mul = [](float xr, float xi, float yr, float yi, float &zr, float &zi) {
    zr = xr * yr - xi * yi;
    zi = xr * yi + xi * yr;
  };
  float t0r, t0i, t1r, t1i;
  // C1 A0 = C1 + C1 a0, C1 B0
  mul(cr[1], ci[1], ar[0], ai[0], t0r, t0i);
  const float c1a0r = cr[1] + t0r, c1a0i = ci[1] + t0i;
  float c1b0r, c1b0i;
  mul(cr[1], ci[1], br[0], bi[0], c1b0r, c1b0i);
  // row 0: A1 A0 - 1, A1 B0, B1
  mul(ar[1], ai[1], ar[0], ai[0], t0r, t0i);
  d[LGT_RE(0, 0)] = (ar[1] + ar[0]) + t0r, d[LGT_IM(0, 0)] = (ai[1] + ai[0]) + t0i;
  mul(ar[1], ai[1], br[0], bi[0], t0r, t0i);
  d[LGT_RE(0, 1)] = br[0] + t0r, d[LGT_IM(0, 1)] = bi[0] + t0i;
  d[LGT_RE(0, 2)] = br[1], d[LGT_IM(0, 2)] = bi[1];
  // row 1: A2 C0 + B2 C1 A0, A2 D0 + B2 C1 B0 - 1, B2 D1
  mul(ar[2], ai[2], cr[0], ci[0], t0r, t0i);
  mul(br[2], bi[2], c1a0r, c1a0i, t1r, t1i);
  d[LGT_RE(1, 0)] = (cr[0] + t0r) + t1r, d[LGT_IM(1, 0)] = (ci[0] + t0i) + t1i;
  mul(ar[2], ai[2], dr[0], di[0], t0r, t0i);
  mul(br[2], bi[2], c1b0r, c1b0i, t1r, t1i);
  d[LGT_RE(1, 1)] = ((ar[2] + dr[0]) + t0r) + t1r, d[LGT_IM(1, 1)] = ((ai[2] + di[0]) + t0i) + t1i;
  mul(br[2], bi[2], dr[1], di[1], t0r, t0i);
  d[LGT_RE(1, 2)] = br[2] + t0r, d[LGT_IM(1, 2)] = bi[2] + t0i;
  // row 2: C2 C0 + D2 C1 A0, C2 D0 + D2 C1 B0, D2 D1 - 1
  mul(cr[2], ci[2], cr[0], ci[0], t0r, t0i);
  mul(dr[2], di[2], c1a0r, c1a0i, t1r, t1i);
  d[LGT_RE(2, 0)] = (t0r + c1a0r) + t1r, d[LGT_IM(2, 0)] = (t0i + c1a0i) + t1i;
  mul(cr[2], ci[2], dr[0], di[0], t0r, t0i);
  mul(dr[2], di[2], c1b0r, c1b0i, t1r, t1i);
  d[LGT_RE(2, 1)] = (cr[2] + t0r) + (c1b0r + t1r), d[LGT_IM(2, 1)] = (ci[2] + t0i) + (c1b0i + t1i);
  mul(dr[2], di[2], dr[1], di[1], t0r, t0i);
  d[LGT_RE(2, 2)] = (dr[2] + dr[1]) + t0r, d[LGT_IM(2, 2)] = (di[2] + di[1]) + t0i;
}

// G <- g G on rows 0 and 1: D <- D + (delta + delta D), D a pair (rows 0, 1), the
// increment in FP32 (dh: D's high parts with row 2)
__device__ __forceinline__ void d_update(f2 D[12], const float dh[18], const float d[18]) {
#pragma unroll
  for (int i = 0; i < 2; i++)
#pragma unroll
    for (int j = 0; j < 3; j++) {
      float re = 0.0f, im = 0.0f;
#pragma unroll
      for (int k = 0; k < 3; k++) {
        re = fmaf(d[LGT_RE(i, k)], dh[LGT_RE(k, j)], re);
        re = fmaf(-d[LGT_IM(i, k)], dh[LGT_IM(k, j)], re);
        im = fmaf(d[LGT_RE(i, k)], dh[LGT_IM(k, j)], im);
        im = fmaf(d[LGT_IM(i, k)], dh[LGT_RE(k, j)], im);
      }
      D[LGT_RE(i, j)] = pair_add(D[LGT_RE(i, j)], f2{d[LGT_RE(i, j)] + re, 0.0f});
      D[LGT_IM(i, j)] = pair_add(D[LGT_IM(i, j)], f2{d[LGT_IM(i, j)] + im, 0.0f});
    }
}

}  // namespace lgt
