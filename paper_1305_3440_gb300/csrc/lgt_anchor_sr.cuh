// lgt_anchor_sr.cuh -- the anchored polish by stochastic relaxation.
//
// The scheme of lgt_anchor.cuh with all of K(x) held in FP32 pairs, K0 too (144 B
// per site), and the terms of C(x) added direction by direction.  Stochastic
// relaxation's squared steps amplify the rounding of its FP32 angles over a polish
// (an all-FP64 polish of the same field ends 1e-9 to 1e-7 away after 20 sweeps at a
// violation of 1e-4), so another order of rounding ends elsewhere within that
// distance.  The body with the anti-Hermitian part apart is no further from 64 bits
// and 20% faster, but it is not this one's result: the sweeps that users have run
// keep theirs.  Overrelaxation contracts rounding (1e-10) and takes the faster body.
// Issue-bound: 83 us per 32^4 half-sweep (configuration 11).
#pragma once

#include "lgt_anchor.cuh"
#include "lgt_sweep.cuh"

namespace lgt {
namespace anchor_sr {

// row 2 of D = G - 1 from rows 0 and 1 through the small entries (lgt_anchor.cuh)
__device__ __forceinline__ void small_row2(float d[18]) {
  float cre[3], cim[3];
#pragma unroll
  for (int k = 0; k < 3; k++) {
    const int k1 = (k + 1) % 3, k2 = (k + 2) % 3;
    const float ar1 = d[LGT_RE(0, k1)], ai1 = d[LGT_IM(0, k1)], ar2 = d[LGT_RE(0, k2)], ai2 = d[LGT_IM(0, k2)];
    const float br1 = d[LGT_RE(1, k1)], bi1 = d[LGT_IM(1, k1)], br2 = d[LGT_RE(1, k2)], bi2 = d[LGT_IM(1, k2)];
    cre[k] = (ar1 * br2 - ai1 * bi2) - (ar2 * br1 - ai2 * bi1);
    cim[k] = (ar1 * bi2 + ai1 * br2) - (ar2 * bi1 + ai2 * br1);
  }
  const float lre[3] = {-d[LGT_RE(0, 2)], -d[LGT_RE(1, 2)], d[LGT_RE(0, 0)] + d[LGT_RE(1, 1)]};
  const float lim[3] = {-d[LGT_IM(0, 2)], -d[LGT_IM(1, 2)], d[LGT_IM(0, 0)] + d[LGT_IM(1, 1)]};
#pragma unroll
  for (int k = 0; k < 3; k++) {
    d[LGT_RE(2, k)] = lre[k] + cre[k];
    d[LGT_IM(2, k)] = -(lim[k] + cim[k]);
  }
}

// D's high parts (row 2 rebuilt), and rows 0, 1 of D as pairs
__device__ __forceinline__ void load_hi(const void *base, int vh, int p, int i, float d[18]) {
  const float4 *b4 = reinterpret_cast<const float4 *>(base) + (size_t)(p * 3) * vh + i;
#pragma unroll
  for (int k = 0; k < 3; k++) {
    const float4 v = __ldg(b4 + (size_t)k * vh);
    d[4 * k] = v.x;
    d[4 * k + 1] = v.y;
    d[4 * k + 2] = v.z;
    d[4 * k + 3] = v.w;
  }
  small_row2(d);
}

__device__ __forceinline__ void load_pair_rows(const void *base, int vh, int p, int i, f2 d[12]) {
  const float4 *h4 = reinterpret_cast<const float4 *>(base) + (size_t)(p * 3) * vh + i;
  const float4 *l4 = h4 + DIO::lo_offset(vh);
#pragma unroll
  for (int k = 0; k < 3; k++) {
    const float4 h = __ldg(h4 + (size_t)k * vh), l = __ldg(l4 + (size_t)k * vh);
    d[4 * k] = {h.x, l.x};
    d[4 * k + 1] = {h.y, l.y};
    d[4 * k + 2] = {h.z, l.z};
    d[4 * k + 3] = {h.w, l.w};
  }
}

// K0(x): one 3x3 complex matrix per site as FP32 pairs, 9 float4 chunks
// (chunk c of parity p at (p * 9 + c) * vh + i).
struct K0IO {
  static __device__ __forceinline__ void load(const void *base, int vh, int p, int i, f2 m[18]) {
    const float4 *b = reinterpret_cast<const float4 *>(base) + (size_t)(p * 9) * vh + i;
#pragma unroll
    for (int c = 0; c < 9; c++) {
      const float4 v = __ldg(b + (size_t)c * vh);
      m[2 * c] = {v.x, v.y};
      m[2 * c + 1] = {v.z, v.w};
    }
  }
  static __device__ __forceinline__ void store(void *base, int vh, int p, int i, const f2 m[18]) {
    float4 *b = reinterpret_cast<float4 *>(base) + (size_t)(p * 9) * vh + i;
#pragma unroll
    for (int c = 0; c < 9; c++)
      b[(size_t)c * vh] = make_float4(m[2 * c].hi, m[2 * c].lo, m[2 * c + 1].hi, m[2 * c + 1].lo);
  }
};

// c += a b^+, each product added as it comes (lgt_anchor.cuh forms the entry first)
__device__ __forceinline__ void acc_mul_dag(const float a[18], const float b[18], float c[18]) {
#pragma unroll
  for (int i = 0; i < 3; i++)
#pragma unroll
    for (int j = 0; j < 3; j++) {
      float re = c[LGT_RE(i, j)], im = c[LGT_IM(i, j)];
#pragma unroll
      for (int k = 0; k < 3; k++) {  // a_ik conj(b_jk)
        re += a[LGT_RE(i, k)] * b[LGT_RE(j, k)] + a[LGT_IM(i, k)] * b[LGT_IM(j, k)];
        im += a[LGT_IM(i, k)] * b[LGT_RE(j, k)] - a[LGT_RE(i, k)] * b[LGT_IM(j, k)];
      }
      c[LGT_RE(i, j)] = re;
      c[LGT_IM(i, j)] = im;
    }
}

// c += a^+ b^+ = (b a)^+
__device__ __forceinline__ void acc_dag_mul_dag(const float a[18], const float b[18], float c[18]) {
#pragma unroll
  for (int i = 0; i < 3; i++)
#pragma unroll
    for (int j = 0; j < 3; j++) {
      float re = c[LGT_RE(i, j)], im = c[LGT_IM(i, j)];
#pragma unroll
      for (int k = 0; k < 3; k++) {  // conj(a_ki) conj(b_jk) = conj(b_jk a_ki)
        re += b[LGT_RE(j, k)] * a[LGT_RE(k, i)] - b[LGT_IM(j, k)] * a[LGT_IM(k, i)];
        im -= b[LGT_RE(j, k)] * a[LGT_IM(k, i)] + b[LGT_IM(j, k)] * a[LGT_RE(k, i)];
      }
      c[LGT_RE(i, j)] = re;
      c[LGT_IM(i, j)] = im;
    }
}

// Sec. 3 local update: the block projections from the pair-precision K, the
// rotation angles and each subgroup element in FP32 near-identity form.
__device__ __forceinline__ void local_update_pair(f2 W[18], RotF rf[3], float omega, uint64_t sr_thr, uint4 draws) {
#pragma unroll
  for (int s = 0; s < 3; s++) {
    const int i = (s == 2) ? 1 : 0;
    const int j = (s == 0) ? 1 : 2;
    const float q0 = pair_to_float(pair_add(W[LGT_RE(i, i)], W[LGT_RE(j, j)]));
    const float q1 = pair_to_float(pair_add(W[LGT_IM(i, j)], W[LGT_IM(j, i)]));
    const float q2 = pair_to_float(pair_add(W[LGT_RE(i, j)], pair_neg(W[LGT_RE(j, i)])));
    const float q3 = pair_to_float(pair_add(W[LGT_IM(i, i)], pair_neg(W[LGT_IM(j, j)])));
    const uint32_t d = s == 0 ? draws.x : (s == 1 ? draws.y : draws.z);
    rf[s] = subgroup_rotation<ALGO_SR>(q0, q1, q2, q3, omega, (uint64_t)d < sr_thr);
    if (s == 0) steer_rows<0, 1>(W, rf[s]);
    if (s == 1) steer_rows<0, 2>(W, rf[s]);
  }
}

// G <- g G on rows 0 and 1: D <- D + delta + delta D, D a pair (rows 0, 1),
// delta and the small product delta D in FP32 (dh: D's high parts with row 2)
__device__ __forceinline__ void d_update_lite(f2 D[12], const float dh[18], const float d[18]) {
#pragma unroll
  for (int i = 0; i < 2; i++)
#pragma unroll
    for (int j = 0; j < 3; j++) {
      float re = 0.0f, im = 0.0f;
#pragma unroll
      for (int k = 0; k < 3; k++) {
        re += d[LGT_RE(i, k)] * dh[LGT_RE(k, j)] - d[LGT_IM(i, k)] * dh[LGT_IM(k, j)];
        im += d[LGT_RE(i, k)] * dh[LGT_IM(k, j)] + d[LGT_IM(i, k)] * dh[LGT_RE(k, j)];
      }
      D[LGT_RE(i, j)] = pair_add(pair_add(D[LGT_RE(i, j)], f2{d[LGT_RE(i, j)], 0.0f}), f2{re, 0.0f});
      D[LGT_IM(i, j)] = pair_add(pair_add(D[LGT_IM(i, j)], f2{d[LGT_IM(i, j)], 0.0f}), f2{im, 0.0f});
    }
}

// One thread per site of parity p: a.links = FP32-12 copy of the anchor field U',
// a.G = D (pairs), a.aux = K0 (pairs); only D(x) is written.
template <int GAUGE>
__device__ __forceinline__ void sweep_body_anchor_sr(const SweepArgs &a, int p, int t, int bx) {
  typedef LinkIO<FMT_F32_12> IO;
  if (a.active && !a.active[t]) return;
  const int j = bx * blockDim.x + threadIdx.x;
  float acc[2] = {0.0f, 0.0f};
  if (j < a.g.vs_half) {
    constexpr int MU0 = GAUGE == GAUGE_COULOMB ? 1 : 0;
    const Coords c = coords_in_slice(a.g, p, t, j);
    const int i = t * a.g.vs_half + j;
    const int q = p ^ 1;
    // C(x) = sum_mu U'_mu(x) D(x+mu)^+ + U'_mu(x-mu)^+ D(x-mu)^+  (small; FP32)
    float C[18];
    mat_zero(C);
#pragma unroll 1
    for (int mu = MU0; mu < 4; mu++) {
      float u[18], dn[18];
      IO::load(a.links, a.g.vh, p, mu, i, u);
      load_hi(a.G, a.g.vh, q, cb_shift(a.g, c, mu, +1), dn);
      acc_mul_dag(u, dn, C);
      const int nb = cb_shift(a.g, c, mu, -1);
      IO::load(a.links, a.g.vh, q, mu, nb, u);
      load_hi(a.G, a.g.vh, q, nb, dn);
      acc_dag_mul_dag(u, dn, C);
    }
    // M = K0 + C, then K = M + D(x) M (the small product in FP32)
    f2 K[18];
    K0IO::load(a.aux, a.g.vh, p, i, K);
#pragma unroll
    for (int e = 0; e < 18; e++) K[e] = pair_add(K[e], f2{C[e], 0.0f});
    float dh[18];  // D(x), high parts, row 2 rebuilt
    load_hi(a.G, a.g.vh, p, i, dh);
    {
      float mh[18], dm[18];
#pragma unroll
      for (int e = 0; e < 18; e++) mh[e] = K[e].hi;
      mat_mul(dh, mh, dm);
#pragma unroll
      for (int e = 0; e < 18; e++) K[e] = pair_add(K[e], f2{dm[e], 0.0f});
    }
    pair_violation(K, acc[0], acc[1]);
    const uint4 draws = sr_draws(a, c);
    RotF rf[3];
    local_update_pair(K, rf, (float)a.omega, a.sr_thr, draws);
    float d[18];
    float_delta(rf, d);
    f2 D[18];
    load_pair_rows(a.G, a.g.vh, p, i, D);
    d_update_lite(D, dh, d);
    DIO::store_pair(a.G, a.g.vh, p, i, D);
  }
  fused_store<float, 1>(a, p, t, bx, acc);
}

}  // namespace anchor_sr
}  // namespace lgt
