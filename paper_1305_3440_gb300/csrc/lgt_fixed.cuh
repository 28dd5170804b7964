// lgt_fixed.cuh -- the bulk half-sweep that leaves the links where they are.
//
// The relaxation only ever changes the field by a gauge transformation, so the
// FP32 bulk phase need not rewrite the links at all: with the input links U
// kept (FP32) and the accumulated transformation G as the only state, the
// update at x sees
//     K(x) = G(x) M(x),   M(x) = sum_mu U_mu(x) G(x+mu)^+ + U_mu(x-mu)^+ G(x-mu)^+,
// which is the K(x) that Sec. 3 gathers from the transformed links G U G^+,
// and G(x) <- g(x) G(x) is the update U_mu(x) <- g U_mu(x), U_mu(x-mu) <-
// U_mu(x-mu) g^+ of those links (Sec. 2 transformation): the paper's sweeps,
// with the transformation kept apart from the links.
//
// What bounds it: memory.  A site update reads 8 links (384 B on 12-real
// links), the 8 neighbours' G (48 B each, every one read by 8 sites: 48 B of
// compulsory traffic) and its own G, and writes its own G: 528 B of compulsory
// traffic against 864 B when the links are rewritten (16 x 48 B) beside G, and
// nothing but 48 B of it is written.  Coulomb gauge reads 6 links and never
// touches the temporal ones: 432 B against 864 B.
#pragma once

#include "lgt_device.cuh"
#include "lgt_internal.h"
#include "lgt_sweep.cuh"

namespace lgt {

// rows 0, 1 of G(x) (FP32, 12 reals); plain loads: a launch writes the G of the
// other parity's sites, and the launch before it wrote these
__device__ __forceinline__ void load_G_rows(const void *G, int vh, int p, int i, float g[18]) {
  const float4 *b4 = reinterpret_cast<const float4 *>(G) + (size_t)(p * 3) * vh + i;
#pragma unroll
  for (int k = 0; k < 3; k++) {
    const float4 v = b4[(size_t)k * vh];
    g[4 * k] = v.x;
    g[4 * k + 1] = v.y;
    g[4 * k + 2] = v.z;
    g[4 * k + 3] = v.w;
  }
}

// 16-byte loads of the sweep, as 32-bit offsets from a uniform base.  Links: read
// once per launch and never written, so they pass L1 by and leave it to G.
__device__ __forceinline__ float4 ld_link(const char *base, unsigned off) {
  float4 v;
  asm volatile("ld.global.nc.L1::no_allocate.v4.f32 {%0,%1,%2,%3}, [%4];"
               : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
               : "l"(base + off));
  return v;
}
__device__ __forceinline__ float2 ld_link2(const char *base, unsigned off) {
  float2 v;
  asm volatile("ld.global.nc.L1::no_allocate.v2.f32 {%0,%1}, [%2];" : "=f"(v.x), "=f"(v.y) : "l"(base + off));
  return v;
}
// The same before griddepcontrol.wait (what a launch may read before it: see
// sweep_start): relaxed at GPU scope, so served by L2 whatever this SM's L1 holds.
__device__ __forceinline__ float4 ld_early(const char *base, unsigned off) {
  float4 v;
  asm volatile("ld.relaxed.gpu.global.L1::no_allocate.v4.f32 {%0,%1,%2,%3}, [%4];"
               : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
               : "l"(base + off)
               : "memory");
  return v;
}
__device__ __forceinline__ float2 ld_early2(const char *base, unsigned off) {
  float2 v;
  asm volatile("ld.relaxed.gpu.global.L1::no_allocate.v2.f32 {%0,%1}, [%2];"
               : "=f"(v.x), "=f"(v.y)
               : "l"(base + off)
               : "memory");
  return v;
}
__device__ __forceinline__ float4 ld_G(const char *base, unsigned off) {
  float4 v;
  asm volatile("ld.global.v4.f32 {%0,%1,%2,%3}, [%4];"
               : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
               : "l"(base + off));
  return v;
}
__device__ __forceinline__ void put4(float m[18], int k, float4 v) {
  m[4 * k] = v.x;
  m[4 * k + 1] = v.y;
  m[4 * k + 2] = v.z;
  m[4 * k + 3] = v.w;
}

// row 2 = conj(row 0 x row 1) as chains of fused multiply-adds (rebuild_row2's
// differences of products take a fifth instruction per entry)
__device__ __forceinline__ void fma_row2(float m[18]) {
#pragma unroll
  for (int c = 0; c < 3; c++) {
    const int a = (c + 1) % 3, b = (c + 2) % 3;
    float re = m[LGT_RE(0, a)] * m[LGT_RE(1, b)], im = -m[LGT_RE(0, a)] * m[LGT_IM(1, b)];
    re = fmaf(-m[LGT_IM(0, a)], m[LGT_IM(1, b)], re);
    im = fmaf(-m[LGT_IM(0, a)], m[LGT_RE(1, b)], im);
    re = fmaf(-m[LGT_RE(0, b)], m[LGT_RE(1, a)], re);
    im = fmaf(m[LGT_RE(0, b)], m[LGT_IM(1, a)], im);
    re = fmaf(m[LGT_IM(0, b)], m[LGT_IM(1, a)], re);
    im = fmaf(m[LGT_IM(0, b)], m[LGT_RE(1, a)], im);
    m[LGT_RE(2, c)] = re;
    m[LGT_IM(2, c)] = im;
  }
}

// rows 0, 1 of a b^+ (a: rows 0, 1 given; b: three rows)
__device__ __forceinline__ void rows_mul_dag(const float a[12], const float b[18], float r[12]) {
#pragma unroll
  for (int i = 0; i < 2; i++)
#pragma unroll
    for (int j = 0; j < 3; j++) {
      float re = a[LGT_RE(i, 0)] * b[LGT_RE(j, 0)], im = a[LGT_IM(i, 0)] * b[LGT_RE(j, 0)];
      re = fmaf(a[LGT_IM(i, 0)], b[LGT_IM(j, 0)], re);
      im = fmaf(-a[LGT_RE(i, 0)], b[LGT_IM(j, 0)], im);
#pragma unroll
      for (int k = 1; k < 3; k++) {
        re = fmaf(a[LGT_RE(i, k)], b[LGT_RE(j, k)], re);
        im = fmaf(a[LGT_IM(i, k)], b[LGT_RE(j, k)], im);
        re = fmaf(a[LGT_IM(i, k)], b[LGT_IM(j, k)], re);
        im = fmaf(-a[LGT_RE(i, k)], b[LGT_IM(j, k)], im);
      }
      r[LGT_RE(i, j)] = re;
      r[LGT_IM(i, j)] = im;
    }
}

// rows 0, 1 of a b (a: rows 0, 1 given; b: three rows)
__device__ __forceinline__ void rows_mul(const float a[12], const float b[18], float r[12]) {
#pragma unroll
  for (int i = 0; i < 2; i++)
#pragma unroll
    for (int j = 0; j < 3; j++) {
      float re = a[LGT_RE(i, 0)] * b[LGT_RE(0, j)], im = a[LGT_RE(i, 0)] * b[LGT_IM(0, j)];
      re = fmaf(-a[LGT_IM(i, 0)], b[LGT_IM(0, j)], re);
      im = fmaf(a[LGT_IM(i, 0)], b[LGT_RE(0, j)], im);
#pragma unroll
      for (int k = 1; k < 3; k++) {
        re = fmaf(a[LGT_RE(i, k)], b[LGT_RE(k, j)], re);
        im = fmaf(a[LGT_RE(i, k)], b[LGT_IM(k, j)], im);
        re = fmaf(-a[LGT_IM(i, k)], b[LGT_IM(k, j)], re);
        im = fmaf(a[LGT_IM(i, k)], b[LGT_RE(k, j)], im);
      }
      r[LGT_RE(i, j)] = re;
      r[LGT_IM(i, j)] = im;
    }
}

// Sec. 3 local update as local_update (lgt_device.cuh; overrelaxation and the heat
// bath), giving rows 0 and 1 of g only (what G <- g G needs of it): each subgroup element is the pair
// (a, b) of [[a, b], [-conj b, conj a]], a = r0 + i r3, b = r2 + i r1, and
// g = R_2 R_1 R_0 is formed from the pairs, whose zeros are known.
template <int ALGO>
__device__ __forceinline__ void local_update_rows(float W[18], float g[12], float omega, const SaDraw *sa) {
  float ar[3], ai[3], br[3], bi[3];
#pragma unroll
  for (int s = 0; s < 3; s++) {
    const int i = (s == 2) ? 1 : 0;
    const int j = (s == 0) ? 1 : 2;
    const float q0 = W[LGT_RE(i, i)] + W[LGT_RE(j, j)];
    const float q1 = W[LGT_IM(i, j)] + W[LGT_IM(j, i)];
    const float q2 = W[LGT_RE(i, j)] - W[LGT_RE(j, i)];
    const float q3 = W[LGT_IM(i, i)] - W[LGT_IM(j, j)];
    const float n2 = q0 * q0 + q1 * q1 + q2 * q2 + q3 * q3;
    float r0 = 1.0f, r1 = 0.0f, r2 = 0.0f, r3 = 0.0f;
    if (ALGO == ALGO_SA) {
      su2_heatbath<float>(q0, q1, q2, q3, *sa, s, r0, r1, r2, r3);
    } else if (n2 > 0.0f) {
      const float inv = rsqrtf(n2);
      r0 = q0 * inv;
      r1 = -q1 * inv;
      r2 = -q2 * inv;
      r3 = -q3 * inv;
    }
    if (ALGO == ALGO_OR) {
      r0 = (1.0f - omega) + omega * r0;
      r1 *= omega;
      r2 *= omega;
      r3 *= omega;
      const float inv = rsqrtf(r0 * r0 + r1 * r1 + r2 * r2 + r3 * r3);
      r0 *= inv;
      r1 *= inv;
      r2 *= inv;
      r3 *= inv;
    }
    ar[s] = r0, ai[s] = r3, br[s] = r2, bi[s] = r1;
    if (s < 2) {
#pragma unroll
      for (int c = 0; c < 3; c++) {
        const float wire = W[LGT_RE(i, c)], wiim = W[LGT_IM(i, c)];
        const float wjre = W[LGT_RE(j, c)], wjim = W[LGT_IM(j, c)];
        W[LGT_RE(i, c)] = r0 * wire - r3 * wiim + r2 * wjre - r1 * wjim;
        W[LGT_IM(i, c)] = r0 * wiim + r3 * wire + r2 * wjim + r1 * wjre;
        W[LGT_RE(j, c)] = -r2 * wire - r1 * wiim + r0 * wjre + r3 * wjim;
        W[LGT_IM(j, c)] = -r2 * wiim + r1 * wire + r0 * wjim - r3 * wjre;
      }
    }
  }
  // R_1 R_0: row 0 = (a1 a0, a1 b0, b1), row 1 = (-conj b0, conj a0, 0),
  // row 2 = (-conj b1 a0, -conj b1 b0, conj a1); R_2 mixes rows 1 and 2
  g[LGT_RE(0, 0)] = ar[1] * ar[0] - ai[1] * ai[0];
  g[LGT_IM(0, 0)] = ar[1] * ai[0] + ai[1] * ar[0];
  g[LGT_RE(0, 1)] = ar[1] * br[0] - ai[1] * bi[0];
  g[LGT_IM(0, 1)] = ar[1] * bi[0] + ai[1] * br[0];
  g[LGT_RE(0, 2)] = br[1];
  g[LGT_IM(0, 2)] = bi[1];
  const float c0r = -(br[1] * ar[0] + bi[1] * ai[0]), c0i = -(br[1] * ai[0] - bi[1] * ar[0]);
  const float c1r = -(br[1] * br[0] + bi[1] * bi[0]), c1i = -(br[1] * bi[0] - bi[1] * br[0]);
  // row 1 = a2 (row 1) + b2 (row 2)
  g[LGT_RE(1, 0)] = -(ar[2] * br[0] + ai[2] * bi[0]) + (br[2] * c0r - bi[2] * c0i);
  g[LGT_IM(1, 0)] = (ar[2] * bi[0] - ai[2] * br[0]) + (br[2] * c0i + bi[2] * c0r);
  g[LGT_RE(1, 1)] = (ar[2] * ar[0] + ai[2] * ai[0]) + (br[2] * c1r - bi[2] * c1i);
  g[LGT_IM(1, 1)] = (ai[2] * ar[0] - ar[2] * ai[0]) + (br[2] * c1i + bi[2] * c1r);
  g[LGT_RE(1, 2)] = br[2] * ar[1] + bi[2] * ai[1];
  g[LGT_IM(1, 2)] = bi[2] * ar[1] - br[2] * ai[1];
}

// Neighbours' G loaded ahead, in terms: 2 at the 128-register budget (512 threads
// per SM), 1 at fewer registers or with the longer 18-real links, 4 or 3 at 255
// registers, which also hold the links of all terms (fixed_links_ahead).
__host__ __device__ constexpr int fixed_depth(int lfmt, int threads_per_sm) {
  return threads_per_sm <= 256 ? (lfmt == FMT_F32_12 ? 4 : 3) : (lfmt == FMT_F32_12 && threads_per_sm <= 512 ? 2 : 1);
}
// links loaded before the wait for the launch before, in terms
__host__ __device__ constexpr int fixed_links_ahead(int depth, int n) { return depth >= 3 ? n : depth + 1; }

// Start of a sweep over links that no sweep writes.  What the launches before it
// in its run leave alone -- the links, K0, the activity mask -- may be read before
// griddepcontrol.wait: a launch is let in only after every block of the launch
// before has passed its own wait, and a run's first launch, which is a plain one,
// after all that wrote those.  G, the loop state and the slots are touched after
// the wait only.  On a lattice that leaves the SMs room the next launch's blocks
// so have their indices and links ready when the launch before ends, and only the
// G loads and the update lie between one launch's end and the next one's; on a
// large one they fill the last wave's gap.  Half-sweep with all loads after the
// wait -> as here: 8^4 bulk 3.46 -> 2.99 us, polish 3.87 -> 3.33; 16^4 5.13 -> 4.83
// and 6.73 -> 6.32; 32^4 bulk 46.0 -> 44.7.
__device__ __forceinline__ bool sweep_slice_active(const SweepArgs &a, int t) {
  if (!a.active) return true;
  unsigned v;
  asm volatile("ld.relaxed.gpu.global.u8 %0, [%1];" : "=r"(v) : "l"(a.active + t) : "memory");
  return v != 0;
}
// the wait, and the arguments with the loop state's values
__device__ __forceinline__ SweepArgs sweep_start(const SweepArgs &in) {
  pdl_enter();
  return resolve_loop(in);
}

// Rows 0, 1 of G orthonormalised to first order in their error.  G is a factor
// of every K(x) around it and row 2 of every product is rebuilt from rows 0, 1,
// so an error of its rows would be passed on (by about 4/3 per update while the
// rotations are large) and would distort K: theta 1e-4 off after 40 sweeps.  Every
// update therefore brings its G back: the rows come in with errors of a few
// 2^-24, whose squares vanish, so no roots are needed.
__device__ __forceinline__ void orthonormalise_rows(float r[12]) {
  float n = 0.0f;
#pragma unroll
  for (int e = 0; e < 6; e++) n = fmaf(r[e], r[e], n);
  n = fmaf(-0.5f, n, 1.5f);
#pragma unroll
  for (int e = 0; e < 6; e++) r[e] *= n;
  float dr = 0.0f, di = 0.0f;  // <row 0, row 1>
#pragma unroll
  for (int c = 0; c < 3; c++) {
    dr = fmaf(r[LGT_RE(0, c)], r[LGT_RE(1, c)], dr);
    di = fmaf(r[LGT_RE(0, c)], r[LGT_IM(1, c)], di);
    dr = fmaf(r[LGT_IM(0, c)], r[LGT_IM(1, c)], dr);
    di = fmaf(-r[LGT_IM(0, c)], r[LGT_RE(1, c)], di);
  }
  n = 0.0f;
#pragma unroll
  for (int c = 0; c < 3; c++) {
    float re = fmaf(-dr, r[LGT_RE(0, c)], r[LGT_RE(1, c)]);
    float im = fmaf(-dr, r[LGT_IM(0, c)], r[LGT_IM(1, c)]);
    re = fmaf(di, r[LGT_IM(0, c)], re);
    im = fmaf(-di, r[LGT_RE(0, c)], im);
    r[LGT_RE(1, c)] = re;
    r[LGT_IM(1, c)] = im;
    n = fmaf(re, re, n);
    n = fmaf(im, im, n);
  }
  n = fmaf(-0.5f, n, 1.5f);
#pragma unroll
  for (int e = 6; e < 12; e++) r[e] *= n;
}

// M += U G^+ (forward) or (G U)^+ (backward).  With 12-real storage rows 0, 1 of
// the product and its row 2 from those (it is in SU(3)); each entry is formed
// before it is added, one rounding at M's size per term.
template <int LFMT>
__device__ __forceinline__ void fixed_term(float u[18], float g[18], bool fwd, float M[18]) {
  float r[18];
  if (fwd) {
    fma_row2(g);
    if constexpr (LFMT == FMT_F32_12) {
      rows_mul_dag(u, g, r);
      fma_row2(r);
    } else {
      mat_mul_dag(u, g, r);
    }
    acc_add(M, r);
  } else {
    if constexpr (LFMT == FMT_F32_12) {
      fma_row2(u);
      rows_mul(g, u, r);
      fma_row2(r);
    } else {
      fma_row2(g);
      mat_mul(g, u, r);
    }
    acc_add_dag(M, r);
  }
}

// Half-sweep body, one thread per site of parity p: a.links = the FP32 links
// (LFMT: 12- or 18-real storage, not written), a.G = G.
//
// The eight terms (six for Coulomb gauge) are unrolled and their loads issued
// DEPTH terms ahead of their products (term by term in a loop: 51 us per 32^4
// half-sweep against 43; the links staged in shared memory by cp.async: 52 us,
// since the staging buffers take the L1 that serves the neighbours' G).  Links
// skip L1 (each is read once per launch).  Site indices by reciprocal
// multiplication, neighbour offsets as one select each and 32-bit byte offsets
// from uniform bases: 1840 warp instructions per 32 sites instead of 2150.
// Measured with CUDA events, launches back to back, against the rewritten links'
// fastest configuration: 12-real links 32^4 Landau 59.7 -> 43 us, 64^4 Landau
// 1034 -> 700 us and 48^3x96 Coulomb 620 -> 360 us (both at 6.3 to 6.6 TB/s of
// DRAM traffic); 18-real links 14x10x12x18 6.2 -> 5.2 us.
template <int LFMT, int GAUGE, int ALGO, int DEPTH>
__device__ __forceinline__ void sweep_body_fixed(const SweepArgs &in, int p, int t, int bx) {
  constexpr bool kRows = LFMT == FMT_F32_12;  // row 2 of a link is rebuilt, not stored
  constexpr int MU0 = GAUGE == GAUGE_COULOMB ? 1 : 0;
  constexpr int N = 2 * (4 - MU0);
  constexpr int NU = fixed_links_ahead(DEPTH, N), DG = DEPTH < N ? DEPTH : N;
  constexpr int NC = kRows ? 3 : 4;  // 16-byte chunks per link
  if (!sweep_slice_active(in, t)) {  // whole block belongs to one slice
    pdl_enter();  // (a launch ends only after the one before it)
    return;
  }
  const int j = bx * (int)blockDim.x + (int)threadIdx.x;
  const bool valid = j < in.g.vs_half;
  const SiteNb nb(in.g, in.inv_half1, in.inv_n2, p, t, valid ? j : 0);
  const int q = p ^ 1;
  const size_t S = (size_t)in.g.vh * 16;  // bytes of one chunk's stream
  const char *const L = (const char *)in.links;
  const char *const Lp = L + (size_t)(p * 4 * NC) * S, *const Lq = L + (size_t)(q * 4 * NC) * S;
  const char *const L2 = L + 32 * S;  // 18-real storage: the float2 chunk's streams
  const char *const Gq = (const char *)in.G + (size_t)(q * 3) * S;
  char *const Gp = (char *)in.G + (size_t)(p * 3) * S;
  const unsigned o = (unsigned)(t * in.g.vs_half + j) * 16u;
  // term n: direction MU0 + n / 2, forward link if n is even
  auto site = [&](int n) { return o + nb.bytes(in.g, MU0 + n / 2, (n & 1) ? -1 : 1); };
  float U[NU][18], G[DG + 1][18];
  auto load_u = [&](int n, bool early) {
    const int mu = MU0 + n / 2;
    const bool fwd = !(n & 1);
    const char *const Lb = (fwd ? Lp : Lq) + (size_t)(mu * NC) * S;
    const unsigned ou = fwd ? o : site(n);
#pragma unroll
    for (int k = 0; k < NC; k++) put4(U[n % NU], k, early ? ld_early(Lb + (size_t)k * S, ou) : ld_link(Lb + (size_t)k * S, ou));
    if (!kRows) {
      const char *const Lw = L2 + (size_t)((fwd ? p : q) * 4 + mu) * (S / 2);
      const float2 w = early ? ld_early2(Lw, ou / 2) : ld_link2(Lw, ou / 2);
      U[n % NU][16] = w.x, U[n % NU][17] = w.y;
    }
  };
  auto load_g = [&](int n) {
#pragma unroll
    for (int k = 0; k < 3; k++) put4(G[n % (DG + 1)], k, ld_G(Gq + (size_t)k * S, site(n)));
  };
  if (valid) {
#pragma unroll
    for (int n = 0; n < NU; n++) load_u(n, true);
  }
  const SweepArgs a = sweep_start(in);
  float acc[2] = {0.0f, 0.0f};
  if (valid) {
    float W[18], gx[18];
    {
      float M[18];
      mat_zero(M);
#pragma unroll
      for (int n = 0; n < DG; n++) load_g(n);
#pragma unroll
      for (int n = 0; n < N; n++) {
        if (n + DG < N) {
          if (n > 0 && n + NU - 1 < N) load_u(n + NU - 1, false);
          load_g(n + DG);
        } else if (n + DG == N) {
#pragma unroll
          for (int k = 0; k < 3; k++) put4(gx, k, ld_G(Gp + (size_t)k * S, o));
        }
        fixed_term<LFMT>(U[n % NU], G[n % (DG + 1)], !(n & 1), M);
      }
      fma_row2(gx);
      mat_mul(gx, M, W);  // K(x) = G(x) M(x)
    }
    violation_of_K(W, acc[0], acc[1]);
    SaDraw sd;
    if (ALGO == ALGO_SA) sd = sa_draw_of(a, nb.coords(t));
    float g[12];
    local_update_rows<ALGO>(W, g, (float)a.omega, &sd);
    float r[18];
    rows_mul(g, gx, r);
    if (a.reunit) reunitarise(r);
    else orthonormalise_rows(r);
#pragma unroll
    for (int k = 0; k < 3; k++)
      *reinterpret_cast<float4 *>(Gp + (size_t)k * S + o) = make_float4(r[4 * k], r[4 * k + 1], r[4 * k + 2], r[4 * k + 3]);
  }
  fused_store<float, 1>(a, p, t, bx, acc);
}

// The same half-sweep by four threads per site, thread m of a site's quad taking
// the two terms of direction m (thread 0 none in Coulomb gauge); two xor shuffles
// sum M(x) to all four, which then run the same update, and three of them store a
// chunk of G each.  For lattices that leave most of the chip's schedulers with a
// warp or none: the chain of a site is about half as long.  The autotuner takes it
// up to 10^4 sites or so (half-sweep at 8^4: bulk 4.0 -> 3.5 us, polish 6.3 -> 3.9,
// both 3.0 and 3.3 with the links read early; at 12^4 one thread per site is ahead
// in the bulk).
template <int LFMT, int GAUGE>
__device__ __forceinline__ void sweep_body_fixed_quad(const SweepArgs &in, int p, int t, int bx) {
  if (!sweep_slice_active(in, t)) {  // whole block belongs to one slice
    pdl_enter();
    return;
  }
  constexpr int MU0 = GAUGE == GAUGE_COULOMB ? 1 : 0;
  constexpr int NC = LFMT == FMT_F32_12 ? 3 : 4;
  const int m = (int)threadIdx.x & 3;
  const int j = bx * (int)(blockDim.x >> 2) + (int)(threadIdx.x >> 2);
  const bool valid = j < in.g.vs_half;  // the shuffles below need every lane
  const SiteNb nb(in.g, in.inv_half1, in.inv_n2, p, t, valid ? j : 0);
  const int i = t * in.g.vs_half + (valid ? j : 0);
  const int q = p ^ 1;
  const size_t S = (size_t)in.g.vh * 16;
  const char *const L = (const char *)in.links;
  const char *const Gq = (const char *)in.G + (size_t)(q * 3) * S;
  char *const Gp = (char *)in.G + (size_t)(p * 3) * S;
  const unsigned o = (unsigned)i * 16u;
  float M[18], W[18], gx[18];
  mat_zero(M);
  float U[2][18], G[2][18];
  unsigned on[2];
#pragma unroll
  for (int d = 0; d < 2; d++) {  // forward, backward
    on[d] = o + nb.bytes(in.g, m, d ? -1 : 1);
    const unsigned ou = d ? on[d] : o;
    const int pu = d ? q : p;
    if (m >= MU0) {
#pragma unroll
      for (int k = 0; k < NC; k++) put4(U[d], k, ld_early(L + (size_t)((pu * 4 + m) * NC + k) * S, ou));
      if (LFMT == FMT_F32_18) {
        const float2 w = ld_early2(L + 32 * S + (size_t)(pu * 4 + m) * (S / 2), ou / 2);
        U[d][16] = w.x, U[d][17] = w.y;
      }
    }
  }
  const SweepArgs a = sweep_start(in);
  if (m >= MU0) {
#pragma unroll
    for (int d = 0; d < 2; d++)
#pragma unroll
      for (int k = 0; k < 3; k++) put4(G[d], k, ld_G(Gq + (size_t)k * S, on[d]));
  }
  // (the lanes past the slice have site 0's indices, whose G another warp writes)
  mat_zero(gx);
  if (valid) {
#pragma unroll
    for (int k = 0; k < 3; k++) put4(gx, k, ld_G(Gp + (size_t)k * S, o));
  }
  if (m >= MU0) {
    fixed_term<LFMT>(U[0], G[0], true, M);
    fixed_term<LFMT>(U[1], G[1], false, M);
  }
#pragma unroll
  for (int e = 0; e < 18; e++) M[e] += __shfl_xor_sync(0xffffffffu, M[e], 1);
#pragma unroll
  for (int e = 0; e < 18; e++) M[e] += __shfl_xor_sync(0xffffffffu, M[e], 2);
  fma_row2(gx);
  mat_mul(gx, M, W);
  float acc[2] = {0.0f, 0.0f};
  {
    float vr, vd;
    violation_of_K(W, vr, vd);
    if (valid && m == 0) acc[0] = vr, acc[1] = vd;
  }
  float g[12], r[18];
  local_update_rows<ALGO_OR>(W, g, (float)a.omega, nullptr);
  rows_mul(g, gx, r);
  if (a.reunit) reunitarise(r);
  else orthonormalise_rows(r);
  __syncwarp();  // every thread of the quad has read G(x) before one of them writes it (shuffles order no memory)
#pragma unroll
  for (int k = 0; k < 3; k++)
    if (valid && m == k)
      *reinterpret_cast<float4 *>(Gp + (size_t)k * S + o) = make_float4(r[4 * k], r[4 * k + 1], r[4 * k + 2], r[4 * k + 3]);
  fused_store<float, 4>(a, p, t, bx, acc);
}

// neighbours' D loaded ahead, in terms (80 registers, configuration 11: none)
__host__ __device__ constexpr int anchor_depth(int cfg) { return cfg == 16 ? 4 : (cfg == 11 ? 0 : (cfg == 3 ? 1 : 2)); }

// Anchored polishing sweep (lgt_anchor.cuh): a.links = FP32-12 copy of the anchor
// field U', a.G = D = G - 1 (pairs), a.aux = K0.  One thread per site; only D(x) is
// written.  Loads, indices and the unrolled terms as sweep_body_fixed's.  Against
// the looped body with K in pairs at 80 registers: 32^4 half-sweep 83 -> 67 us (5.8
// TB/s in compulsory bytes), 8^4 8.0 -> 6.3 us.
template <int GAUGE, int DEPTH>
__device__ __forceinline__ void sweep_body_anchor(const SweepArgs &in, int p, int t, int bx) {
  constexpr int MU0 = GAUGE == GAUGE_COULOMB ? 1 : 0;
  constexpr int N = 2 * (4 - MU0);
  constexpr int NU = fixed_links_ahead(DEPTH, N), DG = DEPTH < N ? DEPTH : N;
  if (!sweep_slice_active(in, t)) {
    pdl_enter();
    return;
  }
  const int j = bx * (int)blockDim.x + (int)threadIdx.x;
  const bool valid = j < in.g.vs_half;
  const SiteNb nb(in.g, in.inv_half1, in.inv_n2, p, t, valid ? j : 0);
  const int i = t * in.g.vs_half + j;
  const int q = p ^ 1;
  const size_t S = (size_t)in.g.vh * 16;
  const char *const L = (const char *)in.links;
  const char *const Lp = L + (size_t)(p * 12) * S, *const Lq = L + (size_t)(q * 12) * S;
  const char *const Dq = (const char *)in.G + (size_t)(q * 3) * S;
  char *const Dp = (char *)in.G + (size_t)(p * 3) * S;
  char *const Dl = Dp + 6 * S;  // the low parts
  const unsigned o = (unsigned)i * 16u;
  auto site = [&](int n) { return o + nb.bytes(in.g, MU0 + n / 2, (n & 1) ? -1 : 1); };
  float U[NU][18], G[DG + 1][18];
  AnchorK0 k0;
  auto load_u = [&](int n, bool early) {
    const bool fwd = !(n & 1);
    const char *const Lb = (fwd ? Lp : Lq) + (size_t)((MU0 + n / 2) * 3) * S;
    const unsigned ou = fwd ? o : site(n);
#pragma unroll
    for (int k = 0; k < 3; k++) put4(U[n % NU], k, early ? ld_early(Lb + (size_t)k * S, ou) : ld_link(Lb + (size_t)k * S, ou));
  };
  auto load_g = [&](int n) {
#pragma unroll
    for (int k = 0; k < 3; k++) put4(G[n % (DG + 1)], k, ld_G(Dq + (size_t)k * S, site(n)));
  };
  if (valid) {
#pragma unroll
    for (int n = 0; n < NU; n++) load_u(n, true);
    if (NU == N) K0IO::load<true>(in.aux, in.g.vh, p, i, k0);
  }
  const SweepArgs a = sweep_start(in);
  float acc[2] = {0.0f, 0.0f};
  if (valid) {
    // C(x) = sum_mu U'_mu(x) D(x+mu)^+ + U'_mu(x-mu)^+ D(x-mu)^+  (small; FP32)
    float C[18], dh[18];
    mat_zero(C);
#pragma unroll
    for (int n = 0; n < DG; n++) load_g(n);
#pragma unroll
    for (int n = 0; n < N; n++) {
      if (n > 0 && n + NU - 1 < N) load_u(n + NU - 1, false);
      if (n + DG < N) load_g(n + DG);
      if (n == N - 1) {
#pragma unroll
        for (int k = 0; k < 3; k++) put4(dh, k, ld_G(Dp + (size_t)k * S, o));
      }
      float *const u = U[n % NU], *const g = G[n % (DG + 1)];
      fma_row2(u);
      small_row2(g);
      if (!(n & 1)) acc_mul_dag(u, g, C);
      else acc_dag_mul_dag(u, g, C);
    }
    small_row2(dh);  // D(x), high parts
    float d[18];
    {
      if (NU < N) K0IO::load<false>(a.aux, a.g.vh, p, i, k0);
      AnchorK K;
      anchor_K(k0, anchor_diag(GAUGE), C, dh, K);
      anchor_violation(K, acc[0], acc[1]);
      RotF rf[3];
      anchor_local_update(K, anchor_diag(GAUGE), rf, (float)a.omega);
      float_delta(rf, d);
    }
    f2 D[12];
#pragma unroll
    for (int k = 0; k < 3; k++) {
      const float4 l = ld_G(Dl + (size_t)k * S, o);
      D[4 * k] = {dh[4 * k], l.x};
      D[4 * k + 1] = {dh[4 * k + 1], l.y};
      D[4 * k + 2] = {dh[4 * k + 2], l.z};
      D[4 * k + 3] = {dh[4 * k + 3], l.w};
    }
    d_update(D, dh, d);
    DIO::store_pair(a.G, a.g.vh, p, i, D);
  }
  fused_store<float, 1>(a, p, t, bx, acc);
}

// The polish by four threads per site, as sweep_body_fixed_quad.
template <int GAUGE>
__device__ __forceinline__ void sweep_body_anchor_quad(const SweepArgs &in, int p, int t, int bx) {
  if (!sweep_slice_active(in, t)) {  // whole block belongs to one slice
    pdl_enter();
    return;
  }
  constexpr int MU0 = GAUGE == GAUGE_COULOMB ? 1 : 0;
  const int m = (int)threadIdx.x & 3;
  const int j = bx * (int)(blockDim.x >> 2) + (int)(threadIdx.x >> 2);
  const bool valid = j < in.g.vs_half;  // the shuffles below need every lane
  const SiteNb nb(in.g, in.inv_half1, in.inv_n2, p, t, valid ? j : 0);
  const int i = t * in.g.vs_half + (valid ? j : 0);
  const int q = p ^ 1;
  const size_t S = (size_t)in.g.vh * 16;
  const char *const L = (const char *)in.links;
  const char *const Dq = (const char *)in.G + (size_t)(q * 3) * S;
  char *const Dp = (char *)in.G + (size_t)(p * 3) * S;
  const unsigned o = (unsigned)i * 16u;
  float C[18], dh[18];
  mat_zero(C);
  float U[2][18], G[2][18];
  unsigned on[2];
  AnchorK0 k0;
#pragma unroll
  for (int d = 0; d < 2; d++) {  // forward, backward
    on[d] = o + nb.bytes(in.g, m, d ? -1 : 1);
    if (m >= MU0) {
#pragma unroll
      for (int k = 0; k < 3; k++) put4(U[d], k, ld_early(L + (size_t)(((d ? q : p) * 4 + m) * 3 + k) * S, d ? on[d] : o));
    }
  }
  K0IO::load<true>(in.aux, in.g.vh, p, i, k0);
  const SweepArgs a = sweep_start(in);
  if (m >= MU0) {
#pragma unroll
    for (int d = 0; d < 2; d++)
#pragma unroll
      for (int k = 0; k < 3; k++) put4(G[d], k, ld_G(Dq + (size_t)k * S, on[d]));
  }
  // (the lanes past the slice: as sweep_body_fixed_quad)
  mat_zero(dh);
  float4 lo[3] = {};
  if (valid) {
#pragma unroll
    for (int k = 0; k < 3; k++) put4(dh, k, ld_G(Dp + (size_t)k * S, o));
#pragma unroll
    for (int k = 0; k < 3; k++) lo[k] = ld_G(Dp + (6 + k) * S, o);
  }
  if (m >= MU0) {
#pragma unroll
    for (int d = 0; d < 2; d++) {
      fma_row2(U[d]);
      small_row2(G[d]);
      if (d == 0) acc_mul_dag(U[d], G[d], C);
      else acc_dag_mul_dag(U[d], G[d], C);
    }
  }
#pragma unroll
  for (int e = 0; e < 18; e++) C[e] += __shfl_xor_sync(0xffffffffu, C[e], 1);
#pragma unroll
  for (int e = 0; e < 18; e++) C[e] += __shfl_xor_sync(0xffffffffu, C[e], 2);
  small_row2(dh);
  AnchorK K;
  anchor_K(k0, anchor_diag(GAUGE), C, dh, K);
  float acc[2] = {0.0f, 0.0f};
  {
    float vr, vd;
    anchor_violation(K, vr, vd);
    if (valid && m == 0) acc[0] = vr, acc[1] = vd;
  }
  RotF rf[3];
  anchor_local_update(K, anchor_diag(GAUGE), rf, (float)a.omega);
  float d[18];
  float_delta(rf, d);
  f2 D[12];
#pragma unroll
  for (int k = 0; k < 3; k++) {
    D[4 * k] = {dh[4 * k], lo[k].x};
    D[4 * k + 1] = {dh[4 * k + 1], lo[k].y};
    D[4 * k + 2] = {dh[4 * k + 2], lo[k].z};
    D[4 * k + 3] = {dh[4 * k + 3], lo[k].w};
  }
  d_update(D, dh, d);
  __syncwarp();  // every thread of the quad has read D(x) before one of them writes it
#pragma unroll
  for (int k = 0; k < 3; k++) {
    if (valid && m == k) {
      *reinterpret_cast<float4 *>(Dp + (size_t)k * S + o) = make_float4(D[4 * k].hi, D[4 * k + 1].hi, D[4 * k + 2].hi, D[4 * k + 3].hi);
      *reinterpret_cast<float4 *>(Dp + (6 + k) * S + o) = make_float4(D[4 * k].lo, D[4 * k + 1].lo, D[4 * k + 2].lo, D[4 * k + 3].lo);
    }
  }
  fused_store<float, 4>(a, p, t, bx, acc);
}

// ------------------------------------------------------------ working links
// The bulk's working link U_mu(x) -> G(x) U_mu(x) G(x+mu)^+ in FP32 (12-real
// storage: rows 0, 1 formed and row 2 rebuilt, as a stored working link; 18-real:
// all three rows), for measurements and output between sweeps.
// G(x) with its row 2
__device__ __forceinline__ void load_G_full(const void *G, int vh, int p, int i, float g[18]) {
  load_G_rows(G, vh, p, i, g);
  fma_row2(g);
}
// w: the stored link in, the working link out; gx, gy: G at its two ends
template <int LFMT>
__device__ __forceinline__ void form_working(const float gx[18], const float gy[18], float w[18]) {
  float r[18];
  if (LFMT == FMT_F32_12) {
    rows_mul(gx, w, r);
    rows_mul_dag(r, gy, w);
    fma_row2(w);
  } else {
    mat_mul(gx, w, r);
    mat_mul_dag(r, gy, w);
  }
}
template <int LFMT>
__device__ __forceinline__ void load_stored(const void *links, int vh, int p, int mu, int i, float w[18]) {
  LinkIO<LFMT>::load_raw(links, vh, p, mu, i, w);
  if (LFMT == FMT_F32_12) fma_row2(w);
}
template <int LFMT>
__device__ __forceinline__ void load_working(const Geom &g, const void *links, const void *G, int skip_temporal, int p,
                                             int mu, int i, float w[18]) {
  load_stored<LFMT>(links, g.vh, p, mu, i, w);
  if (skip_temporal && mu == 0) return;
  const int t = i / g.vs_half;
  const Coords c = coords_in_slice(g, p, t, i - t * g.vs_half);
  float gx[18], gy[18];
  load_G_full(G, g.vh, p, i, gx);
  load_G_full(G, g.vh, p ^ 1, cb_shift(g, c, mu, +1), gy);
  form_working<LFMT>(gx, gy, w);
}

}  // namespace lgt
