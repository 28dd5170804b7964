// lgt_io.cu -- the field in and out of a context: ingest (public layout -> SoA,
// with the SU(3) check), egress, and the gauge transformations in FP64 that
// promotion and output need.
//
// The public layout keeps a site's four links together (576 B), the device layout
// one stream per (parity, direction, 16-byte chunk).  A block takes 32 consecutive
// pairs of sites (2 i, 2 i + 1): 36 KB of the public layout in one piece, and in
// either parity the within-parity indices i0 .. i0 + 31, 512 B of every stream.  It
// moves the public side through shared memory 16 B per thread in order and the
// device side one stream per warp, so both are whole sectors.  Measured against one
// thread per link on both sides, 144 B apart on the public one: ingest of 32^4 links
// (FP64 and FP32-12) 3.44 -> 0.32 ms (1.4 GB: 4.3 TB/s; 1.7 ms of each of the two
// passes was the SU(3) check below), egress of 36x24x28x20 FP64 links 89 us (6.2
// TB/s), 64^4 FP32-12 working links 12.4 -> 1.9 ms.
#include <cuda_runtime.h>
#include <stdint.h>

#include "lgt_device.cuh"
#include "lgt_internal.h"
#include "lgt_measure.cuh"

namespace lgt {

namespace {

constexpr int kPairs = 32;    // site pairs per block (one per lane)
constexpr int kThreads = 256;  // one warp per (parity, direction)
constexpr int kPairUnits = 72;  // 16-byte units of a pair in the public layout
// a pair's stride in shared memory: odd, so that the lanes' 16-byte accesses fall
// on different banks
constexpr int kPairStride = kPairUnits + 1;

unsigned tile_blocks(const Geom &g) { return (unsigned)((g.vh + kPairs - 1) / kPairs); }

// This thread's link: warp w holds parity w / 4, direction w % 4; lane l the
// within-parity index i of the block's pair l.  The site of parity p in a pair is
// its odd one iff p + x2 + x3 + t is odd.
struct TileLink {
  int p, mu, i, pair, odd;
  bool valid;
  __device__ __forceinline__ explicit TileLink(const Geom &g) : TileLink(g, (int)threadIdx.x >> 5, blockIdx.x) {}
  // warp w of tile number `tile`
  __device__ __forceinline__ TileLink(const Geom &g, int w, long long tile) {
    p = w >> 2;
    mu = w & 3;
    pair = (int)threadIdx.x & 31;
    const long long ii = tile * kPairs + pair;
    valid = ii < g.vh;
    i = valid ? (int)ii : 0;
    const int row = i / g.half1, plane = row / g.n2;
    odd = (p + (row - plane * g.n2) + plane % g.n3 + plane / g.n3) & 1;
  }
  // the link's first unit in the tile
  __device__ __forceinline__ int unit() const { return pair * kPairStride + odd * (kPairUnits / 2) + mu * 9; }
};

__device__ __forceinline__ int tile_units(const Geom &g) {
  const long long left = (long long)g.vh - (long long)blockIdx.x * kPairs;
  return (int)(left < kPairs ? left : kPairs) * kPairUnits;
}

// (a caller's buffer need only be aligned to its doubles: 8-byte accesses then)
__device__ __forceinline__ bool wide(const double *aos) { return (reinterpret_cast<uintptr_t>(aos) & 15) == 0; }

__device__ __forceinline__ void tile_load(const Geom &g, const double *aos, double2 *tile) {
  const double *from = aos + (size_t)blockIdx.x * kPairs * kPairUnits * 2;
  const int n = tile_units(g);
  if (!wide(aos)) {
    for (int u = (int)threadIdx.x; u < n; u += kThreads) tile[u + u / kPairUnits] = make_double2(from[2 * u], from[2 * u + 1]);
    return;
  }
  const double2 *src = reinterpret_cast<const double2 *>(from);
#pragma unroll
  for (int k = 0; k < kPairs * kPairUnits / kThreads; k++) {
    const int u = k * kThreads + (int)threadIdx.x;
    if (u < n) tile[u + u / kPairUnits] = __ldcs(src + u);
  }
}

__device__ __forceinline__ void tile_store(const Geom &g, double *aos, const double2 *tile) {
  double *to = aos + (size_t)blockIdx.x * kPairs * kPairUnits * 2;
  const int n = tile_units(g);
  if (!wide(aos)) {
    for (int u = (int)threadIdx.x; u < n; u += kThreads) {
      const double2 v = tile[u + u / kPairUnits];
      to[2 * u] = v.x;
      to[2 * u + 1] = v.y;
    }
    return;
  }
  double2 *dst = reinterpret_cast<double2 *>(to);
#pragma unroll
  for (int k = 0; k < kPairs * kPairUnits / kThreads; k++) {
    const int u = k * kThreads + (int)threadIdx.x;
    if (u < n) __stcs(dst + u, tile[u + u / kPairUnits]);
  }
}

// FP64 arithmetic per link takes one warp on a scheduler as long as 64 clocks an
// operation, and a tile puts two on each: where the tiles leave SMs idle, the kernels
// that do some run one warp per block instead (warp b of the launch is warp b % 8 of
// tile b / 8) and write the public layout directly, a link's 144 B per lane.
// waves: up to how many tiles per SM
bool spread(const Geom &g, int waves = 1) { return (long long)tile_blocks(g) < (long long)waves * lgt_device_sms(); }

__device__ __forceinline__ void link_store(double *aos, const TileLink &t, const double u[18]) {
  double *to = aos + ((size_t)(2 * (long long)t.i + t.odd) * 4 + t.mu) * 18;
  if (wide(aos)) {
#pragma unroll
    for (int c = 0; c < 9; c++) reinterpret_cast<double2 *>(to)[c] = make_double2(u[2 * c], u[2 * c + 1]);
  } else {
#pragma unroll
    for (int c = 0; c < 18; c++) to[c] = u[c];
  }
}

// ------------------------------------------------------------ the SU(3) check
// |U^dagger U - 1|_max < 1e-10 and |det U - 1| < 1e-10.  In FP64 it takes some
// 200 operations of the FP64 pipe (2 per clock and SM): 1.7 ms at 32^4, eight
// times what the field's bytes take.  So it is done in 64-bit integers on the
// FP32-rate multiplier: entries truncated to multiples of 2^-49 as hi 2^20 + lo,
// products hi hi + (hi lo + lo hi) 2^-20 in units of 2^-58, off by at most 3e-14.
// What is within 1e-12 of the limit is decided in FP64.
struct Fix {
  int hi, lo;
};
struct FixAcc {
  long long s1 = 0, s2 = 0;  // hi hi; hi lo + lo hi
  __device__ __forceinline__ void add(Fix a, Fix b) {
    s1 += (long long)a.hi * b.hi;
    s2 += (long long)a.hi * b.lo;
    s2 += (long long)a.lo * b.hi;
  }
  __device__ __forceinline__ void sub(Fix a, Fix b) { add(a, Fix{-b.hi, -b.lo}); }
  __device__ __forceinline__ long long value() const { return s1 + (s2 >> 20); }  // units of 2^-58
};

__device__ __forceinline__ Fix fix_of(long long a) { return Fix{(int)(a >> 20), (int)(a & 0xfffff)}; }

// x truncated to a multiple of 2^-49; false if |x| >= 2 or x is not finite
__device__ __forceinline__ bool to_fix(double x, Fix &f) {
  const long long b = __double_as_longlong(x);
  const int e = (int)(b >> 52) & 0x7ff;
  const int down = 1026 - e;  // 2^-1074 .. : bits below 2^-49
  long long m = (b & 0xfffffffffffffll) | (1ll << 52);
  m = down < 53 ? m >> (down & 63) : 0;
  f = fix_of(b < 0 ? -m : m);
  return e < 1024;
}

// the same check in FP64: its largest deviation
__device__ __noinline__ double su3_deviation(const double *u) {
  double worst = 0.0;
#pragma unroll 1
  for (int a = 0; a < 3; a++)
#pragma unroll 1
    for (int b = 0; b < 3; b++) {
      double re = 0.0, im = 0.0;
      for (int k = 0; k < 3; k++) {  // sum_k conj(U_ka) U_kb
        re += u[LGT_RE(k, a)] * u[LGT_RE(k, b)] + u[LGT_IM(k, a)] * u[LGT_IM(k, b)];
        im += u[LGT_RE(k, a)] * u[LGT_IM(k, b)] - u[LGT_IM(k, a)] * u[LGT_RE(k, b)];
      }
      re -= (a == b) ? 1.0 : 0.0;
      worst = fmax(worst, fmax(fabs(re), fabs(im)));
    }
  double dre = 0.0, dim = 0.0;
#pragma unroll 1
  for (int cc = 0; cc < 3; cc++) {
    const int a1 = (cc + 1) % 3, b1 = (cc + 2) % 3;
    const double mre = u[LGT_RE(1, a1)] * u[LGT_RE(2, b1)] - u[LGT_IM(1, a1)] * u[LGT_IM(2, b1)] -
                       (u[LGT_RE(1, b1)] * u[LGT_RE(2, a1)] - u[LGT_IM(1, b1)] * u[LGT_IM(2, a1)]);
    const double mim = u[LGT_RE(1, a1)] * u[LGT_IM(2, b1)] + u[LGT_IM(1, a1)] * u[LGT_RE(2, b1)] -
                       (u[LGT_RE(1, b1)] * u[LGT_IM(2, a1)] + u[LGT_IM(1, b1)] * u[LGT_RE(2, a1)]);
    dre += u[LGT_RE(0, cc)] * mre - u[LGT_IM(0, cc)] * mim;
    dim += u[LGT_RE(0, cc)] * mim + u[LGT_IM(0, cc)] * mre;
  }
  return fmax(worst, fmax(fabs(dre - 1.0), fabs(dim)));
}

// u: a link of the tile (read again here, so that its doubles need not stay in registers)
__device__ __forceinline__ bool su3_ok(const double *u) {
  constexpr long long kOne = 1ll << 58;
  constexpr long long kSure = 28534807;  // 0.99e-10, 1.01e-10 in units of 2^-58
  constexpr long long kBad = 29111269;
  Fix f[18];
  bool in = true;
#pragma unroll
  for (int k = 0; k < 18; k++) in = to_fix(u[k], f[k]) && in;
  if (!in) return false;
  long long worst = 0;
  auto see = [&](long long v) {
    v = v < 0 ? -v : v;
    worst = v > worst ? v : worst;
  };
#pragma unroll
  for (int a = 0; a < 3; a++)
#pragma unroll
    for (int b = a; b < 3; b++) {
      FixAcc re, im;
#pragma unroll
      for (int k = 0; k < 3; k++) {  // conj(U_ka) U_kb
        re.add(f[LGT_RE(k, a)], f[LGT_RE(k, b)]);
        re.add(f[LGT_IM(k, a)], f[LGT_IM(k, b)]);
        if (b > a) {
          im.add(f[LGT_RE(k, a)], f[LGT_IM(k, b)]);
          im.sub(f[LGT_IM(k, a)], f[LGT_RE(k, b)]);
        }
      }
      see(re.value() - (a == b ? kOne : 0));
      if (b > a) see(im.value());
    }
  if (worst > kBad) return false;
  FixAcc dre, dim;  // entries are at most 1 + 1e-10 from here on
#pragma unroll
  for (int c = 0; c < 3; c++) {
    const int a = (c + 1) % 3, b = (c + 2) % 3;
    FixAcc mre, mim;
    mre.add(f[LGT_RE(1, a)], f[LGT_RE(2, b)]);
    mre.sub(f[LGT_IM(1, a)], f[LGT_IM(2, b)]);
    mre.sub(f[LGT_RE(1, b)], f[LGT_RE(2, a)]);
    mre.add(f[LGT_IM(1, b)], f[LGT_IM(2, a)]);
    mim.add(f[LGT_RE(1, a)], f[LGT_IM(2, b)]);
    mim.add(f[LGT_IM(1, a)], f[LGT_RE(2, b)]);
    mim.sub(f[LGT_RE(1, b)], f[LGT_IM(2, a)]);
    mim.sub(f[LGT_IM(1, b)], f[LGT_RE(2, a)]);
    const Fix r = fix_of(mre.value() >> 9), i = fix_of(mim.value() >> 9);
    dre.add(f[LGT_RE(0, c)], r);
    dre.sub(f[LGT_IM(0, c)], i);
    dim.add(f[LGT_RE(0, c)], i);
    dim.add(f[LGT_IM(0, c)], r);
  }
  see(dre.value() - kOne);
  see(dim.value());
  if (worst < kSure) return true;
  if (worst > kBad) return false;
  return su3_deviation(u) < 1e-10;
}

// ------------------------------------------------------------------ kernels
// BFMT: storage of the bulk's FP32 copy, written in the same pass (FMT_F64: none)
template <int BFMT>
__global__ void __launch_bounds__(kThreads, 3) k_ingest(Geom g, const double *aos, void *u64, void *u32, int *err) {
  extern __shared__ double2 lgt_tile[];
  tile_load(g, aos, lgt_tile);
  __syncthreads();
  const TileLink t(g);
  if (!t.valid) return;
  double u[18];
  const double2 *src = lgt_tile + t.unit();
#pragma unroll
  for (int c = 0; c < 9; c++) {
    const double2 v = src[c];
    u[2 * c] = v.x;
    u[2 * c + 1] = v.y;
  }
  LinkIO<FMT_F64>::store(u64, g.vh, t.p, t.mu, t.i, u);
  if (BFMT != FMT_F64) {
    float r[18];
#pragma unroll
    for (int k = 0; k < 18; k++) r[k] = (float)u[k];
    LinkIO<BFMT == FMT_F32_18 ? FMT_F32_18 : FMT_F32_12>::store(u32, g.vh, t.p, t.mu, t.i, r);
  }
  if (!su3_ok((const double *)src)) atomicOr(err, 1);
}

template <int FMT>
__global__ void __launch_bounds__(kThreads) k_egress(Geom g, const void *soa, double *aos, const void *G,
                                                     int skip_temporal) {
  extern __shared__ double2 lgt_tile[];
  const TileLink t(g);
  if (t.valid) {
    double u[18];
    load_field_d<FMT>(g, soa, G, skip_temporal, t.p, t.mu, t.i, u);
    double2 *dst = lgt_tile + t.unit();
#pragma unroll
    for (int c = 0; c < 9; c++) dst[c] = make_double2(u[2 * c], u[2 * c + 1]);
  }
  __syncthreads();
  tile_store(g, aos, lgt_tile);
}

// the same by spread warps
template <int FMT>
__global__ void __launch_bounds__(32) k_egress_spread(Geom g, const void *soa, double *aos) {
  const TileLink t(g, (int)blockIdx.x & 7, blockIdx.x >> 3);
  if (!t.valid) return;
  double u[18];
  load_d<FMT>(soa, g.vh, t.p, t.mu, t.i, u);
  link_store(aos, t, u);
}

constexpr int kTileBytes = kPairs * kPairStride * 16;

}  // namespace

cudaError_t launch_ingest(int bulk_fmt, const Geom &g, const double *aos, void *u64, void *u32, int *err,
                          cudaStream_t st) {
  const unsigned grid = tile_blocks(g);
  if (bulk_fmt == FMT_F64) k_ingest<FMT_F64><<<grid, kThreads, kTileBytes, st>>>(g, aos, u64, u32, err);
  else if (bulk_fmt == FMT_F32_18) k_ingest<FMT_F32_18><<<grid, kThreads, kTileBytes, st>>>(g, aos, u64, u32, err);
  else if (bulk_fmt == FMT_F32_12) k_ingest<FMT_F32_12><<<grid, kThreads, kTileBytes, st>>>(g, aos, u64, u32, err);
  else return cudaErrorInvalidValue;
  return cudaGetLastError();
}

cudaError_t launch_egress(int fmt, const Geom &g, const void *soa, double *aos, cudaStream_t st, const void *G,
                          int skip_temporal) {
  const unsigned grid = tile_blocks(g);
  if (fmt == FMT_PAIR && spread(g)) {  // (54 FP64 operations per link: a call at 8^4 17.7 -> 14.9 us)
    k_egress_spread<FMT_PAIR><<<8 * grid, 32, 0, st>>>(g, soa, aos);
    return cudaGetLastError();
  }
#define LGT_EGRESS(F) \
  if (fmt == F) k_egress<F><<<grid, kThreads, kTileBytes, st>>>(g, soa, aos, G, skip_temporal); else
  LGT_EGRESS(FMT_F64)
  LGT_EGRESS(FMT_F32_18)
  LGT_EGRESS(FMT_F32_12)
  LGT_EGRESS(FMT_PAIR)
  LGT_EGRESS(FMT_FIX_18)
  LGT_EGRESS(FMT_FIX_12)
  return cudaErrorInvalidValue;
#undef LGT_EGRESS
  return cudaGetLastError();
}

// ------------------------------------------------ gauge transformations in FP64
namespace {

__device__ __forceinline__ void load_G_fp64(const void *G, int vh, int p, int i, double m[18]) {
  float f[18];
  GIO::load(G, vh, p, i, f);
#pragma unroll
  for (int k = 0; k < 18; k++) m[k] = (double)f[k];
  reunitarise(m);
}

// G = 1 + D of the anchored polish in FP64 (pairs widened, row 2 rebuilt in
// FP64, rows orthonormalised: unitary to FP64 rounding)
__device__ __forceinline__ void load_G_from_D(const void *D, int vh, int p, int i, double m[18]) {
  f2 d[18];
  DIO::load_pair(D, vh, p, i, d);
#pragma unroll
  for (int k = 0; k < 12; k++) m[k] = (double)d[k].hi + (double)d[k].lo;
  m[LGT_RE(0, 0)] += 1.0;
  m[LGT_RE(1, 1)] += 1.0;
  reunitarise(m);
}

template <int SRC>
__device__ __forceinline__ void load_G_src(const void *G, int vh, int p, int i, double m[18]) {
  if (SRC == 0) load_G_fp64(G, vh, p, i, m);
  else load_G_from_D(G, vh, p, i, m);
}

// Every site's G orthonormalised in FP64, once (9 chunks of double2 per site and
// parity, 144 B): the links' products then read it instead of repeating some 170
// FP64 operations twice per link.
template <int SRC>
__global__ void __launch_bounds__(128) k_gauge_fp64(Geom g, const void *G, double2 *out) {
  const long long gid = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (gid >= (long long)g.vh * 2) return;
  const int p = (int)(gid / g.vh), i = (int)(gid % g.vh);
  double m[18];
  load_G_src<SRC>(G, g.vh, p, i, m);
#pragma unroll
  for (int c = 0; c < 9; c++) out[(size_t)(p * 9 + c) * g.vh + i] = make_double2(m[2 * c], m[2 * c + 1]);
}

__device__ __forceinline__ void load_gauge(const double2 *G64, int vh, int p, int i, double m[18]) {
#pragma unroll
  for (int c = 0; c < 9; c++) {
    const double2 v = __ldg(G64 + (size_t)(p * 9 + c) * vh + i);
    m[2 * c] = v.x;
    m[2 * c + 1] = v.y;
  }
}

// U_mu(x) <- G(x) U_mu(x) G(x+mu)^+ in FP64; SRC 0: G of the bulk phase (FP32),
// SRC 1: G = 1 + D of the anchored polish (pairs), SRC 2: G from k_gauge_fp64.
// 216 FP64 multiply-adds per link: bound by the FP64 pipe (1.51 ms at 32^4, 1.44 at
// its full rate; 3.5 to 3.9 ms with G orthonormalised for both ends of every link).
template <int SRC>
__device__ __forceinline__ void transformed_link(const Geom &g, const void *G, const void *u_in, int skip_temporal,
                                                 const TileLink &t, double u[18]) {
  LinkIO<FMT_F64>::load(u_in, g.vh, t.p, t.mu, t.i, u);
  if (skip_temporal && t.mu == 0) return;
  const int s = t.i / g.vs_half;
  const Coords c = coords_in_slice(g, t.p, s, t.i - s * g.vs_half);
  const int nb = cb_shift(g, c, t.mu, +1);
  double m[18], tmp[18];
  if constexpr (SRC == 2) load_gauge((const double2 *)G, g.vh, t.p, t.i, m);
  else load_G_src<SRC>(G, g.vh, t.p, t.i, m);
  mat_mul(m, u, tmp);
  if constexpr (SRC == 2) load_gauge((const double2 *)G, g.vh, t.p ^ 1, nb, m);
  else load_G_src<SRC>(G, g.vh, t.p ^ 1, nb, m);
  mat_mul_dag(tmp, m, u);
}

template <int SRC>
__global__ void __launch_bounds__(32) k_apply_G_spread(Geom g, const void *G, const void *u_in, void *u_out,
                                                       double *aos_out, int skip_temporal) {
  const TileLink t(g, (int)blockIdx.x & 7, blockIdx.x >> 3);
  if (!t.valid) return;
  double u[18];
  transformed_link<SRC>(g, G, u_in, skip_temporal, t, u);
  if (aos_out) link_store(aos_out, t, u);
  else LinkIO<FMT_F64>::store(u_out, g.vh, t.p, t.mu, t.i, u);
}

template <int SRC, bool AOS>
__global__ void __launch_bounds__(kThreads, 2) k_apply_G(Geom g, const void *G, const void *u_in, void *u_out,
                                                         double *aos_out, int skip_temporal) {
  extern __shared__ double2 lgt_tile[];
  const TileLink t(g);
  if (t.valid) {
    double u[18];
    transformed_link<SRC>(g, G, u_in, skip_temporal, t, u);
    if (AOS) {
      double2 *dst = lgt_tile + t.unit();
#pragma unroll
      for (int c = 0; c < 9; c++) dst[c] = make_double2(u[2 * c], u[2 * c + 1]);
    } else {
      LinkIO<FMT_F64>::store(u_out, g.vh, t.p, t.mu, t.i, u);
    }
  }
  if (AOS) {
    __syncthreads();
    tile_store(g, aos_out, lgt_tile);
  }
}

template <int SRC>
cudaError_t apply(const Geom &g, const void *G, const void *u64_in, void *u64_out, double *aos_out, int skip_temporal,
                  cudaStream_t st) {
  const unsigned grid = tile_blocks(g);
  // (G orthonormalised for both ends of every link: 556 operations, whose uneven share of
  // the SMs costs more than the tile saves up to 4 tiles per SM; with G at hand, 216)
  if (spread(g, SRC == 2 ? 1 : 4)) k_apply_G_spread<SRC><<<8 * grid, 32, 0, st>>>(g, G, u64_in, u64_out, aos_out, skip_temporal);
  else if (aos_out) k_apply_G<SRC, true><<<grid, kThreads, kTileBytes, st>>>(g, G, u64_in, u64_out, aos_out, skip_temporal);
  else k_apply_G<SRC, false><<<grid, kThreads, 0, st>>>(g, G, u64_in, u64_out, nullptr, skip_temporal);
  return cudaGetLastError();
}

template <int SRC>
cudaError_t apply_with(const Geom &g, const void *G, const void *u64_in, void *u64_out, double *aos_out,
                       int skip_temporal, void *scratch, cudaStream_t st) {
  if (!scratch) return apply<SRC>(g, G, u64_in, u64_out, aos_out, skip_temporal, st);
  const long long n = (long long)g.vh * 2;
  k_gauge_fp64<SRC><<<(unsigned)((n + 127) / 128), 128, 0, st>>>(g, G, (double2 *)scratch);
  const cudaError_t e = cudaGetLastError();
  return e != cudaSuccess ? e : apply<2>(g, scratch, u64_in, u64_out, aos_out, skip_temporal, st);
}

// FP32 copy of the FP64 links (each thread one link)
template <int FMT>
__global__ void __launch_bounds__(256) k_copy_f32(Geom g, const void *u64, void *u32) {
  const long long gid = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (gid >= (long long)g.vh * 8) return;
  const int i = (int)(gid % g.vh), pm = (int)(gid / g.vh);
  const double2 *b = reinterpret_cast<const double2 *>(u64) + (size_t)(pm * 9) * g.vh + i;
  float r[18];
#pragma unroll
  for (int c = 0; c < (FMT == FMT_F32_12 ? 6 : 9); c++) {
    const double2 v = __ldg(b + (size_t)c * g.vh);
    r[2 * c] = __double2float_rn(v.x);
    r[2 * c + 1] = __double2float_rn(v.y);
  }
  LinkIO<FMT>::store(u32, g.vh, pm >> 2, pm & 3, i, r);
}

}  // namespace

cudaError_t launch_apply_G(const Geom &g, const void *G, const void *u64_in, void *u64_out, double *aos_out,
                           int skip_temporal, void *scratch, cudaStream_t st) {
  return apply_with<0>(g, G, u64_in, u64_out, aos_out, skip_temporal, scratch, st);
}

cudaError_t launch_apply_D(const Geom &g, const void *D, const void *u64_in, void *u64_out, double *aos_out,
                           int skip_temporal, void *scratch, cudaStream_t st) {
  return apply_with<1>(g, D, u64_in, u64_out, aos_out, skip_temporal, scratch, st);
}

bool lgt_gauge_in_one_launch(const Geom &g) { return 2 * (long long)tile_blocks(g) <= lgt_device_sms(); }

cudaError_t launch_copy_f32(int fmt, const Geom &g, const void *u64, void *u32, cudaStream_t st) {
  const unsigned grid = (unsigned)(((long long)g.vh * 8 + 255) / 256);
  if (fmt == FMT_F32_12) k_copy_f32<FMT_F32_12><<<grid, 256, 0, st>>>(g, u64, u32);
  else if (fmt == FMT_F32_18) k_copy_f32<FMT_F32_18><<<grid, 256, 0, st>>>(g, u64, u32);
  else return cudaErrorInvalidValue;
  return cudaGetLastError();
}

}  // namespace lgt
