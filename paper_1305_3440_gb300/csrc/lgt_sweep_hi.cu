// lgt_sweep_hi.cu -- the higher-precision half-sweep kernels: FP64 (every
// operation in FP64), FP32-pair and anchored (the polishing sweeps), one
// instantiation per gauge, algorithm and launch configuration.
#include "lgt_anchor_sr.cuh"
#include "lgt_fixed.cuh"
#include "lgt_sweep.cuh"

namespace lgt {

template <int GAUGE, int ALGO, int CFG>
__global__ void __launch_bounds__(lgt_cfg_threads(CFG), lgt_cfg_minblocks(CFG)) k_sweep_f64(SweepArgs in, int p) {
  pdl_enter();
  const SweepArgs a = resolve_loop(in);
  int t, bx;
  sweep_block_tile(a, p, t, bx);
  if constexpr (GAUGE == GAUGE_MAG) {
    sweep_body_mag<FMT_F64, double, ALGO>(a, p, t, bx);
  } else {
    sweep_body_f64<GAUGE, ALGO>(a, p, t, bx, gridDim.x);
  }
}

template <int GAUGE, int ALGO, int CFG>
__global__ void __launch_bounds__(lgt_cfg_threads(CFG), lgt_cfg_minblocks(CFG)) k_sweep_pair(SweepArgs in, int p) {
  pdl_enter();
  const SweepArgs a = resolve_loop(in);
  int t, bx;
  sweep_block_tile(a, p, t, bx);
  sweep_body_pair<GAUGE, ALGO>(a, p, t, bx, gridDim.x);
}

template <int GAUGE, int CFG>
__global__ void __launch_bounds__(lgt_cfg_threads(CFG), lgt_cfg_minblocks(CFG)) k_sweep_anchor(SweepArgs in, int p) {
  int t, bx;
  sweep_block_tile(in, p, t, bx);
  if constexpr (lgt_cfg_quad(CFG)) sweep_body_anchor_quad<GAUGE>(in, p, t, bx);
  else sweep_body_anchor<GAUGE, anchor_depth(CFG)>(in, p, t, bx);
}

template <int GAUGE, int CFG>
__global__ void __launch_bounds__(lgt_cfg_threads(CFG), lgt_cfg_minblocks(CFG)) k_sweep_anchor_sr(SweepArgs in, int p) {
  pdl_enter();
  const SweepArgs a = resolve_loop(in);
  int t, bx;
  sweep_block_tile(a, p, t, bx);
  anchor_sr::sweep_body_anchor_sr<GAUGE>(a, p, t, bx);
}

// FP64 and FP32-pair sweeps
template <int CFG>
static sweep_fn pick_links(int fmt, int gauge, int algo) {
  if (gauge == GAUGE_MAG) {  // maximally Abelian gauge: FP64 only here, configurations 0-3
    if constexpr (lgt_cfg_mag(CFG)) {
      if (fmt == FMT_F64 && algo == ALGO_OR) return k_sweep_f64<GAUGE_MAG, ALGO_OR, CFG>;
      if (fmt == FMT_F64 && algo == ALGO_SR) return k_sweep_f64<GAUGE_MAG, ALGO_SR, CFG>;
    }
    return nullptr;
  }
  if (fmt == FMT_F64) {
    if constexpr (CFG == 0) {  // the annealing sweeps run in configuration 0 only
      if (algo == ALGO_SA)
        return gauge == GAUGE_LANDAU ? k_sweep_f64<GAUGE_LANDAU, ALGO_SA, CFG> : k_sweep_f64<GAUGE_COULOMB, ALGO_SA, CFG>;
    }
    if (algo == ALGO_SA) return nullptr;
    if (gauge == GAUGE_LANDAU) return algo == ALGO_SR ? k_sweep_f64<GAUGE_LANDAU, ALGO_SR, CFG> : k_sweep_f64<GAUGE_LANDAU, ALGO_OR, CFG>;
    return algo == ALGO_SR ? k_sweep_f64<GAUGE_COULOMB, ALGO_SR, CFG> : k_sweep_f64<GAUGE_COULOMB, ALGO_OR, CFG>;
  }
  if (algo == ALGO_SA) return nullptr;
  if constexpr (lgt_cfg_supported(FMT_PAIR, CFG)) {
    if (fmt == FMT_PAIR) {
      if (gauge == GAUGE_LANDAU) return algo == ALGO_SR ? k_sweep_pair<GAUGE_LANDAU, ALGO_SR, CFG> : k_sweep_pair<GAUGE_LANDAU, ALGO_OR, CFG>;
      return algo == ALGO_SR ? k_sweep_pair<GAUGE_COULOMB, ALGO_SR, CFG> : k_sweep_pair<GAUGE_COULOMB, ALGO_OR, CFG>;
    }
  }
  return nullptr;
}

template <int CFG>
static sweep_fn pick_cfg(int fmt, int gauge, int algo) {
  if (fmt == FMT_ANCHOR || fmt == FMT_ANCHOR_SR) {
    if (gauge == GAUGE_MAG || algo != (fmt == FMT_ANCHOR ? ALGO_OR : ALGO_SR)) return nullptr;
    if (fmt == FMT_ANCHOR) return gauge == GAUGE_LANDAU ? k_sweep_anchor<GAUGE_LANDAU, CFG> : k_sweep_anchor<GAUGE_COULOMB, CFG>;
    if constexpr (lgt_cfg_supported(FMT_ANCHOR_SR, CFG))
      return gauge == GAUGE_LANDAU ? k_sweep_anchor_sr<GAUGE_LANDAU, CFG> : k_sweep_anchor_sr<GAUGE_COULOMB, CFG>;
    return nullptr;
  }
  // (4, four threads per site, and 11, 24 warps per SM at <= 80 registers: the anchored polish only)
  if constexpr (lgt_cfg_supported(FMT_F64, CFG)) return pick_links<CFG>(fmt, gauge, algo);
  else return nullptr;
}

sweep_fn pick_sweep_hi(int fmt, int gauge, int algo, int cfg) {
  switch (cfg) {
    case 0: return pick_cfg<0>(fmt, gauge, algo);
    case 1: return pick_cfg<1>(fmt, gauge, algo);
    case 2: return pick_cfg<2>(fmt, gauge, algo);
    case 3: return pick_cfg<3>(fmt, gauge, algo);
    case 4: return pick_cfg<4>(fmt, gauge, algo);
    case 11: return pick_cfg<11>(fmt, gauge, algo);
    case 16: return pick_cfg<16>(fmt, gauge, algo);
  }
  return nullptr;
}

}  // namespace lgt
