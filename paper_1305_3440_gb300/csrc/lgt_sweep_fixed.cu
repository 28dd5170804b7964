// lgt_sweep_fixed.cu -- the fixed-link FP32 bulk half-sweep kernels
// (lgt_fixed.cuh), one instantiation per link storage, gauge, algorithm and
// launch configuration.
#include "lgt_fixed.cuh"

namespace lgt {

template <int LFMT, int GAUGE, int ALGO, int CFG>
__global__ void __launch_bounds__(lgt_cfg_threads(CFG), lgt_cfg_minblocks(CFG)) k_sweep_fixed(SweepArgs in, int p) {
  int t, bx;
  sweep_block_tile(in, p, t, bx);
  if constexpr (lgt_cfg_quad(CFG)) sweep_body_fixed_quad<LFMT, GAUGE>(in, p, t, bx);
  else sweep_body_fixed<LFMT, GAUGE, ALGO, fixed_depth(LFMT, lgt_cfg_minblocks(CFG) * lgt_cfg_threads(CFG))>(in, p, t, bx);
}

template <int CFG>
static sweep_fn pick_cfg(int lfmt, int gauge, int algo) {
#define LGT_PICK(F, G, A) \
  if (lfmt == F && gauge == G && algo == A) return k_sweep_fixed<F, G, A, CFG>;
  LGT_PICK(FMT_F32_18, GAUGE_LANDAU, ALGO_OR)
  LGT_PICK(FMT_F32_18, GAUGE_COULOMB, ALGO_OR)
  LGT_PICK(FMT_F32_12, GAUGE_LANDAU, ALGO_OR)
  LGT_PICK(FMT_F32_12, GAUGE_COULOMB, ALGO_OR)
  if constexpr (CFG == LGT_FIXED_SA_CFG) {  // the annealing sweeps run in one configuration only
    LGT_PICK(FMT_F32_18, GAUGE_LANDAU, ALGO_SA)
    LGT_PICK(FMT_F32_18, GAUGE_COULOMB, ALGO_SA)
    LGT_PICK(FMT_F32_12, GAUGE_LANDAU, ALGO_SA)
    LGT_PICK(FMT_F32_12, GAUGE_COULOMB, ALGO_SA)
  }
#undef LGT_PICK
  return nullptr;
}

sweep_fn pick_sweep_fixed(int fmt, int gauge, int algo, int cfg) {
  const int lfmt = fmt == FMT_FIX_18 ? FMT_F32_18 : FMT_F32_12;
  switch (cfg) {
    case 3: return pick_cfg<3>(lfmt, gauge, algo);
    case 4: return pick_cfg<4>(lfmt, gauge, algo);
    case 8: return pick_cfg<8>(lfmt, gauge, algo);
    case 9: return pick_cfg<9>(lfmt, gauge, algo);
    case 16: return pick_cfg<16>(lfmt, gauge, algo);
  }
  return nullptr;
}

}  // namespace lgt
