"""How far a driver of its own gets with the FP32 bulk sweeps alone: lgt_sweep and
lgt_estimate, without promotion, down to theta < 1e-13."""
import numpy as np
import pytest

import oracle as O
from test_gpu_fixed_links import lgt  # noqa: F401  (fixture)
from paper_1305_3440_gb300 import synth
from lattice_np import plaquettes

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims", [(8, 8, 8, 8), (4, 6, 10, 14)])
@pytest.mark.parametrize("bulk", ["FP32_18", "FP32_12"])
@pytest.mark.parametrize("gauge,temporal", [(O.LANDAU, 1), (O.COULOMB, 1), (O.COULOMB, 0)])
@pytest.mark.parametrize("read", ["estimate", "measure", "slices"])
def test_sweeps_and_checks_reach_1e_13(lgt, dims, bulk, gauge, temporal, read):
    """10 sweeps and a check, until theta < 1e-13 (what the rewritten links reach within
    700 sweeps on these fields): the working links and the transformed input are that
    far fixed (the former to the FP32 rounding of its links, 3e-14), the latter is a
    gauge transform of the input, and the context goes on: a promotion and a polish."""
    U = synth.field(dims, 0.35, 141)
    p = lgt.lgt_params_default(dims=dims, gauge=gauge, bulk=getattr(lgt, "LGT_" + bulk), omega=1.7,
                               transform_temporal=temporal, theta_tol=1e-15)
    ctx = lgt.lgt_create(p, U)
    try:
        for n in range(90):
            lgt.lgt_sweep(ctx, 10)
            if read == "slices":
                th = lgt.lgt_measure_slices(ctx, dims[0])[1]
                th = th.max() if gauge == O.COULOMB else lgt.lgt_estimate(ctx, dims[0])[1]
            else:
                th = lgt.lgt_estimate(ctx, dims[0])[1] if read == "estimate" else lgt.lgt_measure(ctx)[1]
            if th < 1e-13:
                break
        assert th < 1e-13, (n, th)
        W, V = lgt.lgt_get_working_links(ctx, dims), lgt.lgt_get_links(ctx, dims)
        lgt.lgt_load(ctx, V)  # a new field: the next one starts from its own links
        lgt.lgt_sweep(ctx, 1)
        lgt.lgt_promote(ctx)
        lgt.lgt_sweep(ctx, 20)
        th_polish = lgt.lgt_measure(ctx)[1]
    finally:
        lgt.lgt_destroy(ctx)
    for out in (W, V):
        m = O.measure(out, gauge)
        assert (m["theta_t"].max() if gauge == O.COULOMB else m["theta"]) < 2e-13
    planes = slice(0 if temporal else 3, 6)  # U_0 left alone: the spatial plaquettes are invariant
    assert np.abs(plaquettes(V) - plaquettes(U))[..., planes].max() < 1e-12
    if not temporal:
        assert np.abs(V[..., 0, :, :] - U[..., 0, :, :]).max() < 1e-14
    assert th_polish < 1e-13


def test_a_reading_of_a_rough_field_changes_no_sweep(lgt):
    """Above 1e-10 reading leaves the sweeps bit for bit as they are."""
    dims = (8, 8, 8, 8)
    U = synth.field(dims, 0.35, 142)
    out = []
    for reads in (False, True):
        ctx = lgt.lgt_create(lgt.lgt_params_default(dims=dims, bulk=lgt.LGT_FP32_12, omega=1.7), U)
        try:
            for _ in range(12):
                lgt.lgt_sweep(ctx, 10)
                if reads:
                    assert lgt.lgt_estimate(ctx, dims[0])[1] > 1e-10 and lgt.lgt_measure(ctx)[1] > 1e-10
            out.append(lgt.lgt_get_working_links(ctx, dims))
        finally:
            lgt.lgt_destroy(ctx)
    assert np.array_equal(*out)
