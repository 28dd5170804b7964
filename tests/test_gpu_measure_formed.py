"""Measuring between fixed-link bulk sweeps, where each link is formed from U and G as
it is read: the values at the edges of the block-size rule, and the cost."""
import numpy as np
import pytest

import oracle as O
from test_gpu_fixed_links import lgt  # noqa: F401  (fixture)
from paper_1305_3440_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (2, 4, 6, 10), (8, 8, 8, 8), (10, 10, 10, 12), (16, 10, 10, 12)])
@pytest.mark.parametrize("bulk", ["FP32_18", "FP32_12"])
def test_values_are_those_of_the_links_read_back(lgt, dims, bulk):
    """One block, partial blocks of 64 and of 128, both sides of the rule's line: F, theta
    and plaquette as the oracle has them from the working links (FP64 summation: 1e-13)."""
    ctx = lgt.lgt_create(lgt.lgt_params_default(dims=dims, bulk=getattr(lgt, "LGT_" + bulk), omega=1.6),
                         synth.field(dims, 0.4, 151))
    try:
        lgt.lgt_sweep(ctx, 3)
        F, th, pl = lgt.lgt_measure(ctx)
        F_t, th_t = lgt.lgt_measure_slices(ctx, dims[0])
        W = lgt.lgt_get_working_links(ctx, dims)
    finally:
        lgt.lgt_destroy(ctx)
    m, mc = O.measure(W), O.measure(W, O.COULOMB)
    assert abs(F - m["F"]) < 1e-13 and abs(th - m["theta"]) < 1e-13 * th and abs(pl - m["plaq"]) < 1e-13
    assert np.allclose(F_t, mc["F_t"], rtol=0, atol=1e-13) and np.allclose(th_t, mc["theta_t"], rtol=1e-13, atol=0)


@pytest.mark.parametrize("dims", [(4, 4, 4, 4), (8, 8, 8, 8)])
def test_a_formed_field_takes_no_longer_to_measure_than_a_stored_one(lgt, dims):
    """Device time of a measurement with plaquette after a sweep, against a context whose
    sweeps rewrite their links (launch_config named): at most 1.05 of it."""
    U = synth.field(dims, 0.4, 152)
    ctx, times = {}, {}
    try:
        for name, k in (("formed", 0), ("stored", 9)):
            ctx[name] = lgt.lgt_create(lgt.lgt_params_default(dims=dims, bulk=lgt.LGT_FP32_12, launch_config=k), U)
            lgt.lgt_sweep(ctx[name], 1)
            times[name] = []
        for _ in range(80):  # in turn: a change of clocks meets both
            for name, c in ctx.items():
                a = lgt.lgt_get_stats(c).measure_ms
                lgt.lgt_measure(c)
                times[name].append(lgt.lgt_get_stats(c).measure_ms - a)
    finally:
        for c in ctx.values():
            lgt.lgt_destroy(c)
    us = {name: float(np.median(t[20:])) * 1e3 for name, t in times.items()}
    assert us["formed"] <= 1.05 * us["stored"], us
