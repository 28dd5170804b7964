"""The fixed-link FP32 bulk sweeps (the links stay as loaded, the accumulated
transformation G is the only state) against the FP64 oracle, through the C ABI,
where their index and storage arithmetic has its edges: extents of 2 (both
neighbours the same site), one 2-site row, partial and single blocks, both link
storages, both gauges, U_0 left alone, reunitarisation on and off."""
import numpy as np
import pytest

import oracle as O
from paper_1305_3440_gb300 import synth
from lattice_np import check_fp32_bound, fp32_half_sweep_bound, plaquettes

pytestmark = pytest.mark.gpu

GAUGES = {"landau": O.LANDAU, "coulomb": O.COULOMB}


@pytest.fixture(scope="module")
def lgt():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_1305_3440_gb300 import build
    build.build()
    from paper_1305_3440_gb300 import lgt as mod
    return mod


@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (2, 4, 6, 2), (4, 2, 2, 34), (2, 14, 6, 10)])
@pytest.mark.parametrize("bulk", ["fp32_18", "fp32_12"])
@pytest.mark.parametrize("gauge", list(GAUGES))
@pytest.mark.parametrize("reunit", [0, 1])
def test_half_sweeps_match_the_oracle_at_the_edges(lgt, dims, bulk, gauge, reunit):
    """Either half-sweep from a rough field: every entry of the working links and of
    the transformed FP64 field within max(5e-6, 16 u kappa) of the oracle's (the
    bound of every FP32 kernel: a K(x) off by 8u at the site that wrote the link)."""
    U = synth.field(dims, 0.5, 91)
    kw = dict(gauge=GAUGES[gauge], omega=1.7)
    for parity in (0, 1):
        ref = U.copy()
        O.half_sweep(ref, parity, **kw)
        bound = fp32_half_sweep_bound(O.site_conditioning(U, parity, **kw), parity, 16.0)
        p = lgt.lgt_params_default(dims=dims, bulk=getattr(lgt, "LGT_" + bulk.upper()), reunit_every=reunit, **kw)
        ctx = lgt.lgt_create(p, U)
        try:
            lgt.lgt_half_sweep(ctx, parity)
            work = lgt.lgt_get_working_links(ctx, dims)
            full = lgt.lgt_get_links(ctx, dims)
        finally:
            lgt.lgt_destroy(ctx)
        for out in (work, full):
            ratio, n_above, n_links = check_fp32_bound(np.abs(out - ref), bound)
            assert ratio <= 1.0, (parity, ratio, n_above, n_links)
        assert np.abs(plaquettes(full) - plaquettes(U)).max() < 1e-12


@pytest.mark.parametrize("bulk", ["fp32_18", "fp32_12"])
@pytest.mark.parametrize("temporal", [0, 1])
def test_working_field_is_measured_as_it_is_read(lgt, bulk, temporal):
    """Between bulk sweeps the measured field and the working links read back are one
    and the same (formed from the links and G): F, theta, plaquette and the slices'
    values are the oracle's on those links, to FP64 summation (1e-13; theta
    relative).  With transform_temporal = 0 the temporal links are the input's."""
    dims = (4, 6, 10, 14)
    U = synth.field(dims, 0.5, 92)
    p = lgt.lgt_params_default(dims=dims, bulk=getattr(lgt, "LGT_" + bulk.upper()), gauge=lgt.LGT_COULOMB,
                               omega=1.6, transform_temporal=temporal)
    ctx = lgt.lgt_create(p, U)
    try:
        lgt.lgt_sweep(ctx, 7)
        F, th, pl = lgt.lgt_measure(ctx)
        F_t, th_t = lgt.lgt_measure_slices(ctx, dims[0])
        sums = lgt.lgt_measure_slice_sums(ctx, dims[0])
        W = lgt.lgt_get_working_links(ctx, dims)
        lgt.lgt_sweep(ctx, 1)  # reading changes nothing: the sweeps go on
        after = lgt.lgt_get_working_links(ctx, dims)
    finally:
        lgt.lgt_destroy(ctx)
    m, mc = O.measure(W), O.measure(W, O.COULOMB)
    assert abs(F - mc["F_t"].mean()) < 1e-13 and abs(th - mc["theta_t"].max()) < 1e-13 * th
    assert np.allclose(F_t, mc["F_t"], rtol=0, atol=1e-13) and np.allclose(th_t, mc["theta_t"], rtol=1e-13, atol=0)
    assert abs(pl - m["plaq"]) < 1e-13
    vol = np.prod(dims)
    assert abs(sums[:, 0].sum() / (12 * vol) - m["F"]) < 1e-13
    if not temporal:
        assert np.abs(W[..., 0, :, :] - U[..., 0, :, :]).max() < 1e-6
    ctx = lgt.lgt_create(p, U)
    try:
        lgt.lgt_sweep(ctx, 8)
        straight = lgt.lgt_get_working_links(ctx, dims)
    finally:
        lgt.lgt_destroy(ctx)
    assert np.array_equal(after, straight)
