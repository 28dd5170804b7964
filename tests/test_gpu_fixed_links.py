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


_FORCED = """
import sys
import numpy as np
sys.path.insert(0, {root!r}); sys.path.insert(0, {tests!r})
import oracle as O
from paper_1305_3440_gb300 import lgt, synth
from lattice_np import check_fp32_bound, fp32_half_sweep_bound
cfg = {cfg}
near = synth.field((4, 4, 4, 8), 0.3, 1)
O.fix(near, omega=1.7, tol=1e-12, max_sweeps=2000, check_every=1)
for gauge in (O.LANDAU, O.COULOMB):
    for dims in {dims}:
        U = synth.field(dims, 0.5, 93)
        for bulk in (lgt.LGT_FP32_18, lgt.LGT_FP32_12):
            for parity in (0, 1):
                ref = U.copy()
                O.half_sweep(ref, parity, gauge=gauge, omega=1.7)
                bound = fp32_half_sweep_bound(O.site_conditioning(U, parity, gauge=gauge, omega=1.7), parity, 16.0)
                ctx = lgt.lgt_create(lgt.lgt_params_default(dims=dims, bulk=bulk, gauge=gauge, omega=1.7), U)
                lgt.lgt_half_sweep(ctx, parity)
                out = lgt.lgt_get_working_links(ctx, dims)
                st = lgt.lgt_get_stats(ctx)
                F, th, _, _ = lgt.lgt_estimate(ctx, dims[0])
                lgt.lgt_destroy(ctx)
                assert st.launch_config[0] == cfg, list(st.launch_config)
                ratio, _, _ = check_fp32_bound(np.abs(out - ref), bound)
                assert ratio <= 1.0, (gauge, dims, bulk, parity, ratio)
                if parity == 0 and gauge == O.LANDAU:  # the parity-0 slots hold every link once
                    assert abs(F - O.measure(U)["F"]) < 16 * 2.0**-24
    if cfg == 16:  # FP64 sweeps: the same operations with u smaller by 2^-29
        for dims in {dims}:
            U = synth.field(dims, 0.5, 93)
            for parity in (0, 1):
                ref = U.copy()
                O.half_sweep(ref, parity, gauge=gauge, omega=1.7)
                bound = fp32_half_sweep_bound(O.site_conditioning(U, parity, gauge=gauge, omega=1.7), parity, 16.0) * 2.0**-29
                ctx = lgt.lgt_create(lgt.lgt_params_default(dims=dims, bulk=lgt.LGT_FP64, gauge=gauge, omega=1.7), U)
                lgt.lgt_half_sweep(ctx, parity)
                out = lgt.lgt_get_links(ctx, dims)
                st = lgt.lgt_get_stats(ctx)
                lgt.lgt_destroy(ctx)
                assert st.launch_config[0] == cfg, list(st.launch_config)
                ratio, _, _ = check_fp32_bound(np.abs(out - ref), bound, 5e-6 * 2.0**-29)
                assert ratio <= 1.0, (gauge, dims, parity, ratio)
    if cfg not in (3, 4, 16):
        continue
    for algo in (O.OR, O.SR) if cfg == 3 else (O.OR,):  # the anchored polish (SR: configurations 0-3 and 11)
        kw = dict(gauge=gauge, algo=algo, omega=1.7, p=0.8, seed=5)
        ref = near.copy()
        O.sweeps(ref, 2, **kw)
        ctx = lgt.lgt_create(lgt.lgt_params_default(dims=near.shape[:4], bulk=lgt.LGT_FP32_12, omega_polish=0.0, **kw), near)
        lgt.lgt_promote(ctx)
        lgt.lgt_sweep(ctx, 2)
        out = lgt.lgt_get_links(ctx, near.shape[:4])
        st = lgt.lgt_get_stats(ctx)
        lgt.lgt_destroy(ctx)
        assert st.launch_config[1] == cfg, list(st.launch_config)
        err = np.abs(out - ref).max()
        # theta of the field in this gauge sets |g - 1|, the angles are FP32
        m = O.measure(near, gauge)
        th = m["theta_t"].max() if gauge == O.COULOMB else m["theta"]
        assert err < 1e-12 + 2e-6 * np.sqrt(th), (gauge, algo, err, th)
print("ok")
"""


@pytest.mark.parametrize("cfg", [3, 4, 8, 9, 16])
def test_every_tuned_configuration(lgt, cfg, tmp_path):
    """Each configuration the autotuner may pick for the fixed-link bulk and (3, 4, 16)
    the anchored polish -- one thread per site at four budgets, four threads per site
    (4) -- forced through a tuning cache file, at the edges of its blocks and quads:
    half-sweeps within the per-site FP32 bound of the oracle, the fused F, and two
    polish sweeps within the accuracy of FP32 rotation angles; 16 also for FP64."""
    import os
    import subprocess
    import sys
    import torch
    here = os.path.dirname(os.path.abspath(__file__))
    dims = [(2, 2, 2, 2), (2, 4, 6, 2), (2, 6, 10, 14), (4, 2, 2, 34)]
    name = torch.cuda.get_device_name().replace(" ", "_")
    cache = tmp_path / "tuned"
    with open(cache, "w") as f:
        for fmt in (0, 4, 5, 6, 7):  # FP64; anchored polish (7: SR); fixed links, 18- and 12-real
            if (fmt == 0 and cfg != 16) or (fmt == 7 and cfg != 3):
                continue
            for gauge in (0, 1):
                for algo in (0, 1):
                    for d in dims + [(4, 4, 4, 8)]:
                        f.write(f"{fmt} {gauge} {algo} {d[0]} {d[1]} {d[2]} {d[3]} {name} {cfg if fmt != 4 or cfg in (3, 4, 16) else 0}\n")
    code = _FORCED.format(root=os.path.dirname(here), tests=here, cfg=cfg, dims=dims)
    r = subprocess.run([sys.executable, "-c", code], env=dict(os.environ, LGT_AUTOTUNE_CACHE=str(cache)),
                       capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and r.stdout.strip().endswith("ok"), r.stdout + r.stderr
