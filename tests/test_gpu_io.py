"""The field in and out of a context: tiles of 32 site pairs with a partial last one
(and a lattice smaller than one), every storage, and the SU(3) check's decisions
around its limit."""
import numpy as np
import pytest

from paper_1305_3440_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lgt():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_1305_3440_gb300 import build
    build.build()
    from paper_1305_3440_gb300 import lgt as mod
    return mod


@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (2, 4, 6, 2), (4, 2, 2, 34), (4, 6, 10, 14)])
@pytest.mark.parametrize("bulk", ["fp64", "fp32_18", "fp32_12"])
def test_links_go_in_and_out_exactly(lgt, dims, bulk):
    """Loaded links come back bit for bit (G = 1); the FP32 working links are the
    rounded ones (row 2 of 12-real storage rebuilt: 4 products of FP32 entries)."""
    U = synth.field(dims, 0.5, 41)
    ctx = lgt.lgt_create(lgt.lgt_params_default(dims=dims, bulk=getattr(lgt, "LGT_" + bulk.upper())), U)
    try:
        assert np.array_equal(lgt.lgt_get_links(ctx, dims), U)
        W = lgt.lgt_get_working_links(ctx, dims)
        assert np.array_equal(lgt.lgt_get_links(ctx, dims), U)
    finally:
        lgt.lgt_destroy(ctx)
    R = U.astype(np.complex64).astype(np.complex128)
    rows = slice(0, 2) if bulk == "fp32_12" else slice(0, 3)
    assert np.array_equal(W[..., rows, :], (U if bulk == "fp64" else R)[..., rows, :])
    assert np.abs(W - U).max() < 6 * 2.0**-24


@pytest.mark.parametrize("polish", [0, 1, 2])
@pytest.mark.parametrize("gauge", [0, 1, 2])
def test_output_is_the_same_before_and_after_promotion(lgt, polish, gauge):
    """The field read out of the bulk phase (G applied on the way) and the one that
    promotion forms in place are the same products (bit for bit; FP32 pairs hold 48
    bits of them), with and without memory for the orthonormal G; a read between
    polish sweeps changes nothing."""
    dims = (4, 6, 10, 14)
    U = synth.field(dims, 0.4, 42)
    p = lgt.lgt_params_default(dims=dims, gauge=gauge, bulk=lgt.LGT_FP32_12, polish=polish, omega=1.6)
    out = []
    for read in (True, False):
        ctx = lgt.lgt_create(p, U)
        try:
            lgt.lgt_sweep(ctx, 3)
            before = lgt.lgt_get_links(ctx, dims) if read else None
            lgt.lgt_promote(ctx)
            after = lgt.lgt_get_links(ctx, dims)
            lgt.lgt_sweep(ctx, 2)
            if read:
                mid = lgt.lgt_get_links(ctx, dims)
            lgt.lgt_sweep(ctx, 1)
            end = lgt.lgt_get_links(ctx, dims)
        finally:
            lgt.lgt_destroy(ctx)
        if read:
            assert np.abs(before - after).max() < (2.0**-46 if polish == 0 and gauge != 2 else 1e-15)
            assert not np.array_equal(mid, after)
        out.append(end)
    assert np.array_equal(out[0], out[1])


@pytest.mark.parametrize("bulk", ["fp64", "fp32_18", "fp32_12"])
def test_device_buffers_need_only_the_alignment_of_doubles(lgt, bulk):
    """Links read from and written to device memory that is 8 but not 16 bytes aligned:
    load, output with and without a transformation, the working links, and the
    measurement straight from the caller's buffer, against the aligned buffer's."""
    import torch
    dims = (4, 6, 10, 14)
    U = synth.field(dims, 0.5, 44)
    n = 2 * U.size
    p = lgt.lgt_params_default(dims=dims, bulk=getattr(lgt, "LGT_" + bulk.upper()), omega=1.6)
    got = {}
    for off in (0, 1):
        def buffer():
            t = torch.full((n + 2,), 7.0, dtype=torch.float64, device="cuda")
            return t, t[off:off + n].view(dims + (4, 3, 3, 2))
        whole, links = buffer()
        assert links.data_ptr() % 16 == 8 * off
        links.copy_(torch.view_as_real(torch.from_numpy(U)))
        sums = torch.empty(8 + 2 * dims[0], dtype=torch.float64, device="cuda")
        outs = []
        ctx = lgt.lgt_create(p, links)
        try:
            for sweeps in (0, 2):
                if sweeps:
                    lgt.lgt_sweep(ctx, sweeps)
                for read in (lgt.lgt_get_links, lgt.lgt_get_working_links):
                    w, out = buffer()
                    read(ctx, out=out)
                    assert float(w[n + off:].min()) == 7.0 and (off == 0 or float(w[0]) == 7.0)
                    outs.append(out.cpu().numpy())
            lgt.lgt_promote(ctx)
            lgt.lgt_sweep(ctx, 1)
            w, out = buffer()
            lgt.lgt_get_links(ctx, out=out)
            outs.append(out.cpu().numpy())
        finally:
            lgt.lgt_destroy(ctx)
        torch.cuda.synchronize()
        lgt.lgt_measure_noalloc(dims, links, sums)
        torch.cuda.synchronize()
        got[off] = outs + [sums.cpu().numpy()]
    assert np.array_equal(got[0][0], U.view(np.float64).reshape(dims + (4, 3, 3, 2)))
    for a, b in zip(got[0], got[1]):
        assert np.array_equal(a, b)


def _deviation(u):
    """max(|U^+ U - 1|, |Re det U - 1|, |Im det U|) of one matrix in extended precision."""
    u = u.astype(np.clongdouble)
    h = np.array([[sum(u[k, a].conj() * u[k, b] for k in range(3)) for b in range(3)] for a in range(3)])
    h -= np.eye(3)
    det = sum(u[0, c] * (u[1, (c + 1) % 3] * u[2, (c + 2) % 3] - u[1, (c + 2) % 3] * u[2, (c + 1) % 3]) for c in range(3))
    return float(max(np.abs(h.real).max(), np.abs(h.imag).max(), abs(det.real - 1), abs(det.imag)))


@pytest.mark.parametrize("bulk", ["fp64", "fp32_12"])
def test_the_su3_check_decides_as_in_extended_precision(lgt, bulk):
    """One link off SU(3) by a scale, a phase, a shear or one entry, from far inside
    the limit of 1e-10 to far outside and 1e-14 on either side of it (the check is
    made on 49-bit fixed-point entries, and in FP64 near the limit)."""
    dims = (2, 2, 4, 2)
    base = synth.field(dims, 0.5, 43)
    p = lgt.lgt_params_default(dims=dims, bulk=getattr(lgt, "LGT_" + bulk.upper()))
    ctx = lgt.lgt_create(p, base)

    def accepted(U):
        try:
            lgt.lgt_load(ctx, U)
            return True
        except lgt.LgtError as e:
            assert e.status == lgt.LGT_EINVAL
            return False

    try:
        rng = np.random.default_rng(1)
        kinds = {"scale": lambda u, d: u * (1 + d / 2), "phase": lambda u, d: u * np.exp(1j * d / 3),
                 "shear": lambda u, d: u + d * u[[1, 0, 2]] * np.array([[1], [0], [0]]),
                 "entry": lambda u, d: u + d * np.eye(3)[[2, 1, 0]] * np.array([[1], [0], [0]])}
        for kind, off in kinds.items():
            seen = set()
            for size in (1e-13, 3e-11, 0.9e-10, 0.98e-10, 0.9999e-10, 1.0001e-10, 1.02e-10, 2e-10, 1e-6, 0.3):
                U = base.copy()
                at = tuple(int(rng.integers(n)) for n in dims) + (int(rng.integers(4)),)
                u = U[at]
                d = size
                for _ in range(6):  # to a deviation of `size`
                    got = _deviation(off(u, d))
                    d *= min(max(size / got, 0.2), 5.0)
                U[at] = off(u, d)
                dev = _deviation(U[at])
                if abs(dev - 1e-10) < 1e-15:
                    continue
                ok = accepted(U)
                assert ok == (dev < 1e-10), (kind, size, dev)
                seen.add(ok)
            assert seen == {True, False}, kind
        for bad in (np.nan, np.inf, -np.inf, 2.0, -3.0, 1e300, complex(0, np.nan)):
            for k in range(9):
                U = base.copy()
                U.reshape(-1)[9 * 5 + k] = bad
                assert not accepted(U), (bad, k)
        U = base.copy()
        U[0, 0, 0, 0, 0] = np.diag([1, 1e-320, 1]) + 0j  # a denormal where a one should be
        assert not accepted(U)
        U[0, 0, 0, 0, 0] = np.eye(3)
        U[0, 0, 0, 0, 0, 0, 1] = 1e-320
        assert accepted(U)
    finally:
        lgt.lgt_destroy(ctx)
