"""Output of transformed fields on lattices whose tiles leave SMs idle, which goes link
by link from one warp per block, and just above them, where it goes through tiles."""
import numpy as np
import pytest

import oracle as O
from test_gpu_fixed_links import lgt  # noqa: F401  (fixture)
from paper_1305_3440_gb300 import synth
from lattice_np import plaquettes

pytestmark = pytest.mark.gpu

# 1, 3, 64 and 105 tiles of 32 site pairs (below and above the rule for the scratch), 150,
# 157 and 160 around 152 SMs, 601 and 625 around four tiles per SM
DIMS = [(2, 2, 2, 2), (2, 2, 6, 6), (8, 8, 8, 8), (6, 10, 8, 14), (4, 8, 10, 30), (10, 10, 10, 10), (4, 10, 8, 32),
        (14, 14, 14, 14), (10, 10, 20, 20)]


def out_buffers(torch, dims):
    """The public layout on the device, 16-byte aligned and aligned to its doubles only."""
    n = int(np.prod(dims)) * 72
    raw = torch.zeros(n + 1, dtype=torch.float64, device="cuda")
    for off in (0, 1):
        flat = raw[off:off + n]
        yield flat, torch.view_as_complex(flat.view(-1, 2)).view(*dims, 4, 3, 3) if off == 0 else None


@pytest.mark.parametrize("dims", DIMS)
@pytest.mark.parametrize("kind", ["bulk", "bulk_plain_polish", "mag", "anchor", "anchor_sr", "pair", "no_temporal"])
def test_every_way_out_gives_the_same_gauge_transform(lgt, dims, kind):
    """Host memory, aligned and unaligned device memory: the same doubles; a gauge
    transform of the input (plaquettes to 1e-12, links unitary to 1e-13, those of pair
    storage to 3e-13: 2^-48 per update); and reading changes no later sweep."""
    import ctypes
    import torch
    U = synth.field(dims, 0.35, 161)
    kw = dict(dims=dims, bulk=lgt.LGT_FP32_12, omega=1.5, p=0.8, seed=5)
    kw.update({"bulk_plain_polish": dict(polish=lgt.LGT_POLISH_FP64), "mag": dict(gauge=lgt.LGT_MAG),
               "anchor_sr": dict(algo=lgt.LGT_SR), "pair": dict(polish=lgt.LGT_POLISH_PAIR),
               "no_temporal": dict(gauge=lgt.LGT_COULOMB, transform_temporal=0)}.get(kind, {}))
    after = []
    for read in (True, False):
        ctx = lgt.lgt_create(lgt.lgt_params_default(**kw), U)
        try:
            lgt.lgt_sweep(ctx, 3)
            if kind in ("anchor", "anchor_sr", "pair"):
                lgt.lgt_promote(ctx)
                lgt.lgt_sweep(ctx, 3)
            if read:
                host = lgt.lgt_get_links(ctx, dims)
                for flat, view in out_buffers(torch, dims):
                    assert lgt._lib.lgt_get_links(ctx, ctypes.c_void_p(flat.data_ptr()), 1) == lgt.LGT_OK
                    got = flat.cpu().numpy().view(np.complex128).reshape(host.shape)
                    assert np.array_equal(got, host)
            lgt.lgt_sweep(ctx, 2)
            after.append(lgt.lgt_get_links(ctx, dims))
        finally:
            lgt.lgt_destroy(ctx)
    assert np.array_equal(*after)
    planes = slice(3 if kind == "no_temporal" else 0, 6)
    assert np.abs(plaquettes(host) - plaquettes(U))[..., planes].max() < 1e-12
    one = np.einsum("...ab,...cb->...ac", host, host.conj())
    assert np.abs(one - np.eye(3)).max() < (3e-13 if kind == "pair" else 1e-13)
