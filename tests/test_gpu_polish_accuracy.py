"""Accuracy of the anchored polish by overrelaxation.

At omega = 1 it does the same sweeps as the polish by stochastic relaxation that
never squares (p = 0), whose body holds all of K(x) in FP32 pairs, and as the polish in
FP64: the distances of the two from the FP64 polish of the same field compare them."""
import numpy as np
import pytest

import oracle as O
from test_gpu_fixed_links import lgt  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu

DIMS = [(6, 8, 10, 8), (8, 8, 8, 8), (4, 6, 10, 14), (10, 6, 12, 8)]


def near_one(rng, shape, eps):
    """SU(3) matrices at a distance of about eps from one (polar part of 1 + noise)."""
    m = np.eye(3) + eps * (rng.standard_normal(shape + (3, 3)) + 1j * rng.standard_normal(shape + (3, 3)))
    u, _, vh = np.linalg.svd(m)
    m = u @ vh
    return m / (np.linalg.det(m) ** (1 / 3))[..., None, None]


def nearly_fixed(dims, seed):
    """A constant background, stationary in either gauge, with violations of 1e-4: links
    and a gauge transformation that far from one."""
    rng = np.random.default_rng(seed)
    h = near_one(rng, dims, 1e-4)
    U = np.empty(dims + (4, 3, 3), np.complex128)
    for mu, axis in enumerate((0, 3, 2, 1)):
        link = near_one(rng, (), 0.2) @ near_one(rng, dims, 1e-4)
        U[..., mu, :, :] = h @ link @ np.conj(np.swapaxes(np.roll(h, -1, axis), -1, -2))
    return U


@pytest.mark.parametrize("gauge", [O.LANDAU, O.COULOMB])
def test_no_further_from_64_bits_than_the_polish_in_pairs(lgt, gauge):
    """12 polish sweeps three ways: the rms distance from FP64, averaged over the fields
    (each field's ratio scatters by a tenth), is no larger than that of the body in
    pairs."""
    ratios = []
    for n, dims in enumerate(DIMS):
        U = nearly_fixed(dims, 130 + n)
        out = {}
        for name, kw in {"fp64": dict(algo=lgt.LGT_OR, polish=lgt.LGT_POLISH_FP64),
                         "or": dict(algo=lgt.LGT_OR, polish=lgt.LGT_POLISH_ANCHOR),
                         "pairs": dict(algo=lgt.LGT_SR, p=0.0, polish=lgt.LGT_POLISH_ANCHOR)}.items():
            p = lgt.lgt_params_default(dims=dims, gauge=gauge, bulk=lgt.LGT_FP32_12, omega=1.0, omega_polish=0.0,
                                       polish_algo=lgt.LGT_POLISH_SAME, **kw)
            ctx = lgt.lgt_create(p, U)
            try:
                lgt.lgt_promote(ctx)
                lgt.lgt_sweep(ctx, 12)
                out[name] = lgt.lgt_get_links(ctx, dims)
            finally:
                lgt.lgt_destroy(ctx)
        rms = {k: np.sqrt(np.mean(np.abs(v - out["fp64"]) ** 2)) for k, v in out.items()}
        assert 0 < rms["pairs"] < 1e-9, rms
        ratios.append(rms["or"] / rms["pairs"])
    assert np.mean(ratios) <= 1.0, ratios
