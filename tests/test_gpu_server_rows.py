"""A batch of more rows than a warp has lanes: the batched FP32 sweeps find a
block's row 32 table entries at a time."""
import numpy as np
import pytest

from test_gpu_server import lgt, wait_all  # noqa: F401  (fixture)
from paper_1305_3440_gb300 import synth

pytestmark = pytest.mark.gpu


def test_seventy_rows_each_get_their_own_lattice(lgt):
    """70 jobs of three shapes, live together (a tolerance out of reach keeps each to
    its 2000 sweeps, bulk and polish), end bit for bit as the same job alone."""
    shapes = [(4, 4, 4, 6), (2, 6, 4, 4), (6, 2, 10, 4)]
    fields = {k: synth.field(shapes[k % 3], 0.4, 400 + k) for k in range(70)}

    def run(keys):
        srv = lgt.lgt_server_create(8 << 30, 0)
        try:
            ids = {}
            for k in keys:
                p = lgt.lgt_params_default(dims=shapes[k % 3], gauge=k % 2, bulk=1 + (k // 2) % 2, theta_tol=1e-40,
                                           max_sweeps=2000)
                ids[lgt.lgt_submit(srv, p, fields[k])] = k
            out = wait_all(lgt, srv, list(ids), {j: shapes[k % 3] for j, k in ids.items()})
            return {ids[j]: v for j, v in out.items()}
        finally:
            lgt.lgt_server_destroy(srv)

    mix = run(range(70))
    for k in (0, 1, 31, 32, 33, 63, 64, 65, 69):
        st, res, links = run([k])[k]
        assert mix[k][0] == st and mix[k][1]["sweeps_bulk"] == res["sweeps_bulk"] > 0
        assert mix[k][1]["F"] == res["F"] and np.array_equal(mix[k][2], links)
