"""LGT_SWEEP_PDL=0 stands for plain launches, whoever launches: the sweeps read links,
K0 and job tables before they wait for the launch before them, so the switch has to
reach every launch that may overlap it."""
import glob
import os
import re
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_one_place_sets_the_overlap_and_heeds_the_switch():
    """The launch attribute is set in one function, which asks the switch; both the
    single-lattice and the batched sweeps launch through it."""
    src = {os.path.basename(f): re.sub(r"//[^\n]*", "", open(f).read())
           for f in glob.glob(os.path.join(ROOT, "paper_1305_3440_gb300", "csrc", "*"))}
    setters = [f for f, s in src.items() for _ in re.findall(r"cudaLaunchAttributeProgrammatic\w+", s)]
    assert setters == ["lgt_internal.h"], setters
    body = src["lgt_internal.h"].split("cudaLaunchAttributeProgrammaticStreamSerialization")[1].split("}")[0]
    assert re.search(r"numAttrs = overlap && lgt_use_pdl\(\)", body), body
    for f in ("lgt_kernels.cu", "lgt_batch.cu"):
        assert "launch_sweep(" in src[f]


_RUN = """
import sys
import numpy as np
sys.path.insert(0, {root!r}); sys.path.insert(0, {tests!r})
from paper_1305_3440_gb300 import lgt, synth
from test_gpu_server import JOBS, run_server
out = run_server(lgt, JOBS)
np.savez(sys.argv[1], **{{str(k): v[2] for k, v in enumerate(out)}}, F=[v[1]["F"] for v in out])
"""


@pytest.mark.gpu
def test_served_jobs_do_not_depend_on_the_overlap(tmp_path):
    """The server's mix of jobs with and without overlapping launches: bit for bit the
    same fields."""
    import numpy as np
    got = {}
    for v in ("1", "0"):
        path = str(tmp_path / f"out{v}.npz")
        r = subprocess.run([sys.executable, "-c", _RUN.format(root=ROOT, tests=os.path.join(ROOT, "tests")), path],
                           env=dict(os.environ, LGT_SWEEP_PDL=v), capture_output=True, text=True, timeout=600)
        assert r.returncode == 0, r.stdout + r.stderr
        got[v] = np.load(path)
    assert sorted(got["0"].files) == sorted(got["1"].files) and len(got["0"].files) > 2
    for k in got["0"].files:
        assert np.array_equal(got["0"][k], got["1"][k]), k
