"""The forms in which a V-cycle's levels run, against the FP64 oracle: the up
leg as Q = P - D^-1 A P in each of its layouts."""
import json
import os
import subprocess
import sys

import numpy as np
import pytest

from paper_2002_04958_gb300 import inputs

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

# rows of level 0: one window of 256 less a row, exact, one more; a last window of one slice and a ragged one; 3-D
GRIDS = [(17, 15), (16, 16), (257, 2), (32, 17), (31, 35), (13, 11, 9)]

_APPLY = """
import json, sys
import torch
sys.path.insert(0, sys.argv[1])
from paper_2002_04958_gb300 import inputs, mgdamg
out = []
for dims, prec, interp in json.loads(sys.argv[2]):
    s = inputs.make_system(2, dims, multigroup=True)
    slv = mgdamg.Solver(autotune=1, batched=1, precision=prec, interp_type=interp, fuse_rows=-1).setup_system(s, "bd")
    out.append(slv.precond_apply(torch.from_numpy(s.b)).cpu().tolist())
print(json.dumps(out))
"""


@pytest.fixture(scope="module")
def gpu():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__ as ge
    ge.build()
    from paper_2002_04958_gb300 import mgdamg
    return mgdamg


def _apply(cases, path):
    p = subprocess.run([sys.executable, "-c", _APPLY, ROOT, json.dumps(cases)], capture_output=True, text=True,
                       env=dict(os.environ, MGD_TUNE_CACHE=str(path)), timeout=600)
    assert p.returncode == 0, p.stderr[-2000:]
    return [np.array(z) for z in json.loads(p.stdout.strip().splitlines()[-1])]


def test_q_layouts_match_oracle(gpu, orc, tmp_path):
    # every layout of the up leg forced on every level through the tuning file (0, 1, 9 and 10 name the
    # length-sorted SELL-32, 2 .. 6 CSR with 2 .. 32 threads a row).  The FP64 bound is that of the other
    # applies against the oracle; FP32 rounds some 100 operations deep, well inside 1e-4
    cases = [(d, p, i) for d in GRIDS for p, i in ((0, 0), (0, 1), (1, 0))]
    path = tmp_path / "tune.txt"
    _apply(cases, path)  # writes the tuned entries
    lines = path.read_text().splitlines()
    ref = []
    for dims, _, interp in cases:
        s = inputs.make_system(2, dims, multigroup=True)
        ref.append(orc.Block(orc.csr_of_system(s), s.G, s.N, "bd", orc.opts(interp_type=interp)).apply(s.b))
    same = None
    for f in (0, 1, 9, 10, 2, 3, 4, 5, 6):
        forced = []
        for ln in lines:
            fs = ln.split("|")
            depth = len(fs[1].split())
            if fs[3]:
                fs[3] = " ".join([str(f)] * depth)
            forced.append("|".join(fs))
        path.write_text("\n".join(forced) + "\n")
        got = _apply(cases, path)
        for (dims, prec, interp), z, zo in zip(cases, got, ref):
            tol = 1e-12 if prec == 0 else 1e-4
            assert np.linalg.norm(z - zo) <= tol * np.linalg.norm(zo), (f, dims, prec, interp)
        if f in (0, 1, 9, 10):  # the same kernel
            same = same or got
            assert all(np.array_equal(a, b) for a, b in zip(got, same)), f
