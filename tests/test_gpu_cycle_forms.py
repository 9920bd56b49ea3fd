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


# unknowns at which the Gram-Schmidt grid's units grow (116,736, 233,472 and 466,944 on 152 SMs), on either side, and
# the smallest: fewer than a unit, one block, a last unit of one entry
GS_GRIDS = [(3, 3), (64, 32), (11, 31), (512, 76), (357, 109), (304, 256), (275, 283), (512, 304), (395, 395)]


@pytest.mark.parametrize("dims", GS_GRIDS, ids=["x".join(map(str, d)) for d in GS_GRIDS])
def test_gram_schmidt_grid_matches_streaming(gpu, dims):
    # both orthogonalise by modified Gram-Schmidt, to rounding; right-hand sides: dense, one cell, and a
    # scale far from one with a decay over 13 orders of magnitude
    import torch
    s = inputs.make_system(1, dims, multigroup=True)
    rng = np.random.default_rng(5)
    point = np.zeros(s.n)
    point[s.n // 2] = 1.0
    grid = gpu.Solver(autotune=0, arnoldi_resident=1).setup_system(s, "schur1")
    stream = gpu.Solver(autotune=0, arnoldi_resident=0).setup_system(s, "schur1")
    for b in (s.b, point, 1e100 * np.exp(-30.0 * np.arange(s.n) / s.n) * rng.standard_normal(s.n)):
        b = torch.from_numpy(b)
        xg, itg, rg, _ = grid.solve(b)
        xs, its, rs, _ = stream.solve(b)
        assert itg == its
        assert torch.linalg.vector_norm(xg - xs) <= 1e-10 * torch.linalg.vector_norm(xs)
        assert np.allclose(grid.history(), stream.history(), rtol=1e-4, atol=1e-13)


# 8,190 and 8,256 unknowns, on either side of the line below which the blocks are one cluster, and clusters of one to
# sixteen blocks (81, 1,350 and 3,072 unknowns; the smaller grids above)
@pytest.mark.parametrize("dims", [(42, 65), (43, 64), (32, 32), (18, 25), (3, 3, 3)],
                         ids=lambda d: "x".join(map(str, d)))
def test_gram_schmidt_cluster_matches_streaming(gpu, dims):
    test_gram_schmidt_grid_matches_streaming(gpu, dims)


def test_gram_schmidt_grid_not_finite(gpu):
    # an infinity or a NaN in the right-hand side ends the solve with its status, as it did
    import torch
    s = inputs.make_system(1, (64, 32), multigroup=True)
    slv = gpu.Solver(autotune=0).setup_system(s, "schur1")
    for bad in (np.inf, np.nan):
        b = s.b.copy()
        b[777] = bad
        with pytest.raises(gpu.MgdError) as e:
            slv.solve(torch.from_numpy(b))
        assert e.value.code == 5
    x, it, rr, rc = slv.solve(torch.from_numpy(s.b))
    assert rc == 0 and rr <= 1e-8


_DENSE = """
import json, sys
import torch
sys.path.insert(0, sys.argv[1])
from paper_2002_04958_gb300 import inputs, mgdamg
out = []
for G, dims, kind, prec, smoother, trans in json.loads(sys.argv[2]):
    s = inputs.make_system(G, dims, multigroup=True)
    slv = mgdamg.Solver(autotune=1, batched=1, use_graph=1, precision=prec, smoother=smoother,
                        keep_transpose=trans, max_coarse=20).setup_system(s, kind)
    b = torch.from_numpy(s.b)
    lam = slv.solve_transpose(b)[0].cpu().tolist() if trans else []
    out.append(dict(tail=[p["tail"] for p in slv.plan()], depth=[p["depth"] for p in slv.plan()],
                    z=slv.precond_apply(b).cpu().tolist(), lam=lam))
print(json.dumps(out))
"""


def test_dense_coarse_levels_match_oracle(gpu, orc, tmp_path):
    # the levels from any one down as a dense matrix per subsystem (tail "level 1" in the tuning file), for both
    # smoothers, a stalled coarsest level (20 groups) and the transposed cycle; the FP64 bounds are those of the
    # other applies and transposed solves, FP32 as above
    cases = [(2, (19, 17), "bd", 0, 0, 1), (2, (19, 17), "amg", 0, 1, 1), (20, (13, 11), "schur2", 0, 0, 0),
             (20, (13, 11), "schur1", 0, 1, 0), (4, (23, 19), "bd", 1, 0, 0), (1, (40, 37), "amg", 0, 0, 1)]
    path = tmp_path / "tune.txt"

    def run():
        p = subprocess.run([sys.executable, "-c", _DENSE, ROOT, json.dumps(cases)], capture_output=True, text=True,
                           env=dict(os.environ, MGD_TUNE_CACHE=str(path)), timeout=600)
        assert p.returncode == 0, p.stderr[-2000:]
        return json.loads(p.stdout.strip().splitlines()[-1])

    run()
    lines = path.read_text().splitlines()
    ref = []
    for G, dims, kind, _, smoother, trans in cases:
        s = inputs.make_system(G, dims, multigroup=True)
        A = orc.csr_of_system(s)
        M = orc.Block(A, s.G, s.N, kind, orc.opts(smoother=smoother, max_coarse=20))
        ref.append((M.apply(s.b), orc.fgmres(A, s.b, M, tol=1e-8, transpose=True)[0] if trans else None))
    seen = set()
    for level in (1, 2, 3, 99):  # 99: no dense level
        forced = []
        for ln in lines:
            fs = ln.split("|")
            if len(fs[0].split()) > 3:
                fs[5] = f"{level} 1"
            forced.append("|".join(fs))
        path.write_text("\n".join(forced) + "\n")
        for case, r, (zo, lo) in zip(cases, run(), ref):
            for t, d in zip(r["tail"], r["depth"]):
                assert t == min(level, d), (level, case)
                seen.add(t < d)
            z = np.array(r["z"])
            tol = 1e-12 if case[3] == 0 else 1e-4
            assert np.linalg.norm(z - zo) <= tol * np.linalg.norm(zo), (level, case)
            if lo is not None:
                lam = np.array(r["lam"])
                assert np.linalg.norm(lam - lo) <= 1e-10 * np.linalg.norm(lo), (level, case)
    assert seen == {True, False}


@pytest.mark.parametrize("kind,interp,prec", [("bd", 0, 0), ("schur2", 1, 0), ("schur1", 0, 1)])
def test_joint_setup_many_operators(gpu, orc, kind, interp, prec):
    # the most operators one joint setup takes (30 groups, E and I), of which E stalls at once and the others end on
    # different levels: every level as the oracle sets it up alone, and the apply (bounds as above)
    import torch
    s = inputs.make_system(30, (23, 17), multigroup=True)
    slv = gpu.Solver(batched=1, precision=prec, interp_type=interp, max_coarse=20).setup_system(s, kind)
    M = orc.Block(orc.csr_of_system(s), s.G, s.N, kind, orc.opts(interp_type=interp, max_coarse=20))
    depths = set()
    for k in range(slv.stats()["n_ops"]):
        info = slv.op_info(k)
        h = M.amg(info["kind"], info["comp"])
        assert info["nlevels"] == h.nlevels
        depths.add(h.nlevels)
        for l in range(h.nlevels):
            g = slv.level(k, l)
            for name, m in (("", h.A(l)), ("p", h.P(l) if l < h.nlevels - 1 else None)):
                if m is not None:
                    rp, ci, v = m.arrays()
                    assert np.array_equal(g[name + "rp"], rp) and np.array_equal(g[name + "ci"], ci)
                    assert np.array_equal(g[name + "v"], v), (k, l, name)
    assert len(depths) > 1
    z = slv.precond_apply(torch.from_numpy(s.b)).cpu().numpy()
    zo = M.apply(s.b)
    assert np.linalg.norm(z - zo) <= (1e-12 if prec == 0 else 1e-4) * np.linalg.norm(zo)


def test_relres_refuses_matrices_it_refused(gpu):
    # the matrix check on the device: what the host-side checks refused, and the output stays as it was; an empty
    # matrix may have any columns (none is read)
    import torch
    s = inputs.make_system(2, (31, 17), multigroup=True)
    dev = torch.device("cuda")
    rp, ci, va, b = (torch.from_numpy(a).to(dev) for a in (s.rowptr, s.col, s.val, s.b))
    x = torch.zeros_like(b)
    out = torch.full((3,), -1.0, dtype=torch.float64, device=dev)
    assert gpu.relres_noalloc(rp, ci, va, b, x, out) == 0
    assert out[2].item() == pytest.approx(1.0, rel=1e-14)

    def changed(a, at, value):
        a = a.clone()
        a[at] = value
        return a
    bad = [(changed(rp, 0, 1), ci, va, "rowptr\\[0\\]"), (rp, ci[:-1], va, "rowptr\\[0\\]"), (rp, ci, va[:-1], "rowptr\\[0\\]"),
           (changed(rp, 100, int(rp[101]) + 1), ci, va, "non-decreasing"), (rp, changed(ci, 500, -1), va, "columns"),
           (rp, changed(ci, -1, s.n), va, "columns")]
    for r, c, v, msg in bad:
        out.fill_(-1.0)
        with pytest.raises(ValueError, match=msg):
            gpu.relres_noalloc(r, c.contiguous(), v.contiguous(), b, x, out)
        assert torch.equal(out, torch.full_like(out, -1.0))
    assert gpu.relres_noalloc(torch.zeros_like(rp), torch.full_like(ci, -7), va, b, x, out) == 0
    assert out[0].item() == out[1].item()
    side = torch.cuda.Stream()
    assert gpu.relres_noalloc(rp, ci, va, b, x, out, stream=side) == 0
