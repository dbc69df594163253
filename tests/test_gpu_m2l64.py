"""The FP64 M2L at orders and list lengths at the edges of its unrolled
degrees and lane batches, against the oracle's FMM."""
import numpy as np
import pytest

import ics
import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover - CPU container
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2012_02207_gb300 as gb  # noqa: E402


def solve(pos, m, **kw):
    f = gb.FMM(precision="fp64", **kw)
    cols = [torch.tensor(np.ascontiguousarray(c), dtype=torch.float64, device="cuda") for c in (*pos.T, m)]
    out = f.solve(*cols)
    return f, torch.stack(out[:3], 1).cpu().numpy(), out[3].cpu().numpy()


# the lowest orders, odd ones, both sides of the per-thread array sizes (16 and 30); a tolerance that accepts
# nearly every pair of a small tree, so lists are shorter than a warp; leaves of one body (r = 0)
@pytest.mark.parametrize("p,n,leaf,eps", [(1, 600, 8, 1e-2), (2, 600, 8, 1e-3), (3, 2000, 16, 1e-4), (7, 2000, 1, 1e-5),
                                          (11, 2000, 16, 1e-7), (15, 1500, 8, 1e-8), (17, 1500, 8, 1e-8),
                                          (25, 1000, 8, 1e-9), (29, 800, 4, 1e-9)])
def test_fp64_m2l_orders(p, n, leaf, eps):
    pos, _, _ = ics.plummer(n, 300 + p)
    m = ics.kroupa_masses(n, 301 + p)
    f, acc, pot = solve(pos, m, p=p, eps=eps, leaf_size=leaf)
    assert f.stats()["n_m2l"] > 100
    oacc, opot = oracle.fmm(pos, m, p=p, eps=eps, leaf_size=leaf)
    run = oracle.OracleRun(pos, m, p=p, eps=eps, leaf_size=leaf, stage=oracle.STAGE_F)
    fi = np.empty(n)
    fi[run.tree()["perm"]] = run.geometry()["f"]
    assert np.max(np.linalg.norm(acc - oacc, axis=1) / fi) <= 1e-12
    assert np.max(np.abs(pot - opot) / np.abs(opot)) <= 1e-12


def test_fp64_m2l_one_warp_per_target():
    """Enough cells that every warp takes targets of its own (above 16384), against the
    oracle."""
    pos, _, m = ics.plummer(60000, 9)
    f, acc, pot = solve(pos, m, p=5, eps=1e-6, leaf_size=4)
    assert f.stats()["nnodes"] > 16384
    oacc, opot = oracle.fmm(pos, m, p=5, eps=1e-6, leaf_size=4)
    run = oracle.OracleRun(pos, m, p=5, eps=1e-6, leaf_size=4, stage=oracle.STAGE_F)
    fi = np.empty(len(m))
    fi[run.tree()["perm"]] = run.geometry()["f"]
    assert np.max(np.linalg.norm(acc - oacc, axis=1) / fi) <= 1e-12
    assert np.max(np.abs(pot - opot) / np.abs(opot)) <= 1e-12


def test_fp64_forest_equals_separate_solves():
    """A forest above the cell count where a warp takes a whole target, of clusters that are below it alone."""
    sizes = [30000, 300, 35000, 1]
    offs = np.concatenate([[0], np.cumsum(sizes)])
    parts = [ics.plummer(n, 20 + n) for n in sizes]
    pos, m = np.concatenate([q[0] for q in parts]), np.concatenate([q[2] for q in parts])
    cols = [torch.tensor(np.ascontiguousarray(c), dtype=torch.float64, device="cuda") for c in (*pos.T, m)]
    f = gb.FMM(p=5, eps=1e-6, leaf_size=4, precision="fp64")
    out = torch.stack(f.solve_batch(offs, *cols))
    assert f.stats()["nnodes"] > 16384
    for a, b in zip(offs[:-1], offs[1:]):
        g = gb.FMM(p=5, eps=1e-6, leaf_size=4, precision="fp64")
        one = torch.stack(g.solve(*(c[a:b].contiguous() for c in cols)))
        assert torch.equal(one, out[:, a:b])


def test_fp64_m2l_source_counts():
    """A block takes a target; its four warps take the sources in batches of 32. Targets without sources, of one,
    part of one, two, three, four and more batches, against the oracle."""
    n, p, leaf, eps = 12000, 5, 8, 1e-5
    pos, _, m = ics.plummer(n, 10)
    f, acc, pot = solve(pos, m, p=p, eps=eps, leaf_size=leaf)
    count = np.bincount(f.export_pairs("m2l").ravel(), minlength=f.stats()["nnodes"])
    batches = np.bincount((count + 31) // 32)
    assert np.all(batches[:6] > 0) and np.any((count > 0) & (count < 32)) and np.any(count % 32 == 0)
    oacc, opot = oracle.fmm(pos, m, p=p, eps=eps, leaf_size=leaf)
    run = oracle.OracleRun(pos, m, p=p, eps=eps, leaf_size=leaf, stage=oracle.STAGE_F)
    fi = np.empty(n)
    fi[run.tree()["perm"]] = run.geometry()["f"]
    assert np.max(np.linalg.norm(acc - oacc, axis=1) / fi) <= 1e-12
    assert np.max(np.abs(pot - opot) / np.abs(opot)) <= 1e-12
