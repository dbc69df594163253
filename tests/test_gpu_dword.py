"""P2M and M2M in double-word arithmetic against FP64, by the degree norms.

Sizes around the places where the kernels divide their work: leaves of one
body to several chunks of 32, columns whose entries take 1, 2, 4 or 8 lanes
(2 (p - m + 1) entries of order m), the lowest and the highest order.
Harmonics in hat form are at most 1, so a degree norm is at most M s^n. A step
of a recurrence or a translation is a few operations of at most 8 u^2 each
(u = 2^-24) relative to that, with some p steps in a chain, over the levels
of the tree: the bound is 64 (p + 4) u^2.
"""
import numpy as np
import pytest

import ics

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,leaf", [(1, 1), (31, 64), (33, 64), (257, 256), (700, 1), (3000, 9), (20000, 100)])
@pytest.mark.parametrize("p", [1, 2, 4, 7, 10, 16])
def test_double_word_moments(n, leaf, p):
    import torch

    import paper_2012_02207_gb300 as gb

    pos = ics.plummer(n, 5)[0]
    m = ics.kroupa_masses(n, 6)
    cols = [torch.tensor(np.ascontiguousarray(pos[:, d]), device="cuda") for d in range(3)]
    cols.append(torch.tensor(m, device="cuda"))
    g = {}
    for precision in ("mixed", "fp64"):
        f = gb.FMM(p=p, eps=1e-3, leaf_size=leaf, precision=precision)
        f.solve(*cols)
        g[precision] = f.export_geometry()
    r, mass = g["fp64"]["r"], g["fp64"]["M"]
    wide = r > 2.0**-9 * r.max()
    size = r[wide, None] ** np.arange(p + 1) * mass[wide, None]
    err = np.abs(g["mixed"]["P"] - g["fp64"]["P"])[wide]
    assert np.all(err <= 64 * (p + 4) * 2.0**-48 * size)


@pytest.mark.parametrize("n,leaf,more_than", [(20000, 9, 2048), (60000, 9, 16384)])
@pytest.mark.parametrize("p", [4, 10])
def test_double_word_moments_of_large_trees(n, leaf, more_than, p):
    """A warp per leaf from 2048 nodes on, a thread per node for the norms from 16384 on."""
    import paper_2012_02207_gb300 as gb

    test_double_word_moments(n, leaf, p)
    import torch

    pos = ics.plummer(n, 5)[0]
    cols = [torch.tensor(np.ascontiguousarray(c), device="cuda") for c in (*pos.T, ics.kroupa_masses(n, 6))]
    f = gb.FMM(p=p, eps=1e-3, leaf_size=leaf)
    f.solve(*cols)
    assert f.stats()["nnodes"] > more_than


def test_moments_do_not_depend_on_how_the_work_is_divided():
    """A tree of few nodes alone (four warps to a leaf, four threads to a node's norms) and in a forest of
    many (one): the same norms."""
    import torch

    import paper_2012_02207_gb300 as gb

    sizes = [1500, 60000]
    pos = np.concatenate([ics.plummer(n, 5)[0] for n in sizes])
    m = np.concatenate([ics.kroupa_masses(n, 6) for n in sizes])
    cols = [torch.tensor(np.ascontiguousarray(c), device="cuda") for c in (*pos.T, m)]
    f, one = gb.FMM(p=8, eps=1e-3, leaf_size=9), gb.FMM(p=8, eps=1e-3, leaf_size=9)
    f.solve_batch([0, sizes[0], sum(sizes)], *cols)
    one.solve(*(c[: sizes[0]].contiguous() for c in cols))
    assert one.stats()["nnodes"] < 2048 and f.stats()["nnodes"] > 16384
    own = f.export_tree()["begin"] < sizes[0]  # the first cluster's nodes, level by level as in its own tree
    assert np.array_equal(f.export_geometry()["P"][own], one.export_geometry()["P"])
