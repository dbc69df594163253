"""The FP32 near jerk takes a lane's terms in pairs: leaf sizes that give one
to many lanes per target, odd and even counts of terms, and full packs, with
every pair direct, against the direct jerk. Bound: that of the same comparison
at one leaf size in test_gpu_jerk.py, 1e-5 of J_i = sum_j m_j |v_ij| / r_ij^3.
"""
import numpy as np
import pytest

import ics
import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("soft", [0.0, 0.02])
@pytest.mark.parametrize("n,leaf", [(2, 1), (3, 4), (31, 32), (33, 64), (257, 256), (600, 11), (1500, 3), (3000, 40),
                                    (4000, 150)])
def test_mixed_near_jerk(n, leaf, soft):
    import torch

    import paper_2012_02207_gb300 as gb

    pos, vel, _ = ics.plummer(n, 21)
    m = ics.kroupa_masses(n, 22)
    cols = [torch.tensor(np.ascontiguousarray(c), device="cuda") for c in (*pos.T, *vel.T, m)]
    f = gb.FMM(p=4, eps=0.0, leaf_size=leaf, precision="mixed", soft=soft)
    jerk = torch.stack(f.solve_jerk(*cols)[4:7], 1).cpu().numpy()
    ref = oracle.direct_jerk(pos, vel, m, soft=soft)
    scale = np.zeros(n)
    for i in range(0, n, 256):
        d, u = pos[None] - pos[i:i + 256, None], vel[None] - vel[i:i + 256, None]
        r2 = (d * d).sum(-1) + soft * soft
        r2[np.arange(len(r2)), np.arange(i, i + len(r2))] = np.inf  # the body itself
        scale[i:i + 256] = (m[None] * np.linalg.norm(u, axis=-1) / r2**1.5).sum(1)
    assert np.max(np.linalg.norm(jerk - ref, axis=1) / scale) <= 1e-5


def test_fp64_jerk_does_not_depend_on_the_size_of_the_tree():
    """Work items are shorter slices of a leaf's targets below 2048 cells. Two trees with the same cluster,
    one on each side of that: the other bodies are as good as massless and in octants of their own, where the
    cluster sees them as one cell (or one body), so every sum over the cluster has the same terms."""
    import torch

    import paper_2012_02207_gb300 as gb

    rng = np.random.default_rng(5)
    n = 3001
    pos = -0.5 + 0.02 * rng.standard_normal((n, 3)).clip(-2.0, 2.0)
    vel = rng.standard_normal((n, 3))
    corners = np.array([[-1.0, 1.0, -1.0], [1.0, -1.0, 1.0]])  # they set the cube
    out, cells = [], []
    for extra in (1, 9000):
        other = 0.5 + 0.02 * rng.standard_normal((extra, 3)).clip(-2.0, 2.0)
        q = np.concatenate([pos, corners, other])
        u = np.concatenate([vel, np.zeros((2 + extra, 3))])
        m = np.concatenate([np.full(n, 1.0 / n), np.full(2 + extra, 1e-300)])
        f = gb.FMM(p=8, eps=1e-6, leaf_size=13, precision="fp64")
        cols = [torch.tensor(np.ascontiguousarray(c), device="cuda") for c in (*q.T, *u.T, m)]
        out.append(torch.stack(f.solve_jerk(*cols))[:, :n])
        cells.append(f.stats()["nnodes"])
    assert cells[0] < 2048 < cells[1]
    assert torch.equal(out[0], out[1])
