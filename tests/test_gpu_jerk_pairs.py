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
