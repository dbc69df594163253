"""The in-block HOLD step at set sizes around its chunks and mask words: the
oracle's trajectory bit for bit."""
import numpy as np
import pytest

import ics
import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover - CPU container
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2012_02207_gb300 as gb  # noqa: E402


# 31..33 and 1024: whole and broken chunks of 1024 pairs, one row a chunk; a dt at which nobody, some or all are fast
@pytest.mark.parametrize("n,dt,soft", [(1, 0.1, 0.0), (2, 0.5, 0.0), (3, 0.01, 0.0), (31, 1 / 16, 0.0),
                                       (33, 1 / 16, 1e-2), (65, 1 / 8, 0.0), (300, 1 / 64, 0.0), (513, 1e-3, 0.0),
                                       (1024, 2e-4, 0.0), (1024, 1e-6, 1e-3)])
@pytest.mark.parametrize("sym", [True, False])
def test_one_step_bit_exact(n, dt, soft, sym):
    pos, vel, _ = ics.plummer(n, 90 + n, center=False)
    m = ics.kroupa_masses(n, 91)
    w = [torch.tensor(np.ascontiguousarray(c), dtype=torch.float64, device="cuda") for c in (*pos.T, *vel.T)]
    mt = torch.tensor(m, device="cuda")
    got = gb.FMM(soft=soft).hold(*w, mt, dt=dt, nsteps=1, eta=0.025, symmetrize=sym, dt_min=0.0)
    opos, ovel, stats = oracle.hold(pos, vel, m, dt, 1, eta=0.025, sym=sym, soft=soft)
    assert np.array_equal(torch.stack(w[:3], 1).cpu().numpy(), opos)
    assert np.array_equal(torch.stack(w[3:], 1).cpu().numpy(), ovel)
    assert got["kicks"] == stats["kicks"] and got["max_depth"] == stats["max_depth"]
