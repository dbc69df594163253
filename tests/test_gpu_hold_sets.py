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


# both sides of the size where a chunk of pairs is cut into tiles of columns (257), and partly slow sets above it:
# one chunk of a few slow rows, whole and broken chunks of 16
@pytest.mark.parametrize("n,dt", [(256, 1 / 128), (257, 1 / 128), (258, 1e-6), (600, 1 / 512), (777, 1 / 256), (1000, 1 / 2048),
                                  (1023, 1e-6)])
def test_large_sets_bit_exact(n, dt):
    test_one_step_bit_exact(n, dt, 0.0, True)


def test_cost_of_a_kick_grows_with_its_pairs():
    """Steps in which nobody is fast are two kicks of all pairs: four times as many at 1024 bodies as at 512.
    (With one row of pairs at a time, whose sum is a serial chain, 1024 bodies took 6 times as long.)"""
    ms = {}
    for n in (512, 1024):
        pos, vel, m = ics.plummer(n, 7)
        w = [torch.tensor(np.ascontiguousarray(c), dtype=torch.float64, device="cuda") for c in (*pos.T, *vel.T, m)]
        f = gb.FMM()
        t = []
        for _ in range(4):
            a, b = torch.cuda.Event(True), torch.cuda.Event(True)
            a.record()
            st = f.hold(*w, dt=1e-9, nsteps=5, eta=0.025, dt_min=0.0)
            b.record()
            b.synchronize()
            t.append(a.elapsed_time(b))
        assert st["kicks"] == 10 and st["max_depth"] == 0
        ms[n] = min(t[1:])
    assert ms[1024] < 5.0 * ms[512], ms
