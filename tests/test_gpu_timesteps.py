"""Step sizes found through FP32 bounds equal the oracle's bit for bit,
including where the bounds cannot decide and every pair is evaluated."""
import numpy as np
import pytest

import ics
import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover - CPU container
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2012_02207_gb300 as gb  # noqa: E402


def check(pos, vel, m, eta=0.025, G=1.0):
    cols = [torch.tensor(np.ascontiguousarray(c), dtype=torch.float64, device="cuda") for c in (*pos.T, *vel.T, m)]
    f = gb.FMM(G=G)
    for sym in (False, True):
        got = f.timesteps(*cols, eta=eta, symmetrize=sym).cpu().numpy()
        assert np.array_equal(got, oracle.taus(pos, vel, m, G=G, eta=eta, sym=sym))


@pytest.mark.parametrize("n", [1, 2, 3, 255, 256, 257, 513, 3000])
def test_sizes(n):
    pos, vel, _ = ics.plummer(n, 70 + n, center=False)
    check(pos, vel, ics.kroupa_masses(n, 71))


@pytest.mark.parametrize("case", ["binaries", "at rest", "same velocity", "far from the origin", "tiny", "huge",
                                  "heavy", "eta 1", "eta small", "G", "head on"])
def test_edges_of_the_bounds(case):
    rng = np.random.default_rng(3)
    n = 400
    pos, vel, _ = ics.plummer(n, 72, center=False)
    m = ics.kroupa_masses(n, 73)
    eta, G = 0.025, 1.0
    if case == "binaries":  # separations down to 1e-13 of the coordinates
        k = n // 2
        pos[k:] = pos[:k] + rng.normal(size=(k, 3)) * 10.0 ** rng.uniform(-13, -1, (k, 1))
        vel[k:] = vel[:k] + rng.normal(size=(k, 3)) * 10.0 ** rng.uniform(-13, 3, (k, 1))
    elif case == "at rest":
        vel[:] = 0.0
    elif case == "same velocity":
        vel[:] = vel[0]
        vel[::7] += 1e-9
    elif case == "far from the origin":
        pos += 1e9
        vel += 1e7
    elif case == "tiny":
        pos *= 1e-12
    elif case == "huge":
        pos *= 1e25
        vel *= 1e15
    elif case == "heavy":
        m = m * 1e12
    elif case == "eta 1":
        eta = 1.0
    elif case == "eta small":
        eta = 1e-9
    elif case == "G":
        G = 4.3e-3
    else:  # nearly radial encounters, in and out, and exactly circular ones
        for i in range(0, n, 2):
            d = rng.normal(size=3)
            pos[i + 1] = pos[i] + 1e-3 * d
            vel[i + 1] = vel[i] + (d if i % 4 else np.cross(d, [1.0, 0.0, 0.0])) * 10.0 ** rng.uniform(-2, 3)
    check(pos, vel, m, eta=eta, G=G)


# lengths, speeds and masses of the caller's units (G to match), from rest, and with bodies whose exponents pull the
# bounds' units away from the rest's: far out, heavy, at the origin or at the same place as another's first
@pytest.mark.parametrize("length,mass,G", [(3.086e16, 1.989e30, 6.674e-11), (3.086e18, 1.989e33, 6.674e-8),
                                           (1.0, 1.0, 4.49e-3), (1e-120, 1e-200, 1.0), (1e30, 1e-40, 1e-20)])
@pytest.mark.parametrize("case", ["", "at rest", "common velocity", "outliers", "at the origin"])
def test_units(length, mass, G, case):
    rng = np.random.default_rng(4)
    n = 300
    pos, vel, _ = ics.plummer(n, 74, center=False)
    m = ics.kroupa_masses(n, 75)
    if case == "at rest":
        vel[:] = 0.0
        vel[::50] = rng.normal(size=(6, 3))
    elif case == "common velocity":
        vel[:] = [0.1, -0.2, 0.3]
    elif case == "outliers":
        pos[::40] *= 1e12
        m[5::40] *= 1e15
        vel[::9] *= 1e-14
    elif case == "at the origin":
        pos[0] = 0.0
        pos[1:200] *= 1e-5
    check(pos * length, vel * np.sqrt(G * mass / length), m * mass, G=G)


def test_time_does_not_depend_on_the_units_or_the_velocities():
    """SI units and a start from rest cost what N-body units do (where no bound decides, every pair is
    evaluated exactly, which takes 18 times as long)."""
    n = 16384
    pos, vel, m = ics.plummer(n, 76)
    L, M, G = 3.086e16, 1.989e30, 6.674e-11
    ms = []
    for p, v, w, g in ((pos, vel, m, 1.0), (pos * L, vel * np.sqrt(G * M / L), m * M, G), (pos, 0.0 * vel, m, 1.0)):
        cols = [torch.tensor(np.ascontiguousarray(c), dtype=torch.float64, device="cuda") for c in (*p.T, *v.T, w)]
        f = gb.FMM(G=g)
        t = []
        for _ in range(5):
            a, b = torch.cuda.Event(True), torch.cuda.Event(True)
            a.record()
            f.timesteps(*cols, eta=0.025)
            b.record()
            b.synchronize()
            t.append(a.elapsed_time(b))
        ms.append(min(t[1:]))
    assert max(ms) < 3.0 * ms[0], ms
