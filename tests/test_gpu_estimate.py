"""The near part of the scalar-force estimate against the oracle, bit for bit,
at the edges of its tiles, in every split of the work and outside the range of
its fast division."""
import numpy as np
import pytest

import ics
import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover - CPU container
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2012_02207_gb300 as gb  # noqa: E402

# one leaf, a leaf of exactly one or two target chunks, one body more; small leaves; many cells above 64 bodies a leaf
SIZES = [(1, 64), (32, 32), (33, 33), (64, 64), (129, 256), (257, 256), (700, 7), (5000, 33), (420000, 65)]


def check(pos, m, leaf, soft=0.0):
    f = gb.FMM(p=4, eps=1e-4, leaf_size=leaf, soft=soft)
    cols = [torch.tensor(np.ascontiguousarray(c), dtype=torch.float64, device="cuda") for c in (*pos.T, m)]
    f.solve(*cols)
    run = oracle.OracleRun(pos, m, p=4, eps=1e-4, leaf_size=leaf, stage=oracle.STAGE_F, soft=soft)
    got, want = f.export_geometry(), run.geometry()
    assert np.array_equal(got["f"], want["f"])
    assert np.array_equal(got["fmin"], want["fmin"])


@pytest.mark.parametrize("soft", [0.0, 1e-3])
@pytest.mark.parametrize("n,leaf", SIZES)
def test_estimate_bit_exact(n, leaf, soft):
    if soft and n > 100000:
        pytest.skip("the softened terms take the general division at every size")
    pos, _, _ = ics.plummer(n, 40 + n, center=False)
    check(pos, ics.kroupa_masses(n, 41 + n), leaf, soft)


@pytest.mark.parametrize("length,mass", [(1e-14, 1.0), (1e13, 1.0), (1.0, 1e-15), (1.0, 1e14), (1e-16, 1e-20)])
def test_estimate_outside_the_fast_range(length, mass):
    """Squared distances below 2^-80 or above 2^80, masses below 2^-40 or above 2^40."""
    pos, _, _ = ics.plummer(900, 5, center=False)
    check(pos * length, ics.kroupa_masses(900, 6) * mass, 64)


@pytest.mark.parametrize("target", [2.0 - 2.0**-23, 1.0 + 2.0**-23, 2.0 - 2.0**-22, 1.0])
def test_estimate_at_extreme_significands(target):
    """Squared distances whose significand is all ones, just above one, or one, by masses of a power of two and
    others: where a reciprocal that is off by an ulp would show in the quotient. The pair's offsets in x and y
    are chosen so that the FP32 sum of their squares is the wanted number."""
    def squared(x, y):
        return np.float32(np.float32(x * x) + np.float32(y * y))

    t32, found = np.float32(target), None
    x = np.float32(np.sqrt(target))
    while found is None:  # x * x at or below the target, the rest by y
        rest = target - float(x) ** 2
        for y in np.float32(np.sqrt(max(rest, 0.0))) * np.linspace(0.9, 1.1, 201, dtype=np.float32):
            if squared(x, y) == t32:
                found = (x, y)
        x = np.nextafter(x, np.float32(0))
    dx, dy = (float(v) for v in found)
    for scale in (2.0**-30, 1.0, 2.0**20):
        pos = 0.5 * scale * np.array([[-dx, -dy, 0.0], [dx, dy, 0.0]])
        for mass in (1.0, 2.0**-20, 2.0**-17, 1.5, 2.0 - 2.0**-23, 1.0 + 2.0**-23, 1 / 3):
            check(pos, np.array([mass, mass]), 64)
