"""The radix sort at the edges of its tiles, with one and many tiles, ties and
constant digits: keys and permutation of the tree against numpy."""
import numpy as np
import pytest

import ics

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover - CPU container
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2012_02207_gb300 as gb  # noqa: E402


def keys_of(pos):
    """21-bit-per-axis Morton keys in the cube of the library's reading (x highest in each digit)."""
    lo, hi = pos.min(0), pos.max(0)
    c, h = 0.5 * (lo + hi), float((0.5 * (hi - lo)).max()) or 1.0
    q = np.clip(np.floor((pos - (c - h)) / (2.0 * h) * 2097152.0), 0, 2097151).astype(np.uint64)
    key = np.zeros(len(pos), np.uint64)
    for b in range(21):
        for d in range(3):
            key |= ((q[:, d] >> np.uint64(b)) & np.uint64(1)) << np.uint64(3 * b + 2 - d)
    return key


@pytest.mark.parametrize("n", [1, 2, 31, 4095, 4096, 4097, 8192, 12289, 300001])
@pytest.mark.parametrize("kind", ["plummer", "packed", "line"])
def test_body_sort(n, kind):
    pos, _, m = ics.plummer(n, 7 + n, center=False)
    if kind == "packed" and n > 2:  # nearly all bodies in a few cells of the finest level: ties, constant high digits
        pos[1:-1] = 1e-6 * pos[1:-1]
    elif kind == "line":
        pos[:, 1:] = 0.0
    cols = [torch.tensor(np.ascontiguousarray(c), dtype=torch.float64, device="cuda") for c in (*pos.T, m)]
    f = gb.FMM(p=4, eps=1e-2, leaf_size=128)
    f.solve(*cols)
    t = f.export_tree()
    key = keys_of(pos)
    order = np.argsort(key, kind="stable")
    assert np.array_equal(t["perm"], order)
    assert np.array_equal(t["keys"], key[order])
