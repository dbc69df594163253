"""FP32 M2L: every order, by degrees or in straight-line steps, against FP64.

The interaction lists do not depend on the precision, so a mixed-precision
solve differs from an FP64 one of the same order only by FP32 rounding in the
M2L and P2P: the bounds are those the mixed-precision error has over the FP64
one elsewhere in the tests (5e-7 rms to order 10, 1e-6 above). A target cell's
sources go to the lanes 32 at a time and the next batch is loaded early: the
trees here have targets with less than one batch, one and several, and the
lattice has pairs of cells along z (no azimuth).
"""
import numpy as np
import pytest

import ics

pytestmark = pytest.mark.gpu


def bodies(kind):
    if kind == "lattice":
        g = np.stack(np.meshgrid(*[np.arange(12.0)] * 3, indexing="ij"), -1).reshape(-1, 3)
        return g, np.full(len(g), 1.0 / len(g))
    n = int(kind)
    return ics.plummer(n, 11)[0], ics.kroupa_masses(n, 12)


@pytest.mark.parametrize("kind", ["97", "700", "5000", "lattice"])
@pytest.mark.parametrize("p", [4, 6, 8, 10, 12, 14])
def test_fp32_m2l_against_fp64(kind, p):
    import torch

    import paper_2012_02207_gb300 as gb

    pos, m = bodies(kind)
    cols = [torch.tensor(np.ascontiguousarray(pos[:, d]), device="cuda") for d in range(3)]
    cols.append(torch.tensor(m, device="cuda"))
    acc = {}
    for precision in ("mixed", "fp64"):
        f = gb.FMM(p=p, eps=1e-5 if p < 8 else 1e-6, leaf_size=4, precision=precision)
        acc[precision] = torch.stack(f.solve(*cols)[:3]).cpu().numpy()
        if precision == "mixed":
            pairs = f.export_pairs("m2l")
            fill = np.unique(pairs[:, 1], return_counts=True)[1]
            if kind == "5000":
                assert fill.min() < 32 < fill.max()
    size = np.linalg.norm(acc["fp64"], axis=0)
    err = np.linalg.norm(acc["mixed"] - acc["fp64"], axis=0) / np.maximum(size, np.median(size))
    assert np.sqrt(np.mean(err**2)) <= (5e-7 if p <= 10 else 1e-6)
