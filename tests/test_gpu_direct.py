"""The segmented FP64 direct sum against the oracle's, around the sizes where
the sources are split."""
import numpy as np
import pytest

import ics
import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover - CPU container
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2012_02207_gb300 as gb  # noqa: E402


@pytest.mark.parametrize("soft", [0.0, 1e-3])
@pytest.mark.parametrize("n,ntgt", [(1, 1), (2, 2), (255, 255), (511, 7), (512, 129), (1025, 1025), (40000, 128),
                                    (40000, 1000)])
def test_direct_sum(n, ntgt, soft):
    pos, _, _ = ics.plummer(n, 60 + n, center=False)
    m = ics.kroupa_masses(n, 61)
    tg = np.sort(np.random.default_rng(n).choice(n, ntgt, replace=False))
    cols = [torch.tensor(np.ascontiguousarray(c), dtype=torch.float64, device="cuda") for c in (*pos.T, m)]
    f = gb.FMM(soft=soft)
    out = f.direct(*cols, targets=None if ntgt == n else torch.tensor(tg, device="cuda"))
    acc, pot = torch.stack(out[:3], 1).cpu().numpy(), out[3].cpu().numpy()
    oacc, opot = oracle.direct(pos, m, targets=tg, soft=soft)
    # both round to FP64 a sum of n terms of one sign: n 2^-53 of the sum of the terms' magnitudes at most
    scale = np.array([(m / np.maximum(((pos - pos[i]) ** 2).sum(1) + soft * soft, 1e-300))[np.arange(n) != i].sum()
                      for i in tg])
    assert np.all(np.linalg.norm(acc - oacc, axis=1) <= 2.0 ** -53 * (n + 16) * scale)
    assert np.all(np.abs(pot - opot) <= 2.0 ** -53 * (n + 16) * np.abs(opot))


def test_direct_out_of_seed_range():
    """Squared distances below 2^-999 and above 2^993 take the general division."""
    x = torch.tensor([0.0, 1e-155, 1.0, 1e152], dtype=torch.float64, device="cuda")
    z = torch.zeros_like(x)
    m = torch.tensor([1.0, 1e-30, 2.0, 3.0], dtype=torch.float64, device="cuda")
    out = gb.FMM().direct(x, z, z, m)
    ox, opot = oracle.direct(np.stack([x.cpu().numpy(), np.zeros(4), np.zeros(4)], 1), m.cpu().numpy())
    ok = np.isfinite(ox[:, 0])  # the first two bodies' accelerations overflow
    assert ok.sum() == 2
    assert np.allclose(out[0].cpu().numpy()[ok], ox[ok, 0], rtol=1e-14, atol=0.0)
    assert np.allclose(out[3].cpu().numpy(), opot, rtol=1e-14, atol=0.0)


@pytest.mark.parametrize("soft", [0.0, 1e-3])
@pytest.mark.parametrize("n,ntgt", [(9001, 9001), (33000, 0), (33000, -1)])
def test_direct_sum_of_many_targets(n, ntgt, soft):
    """Eight targets a warp from 32 per SM on, four below: the last warp of either incomplete, sources that do
    not fill a batch of 32. The same bits from both, and the oracle's sum at some of the targets."""
    few = 32 * torch.cuda.get_device_properties(0).multi_processor_count  # the first count with eight
    ntgt = ntgt if ntgt > 0 else few + ntgt
    assert n % 32 and (n < 32000) == (ntgt == n)
    pos, _, _ = ics.plummer(n, 62, center=False)
    m = ics.kroupa_masses(n, 63)
    rng = np.random.default_rng(n)
    tg = np.arange(n) if ntgt == n else rng.choice(n, ntgt, replace=False)
    cols = [torch.tensor(np.ascontiguousarray(c), dtype=torch.float64, device="cuda") for c in (*pos.T, m)]
    f = gb.FMM(soft=soft)
    out = torch.stack(f.direct(*cols, targets=torch.tensor(tg, device="cuda")))
    some = np.concatenate([np.arange(9), rng.integers(0, ntgt, 180), np.arange(ntgt - 9, ntgt)])  # four a warp
    part = torch.stack(f.direct(*cols, targets=torch.tensor(tg[some], device="cuda")))
    assert torch.equal(part, out[:, torch.tensor(some, device="cuda")])
    oacc, opot = oracle.direct(pos, m, targets=tg[some], soft=soft)
    got = part.cpu().numpy()
    # both round to FP64 a sum of n terms: n 2^-53 of the sum of the terms' magnitudes at most
    scale = np.array([(m / np.maximum(((pos - pos[i]) ** 2).sum(1) + soft * soft, 1e-300))[np.arange(n) != i].sum()
                      for i in tg[some]])
    assert np.all(np.linalg.norm(got[:3].T - oacc, axis=1) <= 2.0 ** -53 * (n + 16) * scale)
    assert np.all(np.abs(got[3] - opot) <= 2.0 ** -53 * (n + 16) * np.abs(opot))
