"""The radix sort's bounded waits (its look-back, sorts of more than 4096 keys):
a test hook makes them wait for records that no tile writes."""
import numpy as np
import pytest

import ics

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover - CPU container
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2012_02207_gb300 as gb  # noqa: E402

FMM_ERR_TIMEOUT = -7


def bodies(n, seed):
    pos, _, m = ics.plummer(n, seed)
    return [torch.tensor(np.ascontiguousarray(c), device="cuda") for c in (*pos.T, m)]


@pytest.mark.parametrize("hook,what", [(8, "body sort"), (16, "list sort")])
def test_sort_wait_that_runs_out_reports_a_timeout(hook, what):
    """The first wait runs out after a second and the later ones soon after it; the call returns
    FMM_ERR_TIMEOUT and the device stays usable. A failed list sort ends the solve at the second walk's
    first check: with no estimate its MAC refuses every pair, and going on it would list all pairs of
    some 6,000 leaves in ever larger buffers."""
    cols = bodies(20000, 45)
    f = gb.FMM(p=8, eps=1e-7, leaf_size=8, fault_inject=hook)
    with pytest.raises(gb.FmmError) as e:
        f.solve(*cols)
    assert e.value.status == FMM_ERR_TIMEOUT and what in str(e.value)
    s = f.stats()
    assert s["regrows"] == 0 and s["n_p2p"] == 0
    one = gb.FMM(p=8, eps=1e-7, leaf_size=8)
    a = torch.stack(one.solve(*cols))
    assert one.stats()["n_p2p"] > 0
    assert torch.equal(a, torch.stack(gb.FMM(p=8, eps=1e-7, leaf_size=8).solve(*cols)))


def test_stalled_hooks_do_not_touch_sorts_of_one_tile():
    """Up to 4096 keys are sorted in one launch without waits."""
    cols = bodies(4096, 46)
    f = gb.FMM(p=8, eps=1e-7, leaf_size=64, fault_inject=8)
    assert torch.equal(torch.stack(f.solve(*cols)), torch.stack(gb.FMM(p=8, eps=1e-7, leaf_size=64).solve(*cols)))
