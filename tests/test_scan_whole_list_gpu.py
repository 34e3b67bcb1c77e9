"""lr_scan refuses an input that is not one list whichever element is missing
from it: single elements taken out (first-level splitters and others), pieces
between two splitters skipped, on both sides of the limits of its forms."""
import numpy as np
import pytest
import torch

import gen
import oracle
import paper_1002_4482_gb300 as lrcc
from tests.test_direct_level0_gpu import SEED, _splitters

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
NEAR = 1 << 22   # up to here the records are kept apart from the walk words


@pytest.fixture(autouse=True)
def seed():
    lrcc.set_plan(lrcc.KIND_LR, 0, 32, seed=SEED, rs_spacing0=8, rs_spacing=4)
    yield
    lrcc.reset_plans()


def _refused(succ, val, head, out):
    lrcc.lr_scan(succ, val, head, out=out)
    return lrcc.last_status() == lrcc.ERR_INVALID_INPUT


@pytest.mark.parametrize("n", [20_000, 140_000, 300_000, 1 << 20, NEAR, NEAR + 1, 5_000_000])
def test_missing_elements(n):
    host, head, perm = gen.list_random(n, n, with_perm=True)   # perm: the ids in list order
    pos = np.empty(n, np.int64)
    pos[perm] = np.arange(n)
    spl = _splitters(n, 8 if n <= NEAR else 16, head)   # first-level splitters
    rng = np.random.default_rng(n)
    succ, val = torch.from_numpy(host).to(DEV), torch.ones(n, dtype=torch.int32, device=DEV)
    out = torch.empty_like(succ)
    for x in np.concatenate([rng.choice(spl, 60), rng.choice(n, 40)]):
        p = int(pos[x])
        if p in (0, n - 1):
            continue
        before, after = int(perm[p - 1]), int(perm[p + 1])
        succ[before], succ[int(x)] = after, -1                  # x is a list of its own
        assert _refused(succ, val, head, out), int(x)
        succ[before], succ[int(x)] = int(x), after
    order = np.sort(pos[spl])
    for k in rng.choice(len(order) - 3, 40):
        a, b = (int(order[k + 1]), int(order[k + 2]))           # the piece from one splitter to the next
        if a == 0:
            continue
        before = int(perm[a - 1])
        succ[before] = int(perm[b])                             # skipped, with its end still linked
        assert _refused(succ, val, head, out), (a, b)
        succ[before] = int(perm[a])
    lrcc.lr_scan(succ, val, head, out=out)
    lrcc.check()
    assert np.array_equal(out.cpu().numpy()[perm], np.arange(n, 0, -1, dtype=np.int32))


@pytest.mark.parametrize("n", [NEAR - 1, NEAR, NEAR + 1])
@pytest.mark.parametrize("shift", [0, 1])
def test_values_around_the_limit_of_the_forms(n, shift):
    host, head = gen.list_random(n, n)
    val = (np.arange(n) % 13).astype(np.int32)
    bufs = [torch.empty(n + shift, dtype=torch.int32, device=DEV)[shift:] for _ in range(3)]
    bufs[0].copy_(torch.from_numpy(host))
    bufs[1].copy_(torch.from_numpy(val))
    lrcc.lr_scan(bufs[0], bufs[1], head, out=bufs[2])
    lrcc.check()
    assert np.array_equal(bufs[2].cpu().numpy(), oracle.lr_scan(host, val, head))
    lrcc.lr_scan_forest(bufs[0], bufs[1], out=bufs[2])
    lrcc.check()
    assert np.array_equal(bufs[2].cpu().numpy(), oracle.lr_scan(host, val, head))
