"""The one-block ranking of a list in shared memory, at the sizes where the
splitter spacing, the thread tiles and the walk change (oracle: exact)."""
import numpy as np
import pytest
import torch

import gen
import oracle
import paper_1002_4482_gb300 as lrcc

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _layouts(n):
    yield gen.list_random(n, n)
    yield gen.list_ordered(n)
    yield np.arange(-1, n - 1, dtype=np.int32), n - 1          # reversed
    # stride order: position k is element (k * 7) mod n, for n not a multiple of 7
    if n % 7:
        order = (np.arange(n, dtype=np.int64) * 7 % n).astype(np.int32)
        succ = np.full(n, -1, np.int32)
        succ[order[:-1]] = order[1:]
        yield succ, int(order[0])


@pytest.mark.parametrize("n", [1, 2, 31, 1023, 1024, 1025, 2047, 2048, 2049, 8191, 8193, 16383, 16384])
def test_one_block_lists(n):
    for succ, head in _layouts(n):
        t = torch.from_numpy(succ).to(DEV)
        assert np.array_equal(lrcc.lr_rank(t, head).cpu().numpy(), oracle.lr_rank(succ, head))
        val = (np.arange(n) % 5).astype(np.int32)
        got = lrcc.lr_scan(t, torch.from_numpy(val).to(DEV), head).cpu().numpy()
        assert np.array_equal(got, oracle.lr_scan(succ, val, head))
        # the same list in a batch (one block of 512 threads per list)
        off = torch.tensor([0, n, 2 * n], dtype=torch.int64, device=DEV)
        heads = torch.tensor([head, head], dtype=torch.int32, device=DEV)
        got = lrcc.lr_rank_batched(torch.cat([t, t]), off, heads).cpu().numpy()
        assert np.array_equal(got.reshape(2, n), np.tile(oracle.lr_rank(succ, head), (2, 1)))
    lrcc.check()


@pytest.mark.parametrize("n", [3, 1025, 16384])
def test_one_block_rejects_what_is_not_one_list(n):
    succ, head = gen.list_random(n, 5)
    order = np.empty(n, np.int64)
    order[n - 1 - oracle.lr_rank(succ, head)] = np.arange(n)
    cycle = succ.copy()
    cycle[order[-1]] = order[n // 2]          # the tail leads back into the list
    shared = succ.copy()
    shared[order[n // 2]] = -1                # two lists
    skipped = succ.copy()
    skipped[order[0]] = order[2]              # an element nobody names
    for bad in (cycle, shared, skipped):
        lrcc.lr_rank(torch.from_numpy(bad).to(DEV), head)
        assert lrcc.last_status() == lrcc.ERR_INVALID_INPUT
