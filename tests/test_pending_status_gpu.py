"""A status word that an earlier call left and nobody has read changes nothing
in the calls after it: sampled and plain component labels under every hook rule,
with and without graphs, single and batched, and ranks. Exact."""
import numpy as np
import pytest
import torch

import gen
import oracle
import paper_1002_4482_gb300 as lrcc

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to(DEV)


def _leave_a_timeout():
    lrcc.wait_check(64)
    return lrcc.ERR_TIMEOUT


def _leave_an_invalid_input():
    lrcc.lr_rank(_dev(np.full(1000, 1000, np.int32)), 0)
    return lrcc.ERR_INVALID_INPUT


@pytest.fixture(params=[_leave_a_timeout, _leave_an_invalid_input])
def pending(request):
    lrcc.last_status()
    yield request.param
    lrcc.last_status()
    lrcc.reset_plans()


@pytest.mark.parametrize("hook", [1, 2, 3, 4, 5])
@pytest.mark.parametrize("use_graphs", [1, 2])
def test_components_after_an_unread_error(pending, hook, use_graphs):
    n, m = 1 << 17, 1 << 19   # from 2^19 edges and 2 per vertex on rule 1 samples and filters
    src, dst = gen.er(n, m, 3)
    lrcc.set_cc_plan(0, 32, cc_hook=hook, use_graphs=use_graphs)
    code = pending()
    got = lrcc.cc_label(_dev(src), _dev(dst), n)
    assert lrcc.last_status() == code
    assert np.array_equal(got.cpu().numpy(), oracle.cc_uf(src, dst, n))


@pytest.mark.parametrize("hook", [1, 2])
@pytest.mark.parametrize("use_graphs", [1, 2])
def test_batched_components_after_an_unread_error(pending, hook, use_graphs):
    sizes = [100_000, 300, 70_000]
    parts = [gen.er(n, 3 * n, n) for n in sizes]
    voff = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    src, dst = np.concatenate([p[0] for p in parts]), np.concatenate([p[1] for p in parts])
    lrcc.set_plan(lrcc.KIND_CC_BATCH, 0, 32, cc_hook=hook, use_graphs=use_graphs)
    code = pending()
    got = lrcc.cc_label_batched(_dev(src), _dev(dst), _dev(3 * voff), _dev(voff), n_total=int(voff[-1])).cpu().numpy()
    assert lrcc.last_status() == code
    for k, n in enumerate(sizes):
        assert np.array_equal(got[voff[k]:voff[k + 1]], oracle.cc_uf(*parts[k], n))


def test_ranks_after_an_unread_error(pending):
    for n in (5000, 200_000):
        succ, head = gen.list_random(n, n)
        val = np.ones(n, np.int32)
        code = pending()
        rank, total = lrcc.lr_rank(_dev(succ), head), lrcc.lr_scan(_dev(succ), _dev(val), head)
        forest = lrcc.lr_scan_forest(_dev(succ), _dev(val))
        assert lrcc.last_status() == code
        want = oracle.lr_rank(succ, head)
        assert np.array_equal(rank.cpu().numpy(), want)
        assert np.array_equal(total.cpu().numpy(), want + 1)
        assert np.array_equal(forest.cpu().numpy(), want + 1)
