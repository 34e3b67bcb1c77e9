"""Batches of 2^25 elements and more, whose form the device chooses by the sizes:
mostly in lists that L2 does not hold, or not. Exact."""
import numpy as np
import pytest
import torch

import gen
import oracle
import paper_1002_4482_gb300 as lrcc

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
M = 1 << 20
MIXES = {"just_large": [2 * M] * 16, "one_long": [32 * M] + [100] * 31, "most_long": [0, 17 * M] + [M] * 15 + [1, 0],
         "half_long": [17 * M] + [M] * 17, "just_not_long": [16 * M] + [2 * M] * 8, "short": [1500] * 22_400}


@pytest.mark.parametrize("mix", MIXES)
@pytest.mark.parametrize("shift", [0, 1])
def test_size_mixes(mix, shift):
    succ, off, heads = gen.list_batch(np.asarray(MIXES[mix], np.int64), 5)
    want = oracle.lr_rank_batched(succ, off, heads)
    stream = torch.cuda.Stream()
    with lrcc.Context(0) as ctx, torch.cuda.stream(stream):
        ctx.reserve(stream, lrcc.workspace_query(lrcc.KIND_LR_BATCH, len(succ), len(heads)))
        held = ctx.bytes()
        buf = torch.zeros(len(succ) + shift, dtype=torch.int32, device=DEV)[shift:]
        buf.copy_(torch.from_numpy(succ))
        args = [torch.from_numpy(a).to(DEV) for a in (off, heads)]
        out = torch.empty(len(succ) + shift, dtype=torch.int32, device=DEV)[shift:]
        for _ in range(2):                     # the second call finds the words of the first
            out.fill_(-7)
            lrcc.lr_rank_batched(buf, *args, out=out, stream=stream)
            assert ctx.last_status(stream) == lrcc.OK and ctx.bytes() == held
            assert np.array_equal(out.cpu().numpy(), want)
        # the forms in turn on one workspace, and one of the lists a cycle
        tail = int(np.flatnonzero(succ == -1)[0])
        k = int(np.searchsorted(off, tail, side="right")) - 1
        buf[tail] = int(heads[k])
        if off[k + 1] - off[k] > 1:
            lrcc.lr_rank_batched(buf, *args, out=out, stream=stream)
            assert ctx.last_status(stream) == lrcc.ERR_INVALID_INPUT
        buf[tail] = -1
        lrcc.lr_rank_batched(buf, *args, out=out, stream=stream)
        assert ctx.last_status(stream) == lrcc.OK
        assert np.array_equal(out.cpu().numpy(), want)


def test_without_room_for_both_forms():
    succ, off, heads = gen.list_batch(np.asarray(MIXES["one_long"], np.int64), 6)
    args = [torch.from_numpy(a).to(DEV) for a in (succ, off, heads)]
    stream = torch.cuda.Stream()
    torch.cuda.synchronize()
    lrcc.last_status(stream)                      # the stream's status word is allocated
    lrcc.debug_fail_allocs(1)
    try:
        rank = lrcc.lr_rank_batched(*args, stream=stream)
        lrcc.check(stream)
    finally:
        lrcc.debug_fail_allocs(0)
    assert np.array_equal(rank.cpu().numpy(), oracle.lr_rank_batched(succ, off, heads))
    lrcc.release(stream)
