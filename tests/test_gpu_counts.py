"""The counts entry point at the edges of its work split: 32 tokens per warp, four warps per CTA, at most 296
CTAs; rank masks of one word, of four words and the slot-by-slot variant beyond 128 ranks; slots per token with
a variant of their own (2, 4, 8) and without.  Integers: exact against the oracle."""
import numpy as np
import pytest
import torch

import oracle
from paper_2607_06202_b200 import binding as B
from paper_2607_06202_b200 import workload as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T", [1, 31, 33, 129, 40001])
@pytest.mark.parametrize("E,R,k", [(4, 1, 3), (15, 5, 2), (64, 32, 4), (128, 16, 8), (66, 33, 4), (288, 72, 8),
                                   (256, 128, 16), (390, 130, 8), (200, 200, 2)])
def test_counts_match_the_oracle(T, E, R, k):
    rng = np.random.Generator(np.random.PCG64(T * 1000 + E))
    idx = np.argsort(rng.random((T, E)), axis=1)[:, :k].astype(np.int32)
    idx[rng.random(idx.shape) < 0.1] = -1
    lay = oracle.layout(idx, E, R, R, 0)
    dup = idx.copy()      # the last slot repeats the first one: reported, counted as if it were empty
    if k > 2:
        dup[:, -1] = dup[:, 0]
    clean = dup.copy()
    if k > 2:
        clean[:, -1] = -1
    lay_dup = oracle.layout(clean, E, R, R, 0)
    buf = B.Buffer(num_ranks=R, num_experts=E, hidden=8, topk=k, max_tokens=T, rows_per_rank_cap=1)
    for table, want, code in ((idx, lay, 0), (dup, lay_dup, B.UBEP_ERR_BAD_INDEX if (k > 2 and (dup[:, 0] >= 0).any()) else 0),
                              (idx, lay, 0)):
        npr, npe, itr = buf.get_dispatch_layout(torch.from_numpy(table).cuda())
        assert buf.status() == code
        assert np.array_equal(npr.cpu().numpy(), want.num_tokens_per_rank)
        assert np.array_equal(npe.cpu().numpy(), want.num_tokens_per_expert)
        assert np.array_equal(itr.cpu().numpy(), want.is_token_in_rank)
    # through the C entry point with some of the outputs left out
    only = torch.full((E,), -1, dtype=torch.int32, device="cuda")
    B.ubep_get_dispatch_layout(buf.handle, torch.from_numpy(idx).cuda(), T, None, only, None)
    assert np.array_equal(only.cpu().numpy(), lay.num_tokens_per_expert)


@pytest.mark.parametrize("static", [False, True])
def test_overlapping_calls_do_not_spoil_later_ones(static):
    """Calls on two streams share the totals and the ticket: their counts are undefined, those of a later call are not."""
    E, R, k, most = 64, 8, 4, 9000
    rng = np.random.Generator(np.random.PCG64(3))
    tables = [np.argsort(rng.random((T, E)), axis=1)[:, :k].astype(np.int32) for T in (most, 130, 2500, 31)]
    dev = [torch.from_numpy(t).cuda() for t in tables]
    buf = B.Buffer(num_ranks=R, num_experts=E, hidden=8, topk=k, max_tokens=most, rows_per_rank_cap=1)
    outs = [(torch.empty(R, dtype=torch.int32, device="cuda"), torch.empty(E, dtype=torch.int32, device="cuda")) for _ in range(2)]

    def call(table, out, stream=None):
        if static:
            B.ubep_get_dispatch_layout_static(table, table.shape[0], k, E, R, *out, None, stream)
        else:
            B.ubep_get_dispatch_layout(buf.handle, table, table.shape[0], *out, None, stream)

    call(dev[0], outs[0])   # (the static one's first call looks up its array)
    streams = [torch.cuda.Stream() for _ in range(2)]
    torch.cuda.synchronize()
    for rounds in range(40):
        for i in range(6):
            call(dev[(rounds + i) % 4], outs[i % 2], streams[i % 2])
        torch.cuda.synchronize()
        n = rounds % 4
        call(dev[n], outs[0])
        lay = oracle.layout(tables[n], E, R, R, 0)
        assert np.array_equal(outs[0][0].cpu().numpy(), lay.num_tokens_per_rank)
        assert np.array_equal(outs[0][1].cpu().numpy(), lay.num_tokens_per_expert)


def test_the_results_are_tensors_of_their_own():
    """Each has its own storage: keeping or saving the small ones does not keep or save the mask."""
    buf = B.Buffer(num_ranks=4, num_experts=16, hidden=8, topk=2, max_tokens=500, rows_per_rank_cap=1)
    idx = torch.zeros((500, 2), dtype=torch.int32, device="cuda")
    idx[:, 1] = 5
    out = buf.get_dispatch_layout(idx)
    assert [t.untyped_storage().nbytes() for t in out] == [4 * 4, 4 * 16, 500 * 4]
    assert [t.storage_offset() for t in out] == [0, 0, 0]
    assert len({t.untyped_storage().data_ptr() for t in out}) == 3


@pytest.mark.parametrize("T", [512, 513, 1025, 4096, 4097])
@pytest.mark.parametrize("E,R,k", [(72, 9, 6), (128, 128, 8), (129, 129, 1), (8, 2, 4), (12, 3, 2)])
def test_one_cluster_and_beyond(T, E, R, k):
    """One CTA, clusters of two to eight, and totals in global memory; masks that start on no 16-byte boundary."""
    rng = np.random.Generator(np.random.PCG64(T + E))
    idx = np.argsort(rng.random((T, E)), axis=1)[:, :k].astype(np.int32)
    idx[rng.random(idx.shape) < 0.2] = -1
    lay = oracle.layout(idx, E, R, R, 0)
    buf = B.Buffer(num_ranks=R, num_experts=E, hidden=8, topk=k, max_tokens=T, rows_per_rank_cap=1)
    npr, npe = (torch.full((n,), -1, dtype=torch.int32, device="cuda") for n in (R, E))
    for off in (0, 4, 1):
        raw = torch.full((T * R + 32,), 7, dtype=torch.uint8, device="cuda")
        B.ubep_get_dispatch_layout(buf.handle, torch.from_numpy(idx).cuda(), T, npr, npe, raw[off:off + T * R])
        assert buf.status() == 0
        assert np.array_equal(npr.cpu().numpy(), lay.num_tokens_per_rank)
        assert np.array_equal(npe.cpu().numpy(), lay.num_tokens_per_expert)
        got = raw.cpu().numpy()
        assert np.array_equal(got[off:off + T * R].reshape(T, R), lay.is_token_in_rank)
        assert (got[:off] == 7).all() and (got[off + T * R:] == 7).all()
