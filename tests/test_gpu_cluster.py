"""AUTO where the layout is computed by thread-block clusters: token counts at the edges of the slices, groups of
32 tokens and chunks (fewer tokens than CTAs, than ranks, than a cluster's slices; the cluster sizes' boundaries;
token stealing), rank counts, slots per token, column parts, source ranks whose tokens span many CTAs or
share one, few CTAs, an expert named twice.  Dispatch bit by bit against the oracle, combine within its tolerance."""
import numpy as np
import pytest

from paper_2607_06202_b200 import binding as B
from paper_2607_06202_b200 import workload as W
from tests import harness as Hn

pytestmark = pytest.mark.gpu

PHASED, LOCAL, CLUSTER, FEW = B.UBEP_PIPELINE_PHASED, B.UBEP_PIPELINE_LOCAL, 4, 5   # how a call is scheduled


def _run(cfg, empty=0.0, mode=CLUSTER, **kw):
    """mode: how the call has to be scheduled (None: in any way).  Returns the plan."""
    wl = W.make_workload(cfg)
    if empty:
        wl = W.with_empty_slots(wl, empty, seed=cfg.seed + 1)
    buf = Hn.run_case(wl, threads=8, **kw)[0]
    pl = B.ubep_debug_buffer_plan(buf.handle, cfg.T)
    assert mode is None or pl["mode"] == mode, pl
    return pl


@pytest.mark.parametrize("payload,dedup", [(0, 0), (1, 0), (0, 1), (1, 1)])
@pytest.mark.parametrize("T", [1, 31, 65, 300, 2049, 4096, 4097, 8192])
def test_token_counts(T, payload, dedup):
    # (L = 32 experts per rank keeps the one-row-per-rank cases off the rank-level fast path)
    _run(W.Config("t", T=T, H=256, E=128, R=4, k=8, payload=payload, dedup=dedup, seed=T, num_src_ranks=7), mode=FEW if T < 256 else CLUSTER)
    if T < 256:   # (seven slots: no small batch)
        _run(W.Config("t", T=T, H=256, E=128, R=4, k=7, payload=payload, dedup=dedup, seed=T, num_src_ranks=7))


@pytest.mark.parametrize("E,R,k", [(1, 1, 1), (31, 1, 3), (160, 5, 8), (161, 7, 5), (288, 72, 8), (289, 17, 8),
                                   (512, 128, 8), (512, 2, 12), (256, 64, 16), (513, 27, 8), (258, 129, 8)])
@pytest.mark.parametrize("dedup", [0, 1])
def test_bins(E, R, k, dedup):
    mode = FEW if k == 1 else LOCAL if dedup and 1 < E // R < 32 and R <= 32 else CLUSTER
    _run(W.Config("b", T=777, H=128, E=E, R=R, k=k, dedup=dedup, seed=E + R), empty=0.1, mode=mode)
    _run(W.Config("b", T=4097, H=128, E=E, R=R, k=k, dedup=dedup, payload=1, seed=E + R))


@pytest.mark.parametrize("S", [1, 2, 40, 900])
def test_source_ranks(S):
    for T, k in ((200, 3), (200, 4), (1500, 4)):
        _run(W.Config("s", T=T, H=128, E=64, R=8, k=k, seed=S + T, num_src_ranks=S), mode=FEW if T * k == 800 else CLUSTER)


@pytest.mark.parametrize("num_ctas", [1, 2, 3, 5, 34])
def test_few_ctas(num_ctas):
    _run(W.Config("c", T=400, H=128, E=64, R=8, k=4, seed=num_ctas), num_ctas=num_ctas)


@pytest.mark.parametrize("payload", [0, 1])
def test_replicas_and_wide_rows(payload):
    cfg = W.Config("r", T=1000, H=7168, E=72, R=8, k=8, payload=payload, seed=5, E_logical=64)
    _run(cfg, dest_order=np.arange(8)[::-1].copy())
    for T in (20, 40, 70):
        _run(W.Config("p", T=T, H=7168, E=256, R=8, k=8, payload=payload, seed=6), mode=FEW)
        pl = _run(W.Config("p", T=T, H=7168, E=256, R=8, k=7, payload=payload, seed=6))
        assert pl["parts"] == (4 if T == 20 and not payload else 2)
    for T in (300, 512):   # several tokens per CTA: bf16 rows in halves
        assert _run(W.Config("p", T=T, H=7168, E=256, R=8, k=8, payload=payload, seed=6))["parts"] == 2 - payload


@pytest.mark.parametrize("k", [4, 7, 8, 11])
@pytest.mark.parametrize("dedup", [0, 1])
def test_an_expert_named_twice(k, dedup):
    cfg = W.Config("d", T=1200, H=128, E=128, R=4, k=k, dedup=dedup, seed=k)
    wl = W.make_workload(cfg)
    clean = wl.topk_idx.copy()
    clean[::3, k - 1] = -1
    wl_clean = W.Workload(cfg, wl.x, clean, wl.topk_w)
    _, lay, cap, recv = Hn.oracle_reference(wl_clean)
    buf = Hn.make_buffer(cfg, cap)
    x, _, w, _, _ = Hn.device_inputs(wl)
    dup = wl.topk_idx.copy()
    dup[::3, k - 1] = dup[::3, 0]
    buf.dispatch(x, Hn.to_dev(dup), w)
    assert buf.status() == B.UBEP_ERR_BAD_INDEX
    Hn.check_dispatch(buf, wl_clean, lay, cap, recv)


@pytest.mark.parametrize("cfg,pipeline,mode", [
    (dict(T=22, H=64, E=9360, R=39, k=8), LOCAL, PHASED),
    (dict(T=20, H=64, E=13000, R=1, k=4), LOCAL, PHASED),
    (dict(T=229, H=30816, E=18, R=6, k=4, dedup=1), LOCAL, LOCAL),       # (in halves of rows)
    (dict(T=238, H=34816, E=231, R=33, k=4, payload=1, dedup=1), 0, FEW),
    (dict(T=238, H=34816, E=231, R=33, k=3, payload=1, dedup=1), 0, PHASED),
    (dict(T=260, H=38112, E=144, R=4, k=1), 0, PHASED),
])
def test_where_the_counts_or_whole_rows_do_not_fit(cfg, pipeline, mode):
    _run(W.Config("w", seed=cfg["T"], **cfg), pipeline=pipeline, mode=mode)


@pytest.mark.parametrize("cfg", [
    dict(T=4096, H=4096, E=128, R=16, k=8),   # 28 rows per CTA, ten teams of one warp
    dict(T=4097, H=4096, E=128, R=16, k=8, dedup=1),
    dict(T=8192, H=7168, E=64, R=8, k=4),     # 56 rows per CTA, seven teams
])
def test_short_fp8_rows_whose_ring_is_used_more_than_once(cfg):
    wl = W.make_workload(W.Config("ring", payload=1, seed=cfg["T"], **cfg))
    _, lay, cap, recv = Hn.oracle_reference(wl, num_threads=8)
    buf = Hn.make_buffer(wl.cfg, cap)
    x, idx, w, _, _ = Hn.device_inputs(wl)
    for _ in range(4):
        buf.recv_x.fill_(Hn.FILL)
        buf.dispatch(x, idx, w)
        Hn.check_dispatch(buf, wl, lay, cap, recv)


@pytest.mark.parametrize("H", [4992, 5120, 5248])
@pytest.mark.parametrize("T", [90, 300, 700])
def test_around_the_line_between_short_and_long_fp8_rows(H, T):
    for dedup in (0, 1):
        # (rows of less than 40 KB of copies with one row per (token, rank): every CTA alone)
        mode = FEW if T == 90 else LOCAL if dedup and H < 5120 else CLUSTER
        pl = _run(W.Config("l", T=T, H=H, E=64, R=8, k=8, payload=1, dedup=dedup, seed=H + T), mode=mode)
        assert pl["long_rows"] == (H >= 5120 and T > 90)


@pytest.mark.parametrize("H,payload", [(2048, 0), (5120, 1)])
@pytest.mark.parametrize("T", [4800, 4801, 5919, 6100])
def test_where_tails_of_the_slices_are_handed_out(T, H, payload):
    """Slices of 40 tokens and a few more, some of them one longer than others, on 120 CTAs: heads without claims, tails with."""
    for dedup in (0, 1):
        assert _run(W.Config("tail", T=T, H=H, E=32, R=4, k=8, payload=payload, dedup=dedup, seed=T), num_ctas=120)["steal"]
