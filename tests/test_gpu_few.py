"""Small batches (a warp per slot of the CTA's own tokens): the edges of what is taken that way, against the oracle."""
import numpy as np
import pytest

from paper_2607_06202_b200 import binding as B
from paper_2607_06202_b200 import workload as W
from tests import harness as Hn

FEW = 5
SHAPES = [(7168, 256, 32, 8), (4096, 128, 16, 8), (2048, 128, 8, 4), (256, 16, 4, 2)]


def mode(T, H, E, R, k, payload=0, dedup=0, **kw):
    cfg = B.ubep_config_t(R, E, H, k, T, 128, 0, payload, dedup, 0, kw.get("pipeline", 0), kw.get("num_ctas", 0))
    return B.ubep_debug_plan(cfg, T, 232448, (148, 148, 132, 120), **{n: v for n, v in kw.items() if n == "quant_warps"})


def test_which_calls_are_small_batches():
    for (H, E, R, k), last in zip(SHAPES, (256, 256, 444, 655)):
        for payload, dedup in ((0, 0), (1, 0), (0, 1), (1, 1)):
            small = [T for T in range(1, 800) if mode(T, H, E, R, k, payload, dedup)["mode"] == FEW]
            assert set(range(1, 149)) <= set(small) and max(small) == last, (H, k, payload, dedup, max(small))
            for T in (1, 148, max(small)):
                pl = mode(T, H, E, R, k, payload, dedup)
                assert -(-T // pl["chunks"]) * k <= 16 and pl["stages"] >= -(-T // pl["chunks"])
                assert 118 * 1024 < pl["smem"] <= 232448   # (one CTA per SM)
    assert mode(100, 256, 64, 1, 8)["mode"] != FEW                              # 64 experts on one rank
    assert mode(100, 256, 64, 8, 5)["mode"] != FEW                              # slots that are no vector
    assert mode(100, 256, 64, 8, 8, num_ctas=40)["mode"] != FEW                 # more slots than warps
    assert mode(100, 256, 64, 8, 8, payload=1, quant_warps=3)["mode"] != FEW
    assert mode(8, 16384, 64, 8, 1, num_ctas=1)["mode"] != FEW                  # the rows do not fit
    for pipeline in (1, 2, 3):
        assert mode(16, 256, 64, 8, 8, pipeline=pipeline)["mode"] != FEW


def _run(T, H, E, R, k, payload, dedup, empty=0.0, **kw):
    cfg = W.Config("few", T=T, H=H, E=E, R=R, k=k, payload=payload, dedup=dedup, seed=T + H + k, **kw)
    wl = W.make_workload(cfg)
    if empty:
        wl = W.with_empty_slots(wl, empty, seed=T)
    Hn.run_case(wl, threads=8)


@pytest.mark.gpu
@pytest.mark.parametrize("payload,dedup", [(0, 0), (1, 0), (0, 1), (1, 1)])
@pytest.mark.parametrize("H,E,R,k,tokens", [
    (7168, 256, 32, 8, (1, 2, 19, 37, 75, 148, 149, 256)),   # eight, four, two column parts, whole rows, two tokens per CTA
    (128, 32, 1, 8, (1, 31, 32, 33, 160, 256, 257)),              # every expert on one rank: all bits of a word
    (640, 96, 96, 6, (5, 148, 296)),                         # one expert per rank; scales that no bulk copy can carry
    (1024, 32, 8, 4, (3, 149, 444, 445)),
    (256, 16, 4, 2, (64, 148, 297, 655, 656)),
    (384, 24, 8, 1, (1, 33, 700)),
])
def test_sizes(H, E, R, k, tokens, payload, dedup):
    for T in tokens:
        _run(T, H, E, R, k, payload, dedup, empty=0.15 if T % 2 else 0.0)


@pytest.mark.gpu
@pytest.mark.parametrize("T", [1, 40, 200])
def test_source_ranks_replicas_and_narrow_rows(T):
    for S in (1, 7, 40, 900):
        _run(T, 8, 60, 20, 4, 0, T % 2, num_src_ranks=S)
    for payload in (0, 1):
        _run(T, 256, 288, 72, 8, payload, 1, E_logical=256)
        _run(T, 256, 288, 72, 8, payload, 0, E_logical=256)


@pytest.mark.gpu
@pytest.mark.parametrize("dedup", [0, 1])
def test_bad_ids_experts_named_twice_and_capacity(dedup):
    cfg = W.Config("few", T=90, H=128, E=32, R=4, k=8, dedup=dedup, seed=3)
    wl = W.make_workload(cfg)
    given, clean = wl.topk_idx.copy(), wl.topk_idx.copy()
    clean[::3, 7] = -1
    given[::3, 7] = given[::3, 0]
    clean[1, 2] = clean[4, 0] = -1
    given[1, 2], given[4, 0] = 32, -2
    want = W.Workload(cfg, wl.x, clean, wl.topk_w)
    _, lay, cap, recv = Hn.oracle_reference(want)
    buf = Hn.make_buffer(cfg, cap)
    x, _, w, _, _ = Hn.device_inputs(wl)
    buf.dispatch(x, Hn.to_dev(given), w)
    assert buf.status() == B.UBEP_ERR_BAD_INDEX
    Hn.check_dispatch(buf, want, lay, cap, recv)
    small = int(lay.num_rows_per_rank.max()) - 2
    buf = Hn.make_buffer(cfg, small)
    buf.dispatch(x, Hn.to_dev(clean), w)
    assert buf.status() == B.UBEP_ERR_CAPACITY
    assert np.array_equal(buf.cnt.cpu().numpy(), lay.cnt) and np.array_equal(buf.slot_row[:cfg.T].cpu().numpy(), lay.slot_row)
    for r in range(cfg.R):
        n = min(int(lay.num_rows_per_rank[r]), small)
        assert np.array_equal(buf.recv_src_idx[r, :n].cpu().numpy(), recv.recv_src_idx[r, :n])
        assert np.array_equal(buf.recv_x[r, :n].cpu().numpy(), recv.recv_x[r, :n])


@pytest.mark.gpu
def test_between_calls_of_other_sizes():
    """The arrival counters and the count of tokens handed out of a call are cleared by the call before it."""
    cfgs = [W.Config("mix", T=T, H=2048, E=64, R=8, k=8, seed=T) for T in (13, 6000, 200)]
    refs = [Hn.oracle_reference(W.make_workload(c), cap=8192, num_threads=8) for c in cfgs]
    buf = Hn.make_buffer(cfgs[1], 8192)
    wls = [W.make_workload(c) for c in cfgs]
    dev = [Hn.device_inputs(wl) for wl in wls]
    for i in (0, 1, 2, 1, 1, 0, 0, 1):
        buf.recv_x.fill_(Hn.FILL)
        buf.dispatch(*dev[i][:3])
        Hn.check_dispatch(buf, wls[i], refs[i][1], 8192, refs[i][3], check_tails=False)


@pytest.mark.gpu
def test_rows_are_fetched_behind_the_layout_where_that_is_asked_for():
    """The kernel asks for all rows of a CTA at once, so a call that may not do so goes another way."""
    cfg = W.Config("few", T=200, H=512, E=32, R=4, k=8, payload=1, dedup=1, seed=11)
    wl = W.make_workload(cfg)
    _, lay, cap, recv = Hn.oracle_reference(wl)
    buf = Hn.make_buffer(cfg, cap)
    x, idx, w, _, _ = Hn.device_inputs(wl)
    for n, few in ((1 << 30, True), (2, True), (1, False)):   # (two tokens per CTA)
        B.ubep_debug_set_prefetch_rows(buf.handle, n)
        assert (B.ubep_debug_buffer_plan(buf.handle, cfg.T)["mode"] == FEW) == few
        buf.recv_x.fill_(Hn.FILL)
        buf.dispatch(x, idx, w)
        Hn.check_dispatch(buf, wl, lay, cap, recv)


@pytest.mark.gpu
@pytest.mark.parametrize("payload,dedup", [(0, 0), (1, 1)])
@pytest.mark.parametrize("T", [3, 19, 60, 148, 200])
def test_every_cta_stamps_its_phases(T, payload, dedup):
    """Rows that the first warp does not send, CTAs without tokens, several column parts and several tokens per CTA."""
    cfg = W.Config("few", T=T, H=1024, E=64, R=4, k=8, payload=payload, dedup=dedup, seed=T)
    wl = W.with_empty_slots(W.make_workload(cfg), 0.4, seed=T)
    wl.topk_idx[::2, 0] = -1
    _, lay, cap, recv = Hn.oracle_reference(wl)
    buf = Hn.make_buffer(cfg, cap)
    x, idx, w, _, _ = Hn.device_inputs(wl)
    B.ubep_debug_trace(buf.handle, True)
    pl = B.ubep_debug_buffer_plan(buf.handle, T)
    ctas = pl["chunks"] * pl["parts"]
    assert pl["mode"] == FEW
    buf.trace.zero_()
    for _ in range(2):
        before = buf.trace[:ctas, 10].cpu().numpy().copy()
        buf.dispatch(x, idx, w)
        Hn.check_dispatch(buf, wl, lay, cap, recv)
        tr = buf.trace.cpu().numpy()[:ctas]
        assert (tr[:, 0] > before).all()
        # start, table staged, rows assigned, copies may leave, last copy issued, (counts written,) copies complete, end
        for a, b in ((0, 1), (1, 5), (5, 6), (6, 8), (8, 9), (8, 3), (9, 10), (3, 10)):
            assert (tr[:, a] <= tr[:, b]).all(), (a, b)
        own = [c for c in range(ctas) if (c // pl["parts"]) * T // pl["chunks"] < (c // pl["parts"] + 1) * T // pl["chunks"]]
        assert (tr[own, 6] <= tr[own, 7]).all() and (tr[own, 7] <= tr[own, 8]).all()
        assert (tr[:, 10] - tr[:, 0]).max() < 5e6


@pytest.mark.gpu
@pytest.mark.parametrize("T,k", [(16, 2), (200, 8)])
def test_fp8_special_values(T, k):
    """Zeros, groups below the floor of their maximum, infinities, values beyond the format and NaNs."""
    cfg = W.Config("few", T=T, H=512, E=8 * k, R=4, k=k, payload=1, dedup=1, seed=12)
    wl = W.make_workload(cfg)
    xf = W.bf16_bits_to_f32(wl.x)
    xf[0, :128] = 0.0
    xf[1, 128:256] = 3e-6
    xf[2, :] *= 1e30
    xf[4, :128] = np.linspace(-1, 1, 128)
    xf[5, 7], xf[6, 200] = np.inf, -np.inf
    wl.x = W.f32_to_bf16_bits(xf)
    wl.x[3, 5], wl.x[3, 6] = 0x7FC0, 0xFFC0
    buf = Hn.run_case(wl)[0]
    assert B.ubep_debug_buffer_plan(buf.handle, T)["mode"] == FEW


@pytest.mark.gpu
@pytest.mark.parametrize("E,R", [(65504, 2047), (65535, 65535), (11200, 5600)])
@pytest.mark.parametrize("dedup", [0, 1])
def test_tables_of_many_experts(E, R, dedup):
    """Ids up to the largest that 16 bits hold beside the mark of an empty slot."""
    cfg = W.Config("few", T=40, H=128, E=E, R=R, k=8, payload=dedup, dedup=dedup, seed=31, num_src_ranks=3)
    wl = W.with_empty_slots(W.make_workload(cfg), 0.1, seed=5)
    wl.topk_idx[7, :3] = (E - 1, E - 2, 0)
    _, lay, cap, recv = Hn.oracle_reference(wl, cap=8)
    buf = Hn.make_buffer(cfg, cap)
    assert B.ubep_debug_buffer_plan(buf.handle, cfg.T)["mode"] == FEW
    x, idx, w, _, _ = Hn.device_inputs(wl)
    for _ in range(2):
        buf.recv_x.fill_(Hn.FILL)
        buf.dispatch(x, idx, w)
        Hn.check_dispatch(buf, wl, lay, cap, recv)
