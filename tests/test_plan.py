"""The plans of the dispatch kernel, worked out on the host (no GPU): what its roles rely on."""
import itertools

import pytest

from paper_2607_06202_b200 import binding as B

SMEM = 232448                 # shared memory a CTA of a B200 may use
CTAS = (148, 148, 132, 120)   # CTAs that can run at once on a B200, alone and in clusters of 2, 4, 8
AUTO, PHASED, FUSED, LOCAL = (B.UBEP_PIPELINE_AUTO, B.UBEP_PIPELINE_PHASED, B.UBEP_PIPELINE_FUSED, B.UBEP_PIPELINE_LOCAL)


def plan(T, H, E, R, k, payload=0, dedup=0, pipeline=AUTO, num_ctas=0, smem=SMEM, **warps):
    """None where the call would be refused."""
    cfg = B.ubep_config_t(R, E, H, k, T, 128, 0, payload, dedup, 0, pipeline, num_ctas)
    try:
        return B.ubep_debug_plan(cfg, T, smem, CTAS, **warps)
    except B.UbepError as e:
        assert e.code == B.UBEP_ERR_ARG
        return None


@pytest.mark.parametrize("k", [1, 2, 3, 4, 6, 8, 11, 16, 32])
def test_a_stage_of_short_fp8_rows_belongs_to_one_team(k):
    """A team waits for row n by the parity of its stage's barrier, which tells neighbouring phases apart and no others.
    Loads land in any order, so the row that had the stage before must have been this team's own: the number of
    stages is a multiple of the number of teams, unless the CTA's rows all fit and no stage is used twice."""
    seen = wraps = 0
    for H, T, dedup, pipeline, (count, quant) in itertools.product(
            (128, 384, 512, 1024, 2048, 2560, 4096, 5120, 7168, 16384), (1, 40, 74, 333, 1024, 2048, 4096, 6100, 8192, 16384), (0, 1),
            (AUTO, PHASED, FUSED), ((-1, 14), (0, 1), (0, 3), (0, 14), (1, 14), (4, 2), (8, 14), (13, 14))):
        for E, R in ((32, 8), (256, 32), (288, 72)):
            if k > E:
                continue
            pl = plan(T, H, E, R, k, payload=1, dedup=dedup, pipeline=pipeline, count_warps=count, quant_warps=quant)
            if pl is None or pl["long_rows"]:
                continue
            seen += 1
            rows = -(-T // pl["chunks"])
            assert 1 <= pl["teams"] <= 14 and pl["stages"] >= pl["teams"], pl
            if rows > pl["stages"]:
                wraps += 1
                assert pl["stages"] % pl["teams"] == 0, (T, H, E, R, k, dedup, pipeline, count, quant, pl)
    assert seen > 100 and (k > 8 or wraps > 100)


@pytest.mark.parametrize("pipeline,cfg", [
    # (the layout by clusters needs more words per bin than the kernel that held every bin's bitmaps did)
    (LOCAL, dict(T=22, H=64, E=9360, R=39, k=8)),
    (LOCAL, dict(T=15, H=640, E=10215, R=15, k=20, payload=1)),
    (LOCAL, dict(T=4, H=1128, E=9965, R=5, k=11, dedup=1, num_ctas=4)),
    (AUTO, dict(T=3, H=24656, E=6066, R=1011, k=27)),
    (AUTO, dict(T=179, H=36864, E=988, R=52, k=1, payload=1, dedup=1)),
    (AUTO, dict(T=6, H=18880, E=6714, R=746, k=7, num_ctas=8)),
    # (rank-level rows: the table fits, the maps of the expert-level outputs no longer do)
    (LOCAL, dict(T=5622, H=512, E=12, R=1, k=7, payload=1, dedup=1)),
])
def test_calls_that_were_taken_before_clusters_are_still_taken(pipeline, cfg):
    pl = plan(pipeline=pipeline, **cfg)
    assert pl is not None and pl["smem"] <= SMEM
    assert pl["chunks"] * pl["parts"] <= (cfg.get("num_ctas") or CTAS[0])


def test_a_table_that_does_not_fit_is_refused_by_the_flag_free_schedule():
    for dedup in (0, 1):
        assert plan(T=40000, H=256, E=64, R=8, k=8, dedup=dedup, pipeline=LOCAL) is None
        assert plan(T=40000, H=256, E=64, R=8, k=8, dedup=dedup) is not None


@pytest.mark.parametrize("payload", [0, 1])
def test_a_combine_cta_fits_beside_a_small_dispatch(payload):
    """An SM's shared memory is cut to the smallest size that holds the dispatch's CTA (with its static memory and the 1 KB
    every CTA takes): 1 KB of it must be left, or the combine is placed only when the dispatch has ended."""
    sizes = [kb * 1024 for kb in (8, 16, 32, 64, 100, 132, 164, 196, 228)]
    for H, T, (E, R, k) in itertools.product((256, 512, 1024, 2048, 4096, 5120, 7168), (1, 13, 40, 74, 90, 128, 200, 256, 512),
                                             ((16, 4, 2), (32, 8, 4), (128, 8, 4), (256, 32, 8))):
        pl = plan(T, H, E, R, k, payload=payload, dedup=1)
        for static in (768, 1024, 1280):
            need = pl["smem"] + static + 1024
            size = next(s for s in sizes if s >= need)
            assert size - need >= 1024 or size == sizes[-1], (H, T, E, R, k, pl, static)


@pytest.mark.parametrize("protocol", ["sw", "tff", "dc", "sp"])
def test_protocol_calls_that_were_taken_before_the_receivers_prefix_sums_are_still_taken(protocol):
    """The regions' first rows, which two of the protocols need, take no room from the plan."""
    for E in (5200, 5600):   # the largest tables of one expert per rank that had fitted
        cfg = B.ubep_config_t(E, E, 256, 4, 3000, 128, 0, 0, 0, 0, 0, 0)
        pl = B.ubep_debug_sync_plan(cfg, protocol, 3000, SMEM, CTAS[0])
        assert pl["smem"] <= SMEM and pl["layout"] == B.UBEP_SYNC_LAYOUT_LAUNCHED
