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
