"""The dense kernel's TMA producer and tcgen05 issuer are whole warps of which one lane issues.  Nothing else holds their
lanes together between two barriers, so every wait in them has to be the one that the lanes leave together: a lane that
lags behind the issuing one by two phases of a barrier would wait for a parity that has come round again."""
import pathlib
import re

import pytest

CSRC = pathlib.Path(__file__).parent.parent / "paper_2603_18489_b200" / "csrc"


@pytest.mark.parametrize("role", ["TMA producer", "MMA issuer"])
def test_lanes_of_a_warp_wide_role_leave_a_wait_together(role):
    src = (CSRC / "ec_attend_dense_tc.cu").read_text()
    body = re.search(rf"= {role} =+\n(.*?)\n        // =====", src, re.S).group(1)
    assert "elect_one()" in body and "lane == 0" not in body
    waits = re.findall(r"\bmbar_wait\w*", body)
    assert len(waits) >= 2 and set(waits) == {"mbar_wait_warp"}, waits
    ptx = (CSRC / "ec_tc_ptx.cuh").read_text()
    assert re.search(r"void mbar_wait_warp\([^{]*\{\s*mbar_wait\([^;]*;\s*__syncwarp\(\);\s*\}", ptx)
