"""The tile-width tuner of the mixed dressing times the launch that the dressing makes: both take their jobs
(ladder + oooo and the four ring maps) from one function, and nothing else builds such jobs."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2606_04186_gb300", "csrc")


def _body(src, head):
    at = src.index(head)
    return src[at:src.index("\n}\n", at)]


def test_tuner_and_dressing_share_the_launch():
    src = open(os.path.join(CSRC, "dress.cu")).read()
    for head in ("cudaError_t t2_terms_tc(", "cudaError_t tune_ladder("):
        body = _body(src, head)
        assert len(re.findall(r"prepare_r2\(", body)) == 1 and len(re.findall(r"run_ladder\(l\.js,", body)) == 1
        assert "StoreR2{" not in body
    assert len(re.findall(r"js\.j\[\d\] = job\([^;]*StoreR2\{", src)) == 5
