"""The static-scratch dressing's limit as a caller asks for it: qflow_static_scratch_bytes() is the limit
itself, so a problem whose qflow_dress_workspace() is within it is one the call accepts (its arrays are
never larger than that workspace)."""
import re
from pathlib import Path

from paper_2606_04186_gb300 import qflow


def test_query_returns_the_documented_limit():
    text = (Path(__file__).resolve().parent.parent / "include" / "qflow.h").read_text()
    mib = int(re.search(r"#define QFLOW_STATIC_SCRATCH_BYTES \((\d+)u \* 1024u \* 1024u\)", text).group(1))
    assert qflow.static_scratch_bytes() == mib << 20
    assert qflow.dress_workspace(40, 6) <= qflow.static_scratch_bytes() < qflow.dress_workspace(82, 10)
