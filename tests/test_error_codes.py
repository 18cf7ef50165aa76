"""A failed CUDA call is reported by the code cuda_fail maps it to: CFP_ENOMEM
for a failed allocation, CFP_ECUDA for any other error.  The single-layer calls'
work space, on the source: an allocation cannot be made to fail with another
error in a test."""
import os
import re

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1901_08269_gb300", "csrc")


def test_layer_work_space_reports_the_mapped_code():
    with open(os.path.join(SRC, "cfp_unet.cu")) as h:
        text = re.sub(r"//[^\n]*", "", h.read())
    calls = text[text.index("struct NnWork"):]
    work = calls[:calls.index("\n};")]
    assert all("CFP_CUDA(" in line for line in work.splitlines() if "pool_malloc(" in line)
    # no call names a code of its own for it
    assert "CFP_ENOMEM" not in calls
    assert len(re.findall(r"CFP_TRY\(\w+\.get\(", calls)) == len(re.findall(r"\bNnWork \w+\(ctx\)", calls)) == 2
