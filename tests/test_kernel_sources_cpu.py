"""What the kernels' sources state about synchronisation that no run can show to be missing."""
import os
import re

from paper_2609_23536_b200 import build


def _source(name):
    text = open(os.path.join(build.CSRC, name)).read()
    return re.sub(r"//[^\n]*", "", text)


def test_whole_warp_roles_of_the_gemm_leave_every_wait_together():
    """The producer and the issuer run on whole warps and issue from one lane.  A lane that still polls a barrier while that lane
    goes on can find it two phases further: each wait ends in a vote of the warp before anything is issued."""
    raw = open(os.path.join(build.CSRC, "gemm_sm100.cu")).read()
    roles = raw[raw.index("-- TMA producer"):raw.index("-- epilogue")]
    assert len(re.findall(r"\bmbar_wait_warp\(", roles)) == 3 and not re.findall(r"\bmbar_wait\(", roles)
    assert re.search(r"bool mbar_wait_warp\([^{]*\{\s*return __all_sync\(0xffffffffu, mbar_wait\(", _source("gemm_sm100.cu"))
