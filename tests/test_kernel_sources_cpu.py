"""What the kernels' sources state that no run would show to be missing: synchronisation, registers."""
import os
import re
import subprocess

from paper_2609_23536_b200 import build


def _source(name):
    text = open(os.path.join(build.CSRC, name)).read()
    return re.sub(r"//[^\n]*", "", text)


def test_every_warp_of_the_gemm_leaves_its_waits_together():
    """The producer and the issuer run on whole warps and issue from one lane, the epilogue's tensor-memory loads want all lanes.  A
    lane that still polls a barrier while another has gone on can find it two phases further, or give up alone: each wait ends in
    a vote of the warp."""
    source = _source("gemm_sm100.cu")
    assert len(re.findall(r"\bmbar_wait_warp\(", source)) == 1 + 3 + 2  # the definition; producer and issuer; epilogue
    assert len(re.findall(r"\bmbar_wait\(", source)) == 2  # its definition and the one call
    assert re.search(r"bool mbar_wait_warp\([^{]*\{\s*return __all_sync\(0xffffffffu, mbar_wait\(", source)


def test_every_role_that_loads_into_shared_memory_lets_its_copies_land_before_an_abandoned_launch_ends():
    """The producer, which loads operands, and the storing warp of sums, which loads what they are added to."""
    source = _source("gemm_sm100.cu")
    loads = [m.start() for m in re.finditer(r"\btma_load(_2d)?(<PAIR>)?\((?!uint32_t)", source)]
    roles = [m.start() for m in re.finditer(r"\bif \(warp == 0\) \{|\} else if \([^{]*\bwarp\b[^{]*\) \{", source)] + [len(source)]
    for i in range(len(roles) - 1):
        body = source[roles[i]:roles[i + 1]]
        if any(roles[i] < at < roles[i + 1] for at in loads):
            assert len(re.findall(r"if \(!ok\) let_copies_land\(\);", body)) == 1, body[:60]
    assert len(loads) > 4 and len(re.findall(r"\blet_copies_land\(\)", source)) == 1 + 2


def test_casts_that_share_a_launch_fit_beside_a_gemm_cta(tmp_path):
    """A block of theirs has the registers that a GEMM CTA leaves on its SM, 40 a thread, and needs no more."""
    cmd = [build._nvcc(), "-gencode", "arch=compute_100a,code=sm_100a", "-O3", "-std=c++17", "-Xptxas", "-v", "-I", build.INCLUDE,
           "-I", build.CSRC, "-c", os.path.join(build.CSRC, "kernels_hbm.cu"), "-o", str(tmp_path / "k.o")]
    said = subprocess.run(cmd, check=True, capture_output=True, text=True).stderr
    kernels = re.findall(r"Compiling entry function '\w*quantize_multi_kernel.*?(\d+) bytes spill stores.*?Used (\d+) registers", said, re.S)
    assert len(kernels) == 2 and all(int(spilled) == 0 and int(used) <= 40 for spilled, used in kernels)
