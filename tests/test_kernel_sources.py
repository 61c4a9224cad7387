"""Rules on the kernel sources that no run can show reliably."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2607_20125_b200", "csrc")


def code(name):
    text = open(os.path.join(CSRC, name)).read()
    return re.sub(r"//[^\n]*|/\*.*?\*/", "", text, flags=re.S)


def test_kernels_that_overlap_their_predecessor_read_nothing_through_the_non_coherent_path():
    """They may be resident while the kernel before them still writes; the wait orders ordinary loads only."""
    overlapping = [f for f in sorted(os.listdir(CSRC)) if "pdl_wait" in code(f)]
    assert "attn_kernel.cuh" in overlapping and "score_kernels.cuh" in overlapping and "move_kernels.cuh" in overlapping
    for f in overlapping + ["headcast_api.cu"]:
        assert not re.search(r"__ldg|\.nc\b|__restrict__", code(f).replace("b.nc", "").replace("bx.nc", "")), f


def test_every_kernel_launched_with_overlap_waits_before_it_works():
    launched = set(re.findall(r"launch_pdl\((?:[^,;]*\? )?([a-z_]+_kernel)", code("headcast_api.cu")))
    assert {"attn_kernel", "combine_kernel", "move_kernel", "cls_combine_kernel", "proxy_combine_kernel", "head_decide_kernel",
            "noalloc_list_kernel"} == launched
    sources = {f: code(f) for f in os.listdir(CSRC)}
    for name in launched:
        bodies = [t[m.end():] for t in sources.values() for m in re.finditer(r"\b" + name + r"\((?:[^()]|\([^()]*\))*\)\s*\{", t)]
        assert len(bodies) == 1, name
        before = bodies[0].split("pdl_wait();")[0]
        assert len(before) < 3000 and "__global__" not in before, name
