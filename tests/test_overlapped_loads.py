"""Step kernels overlap: each is resident while the one before still writes the buffer it will
read. Non-coherent loads are undefined there, so no kernel that is launched that way, and no
device function of the step, may use them or let the compiler choose them."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_1507_02518_gb300", "csrc")


def code(name):
    with open(os.path.join(CSRC, name)) as f:
        return re.sub(r"//[^\n]*|/\*.*?\*/", "", f.read(), flags=re.S)


def test_no_non_coherent_loads():
    for name in sorted(os.listdir(CSRC)):
        text = code(name)
        assert "__ldg" not in text, name
        assert not re.search(r"ld(\.\w+)*\.global(\.\w+)*\.nc|__ldcs|__ldlu|__nv_ldg", text), name


def test_overlapped_kernels_have_no_read_only_parameters():
    """const T* __restrict__ parameters are what the compiler turns into non-coherent loads."""
    text = "\n".join(code(n) for n in sorted(os.listdir(CSRC)))
    followers = set(re.findall(r"launch_following\(\s*(\w+)", text)) - {"void"}
    assert {"fix_step_kernel", "adj_step_kernel", "adj_small_kernel", "adj_linear_kernel",
            "pair_linear_kernel", "pair_step_kernel", "fp64_pass_kernel",
            "presolve_fix_kernel"} <= followers
    for k in followers:
        heads = re.findall(r"__global__[^;{]*?\b%s\s*\([^{]*?\)\s*\{" % k, text, flags=re.S)
        assert heads, k
        for h in heads:
            assert "__restrict__" not in h, k
            assert re.search(r"%s\s*\([^{]*\)\s*\{\s*(using[^;]*;\s*)?(follow|wait_before)\(\)" % k,
                             text, flags=re.S), k
