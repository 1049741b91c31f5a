"""Rules that the kernels' sources keep, read from the text: breaking one shows on the GPU only after
another failure, when it is too late to try it there."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1808_01517_gb300", "csrc")


def _source(name):
    with open(os.path.join(CSRC, name)) as f:
        return re.sub(r"//[^\n]*", "", f.read())


def _enclosing_headers(text, pos):
    """Text before each brace that encloses pos, up to the statement's start."""
    out, depth = [], 0
    for i in range(pos - 1, -1, -1):
        if text[i] == "}":
            depth += 1
        elif text[i] == "{":
            if depth == 0:
                j = max(text.rfind(c, 0, i) for c in ";{}")
                out.append(text[j + 1:i])
            else:
                depth -= 1
    return out


def test_a_warp_leaves_its_loop_together():
    """The abort flag may rise between the reads of two lanes of a diverged warp: a loop that whole
    warps run, with warp barriers in it, takes the flag by a vote.  A single thread reads it itself."""
    reads = 0
    for path in sorted(glob.glob(os.path.join(CSRC, "tc_*.cu"))):
        text = _source(os.path.basename(path))
        for m in re.finditer(r"!\s*\*abort_flag", text):
            reads += 1
            single = any("lane == 0" in h for h in _enclosing_headers(text, m.start()))
            assert single, (os.path.basename(path), text[:m.start()].count("\n") + 1)
    assert reads >= 10


def test_in_place_kernels_do_not_declare_their_buffers_apart():
    """delimit_leaky_relu and its backward run in place (dx = dy, as the layers' backward calls it):
    __restrict__ on those two would promise the compiler the opposite."""
    text = _source("elementwise.cu")
    for kernel, names in (("leaky_kernel", "xy"), ("leaky_bf16x8_kernel", "xy"),
                          ("leaky_bwd_kernel", ("dy", "dx")), ("leaky_bwd_bf16x8_kernel", ("dy", "dx"))):
        params = re.search(r"void " + kernel + r"\(([^)]*)\)", text).group(1)
        for name in names:
            assert re.search(r"\* " + name + r"\b", params), (kernel, name, params)
            assert not re.search(r"__restrict__ " + name + r"\b", params), (kernel, name, params)
