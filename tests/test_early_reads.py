"""The last launch of a chunked call reads ahead of its own wait on the launches before it.  Only that wait makes what they wrote
visible to reads that L1 may answer, so what comes ahead of it has to come from L2: TMA, bulk copies, or loads at the scope of the
GPU.  No run can show a stale line of L1 at will; this reads the sources."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2405_18425_b200", "csrc")


def _kernel(name, kernel):
    text = open(os.path.join(CSRC, name)).read()
    text = re.sub(r"//[^\n]*", "", text)
    start = text.index("{", text.index(kernel + "("))
    depth = 0
    for at in range(start, len(text)):
        depth += {"{": 1, "}": -1}.get(text[at], 0)
        if depth == 0:
            return text[start:at]
    raise AssertionError(kernel)


@pytest.mark.parametrize("name,kernel", [("bigla_mma.cu", "bigla_mma_kernel"), ("bigla_grad.cu", "bigla_grad_kernel")])
def test_reads_ahead_of_the_wait_come_from_l2(name, kernel):
    body = _kernel(name, kernel)
    assert "if (MODE != kMain) {\n        pdl_wait();" in body        # the mode that reads ahead, and no other
    assert not re.findall(r"\bflags\[[^\]]*\](?!\s*=[^=])", body)      # flags are written as such, and read ...
    assert len(re.findall(r"ld_gpu4\(\w+\.flags \+", body)) == 1       # ... at the scope of the GPU
    assert set(re.findall(r"\bload_pairs<([^>]*)>", body)) <= {"DK, MODE == kMain"}


def test_early_rows_are_loaded_at_gpu_scope():
    text = open(os.path.join(CSRC, "mma.cuh")).read()
    body = text[text.index("void load_pairs("):]
    body = body[:body.index("\n}\n")]
    loads = [line for line in body.splitlines() if "reinterpret_cast<const" in line and "*reinterpret_cast" in line]
    assert len(loads) == 3 and all(re.search(r"AHEAD \? ld_gpu(16|8|4)\(", line) for line in loads)
    ptx = open(os.path.join(CSRC, "ptx.cuh")).read()
    assert len(re.findall(r"ld\.relaxed\.gpu\.global\.(?:v[24]\.)?u32", ptx)) == 3


def test_kernels_that_may_start_early_do_not_take_inputs_for_read_only():
    """A kernel launched with programmatic serialization may start while the one that writes its inputs still runs: they are not
    read-only for its lifetime, so nothing may lead the compiler to the loads that assume it."""
    early = 0
    for name in sorted(os.listdir(CSRC)):
        if not name.endswith(".cu"):
            continue
        text = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name)).read())
        for m in re.finditer(r"__global__[^{;]*?\b(\w+_kernel)\(([^{;]*?)\) \{", text):
            if re.search(r"<<<", text) and re.search(m.group(1) + r"(?:<[^<>]*>)?<<<", text):
                continue   # an ordinary launch
            early += 1
            assert "__restrict__" not in m.group(2), m.group(1)
    assert early >= 10
    sources = "".join(open(os.path.join(CSRC, n)).read() for n in os.listdir(CSRC) if n.endswith((".cu", ".cuh")))
    assert "__ldg(" not in sources and "ld.global.nc" not in sources
