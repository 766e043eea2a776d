"""Kernels that may start before the launch ahead of them is complete (pdl_wait()) read what that launch writes through
plain pointers: a const __restrict__ parameter or a __ldg lets the compiler move the load ahead of the wait.  Read from
the source; what is constant by then is listed with the reason."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2403_18661_gb300", "csrc")
WEIGHTS = "parameters of the context, complete when it was created"
DESCRIPTORS = "copied to the device before the first launch of the chain"
CONSTANT = {"gamma": WEIGHTS, "beta": WEIGHTS, "fc_w": WEIGHTS, "fc_b": WEIGHTS, "tap": WEIGHTS, "wt": "table",
            "g_ftab": "table", "g_tw": "table", "w": WEIGHTS, "gam": WEIGHTS, "bet": WEIGHTS, "a.fc_w": WEIGHTS,
            "a.fc_b": WEIGHTS, "d": DESCRIPTORS, "pieces": DESCRIPTORS,
            "x": "strain, complete before the filter build that triggers the whitening"}
FILES = sorted(glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cuh")))


def functions(src):
    """(head, body) of the __global__ and __device__ functions of a source."""
    for m in re.finditer(r"__(?:global|device)__[^{};]*?\([^{};]*\)\s*\{", src):
        end, depth = m.end(), 1
        while depth:
            depth += {"{": 1, "}": -1}.get(src[end], 0)
            end += 1
        yield m.group(0), src[m.end():end]


def violations(src):
    out = []
    for head, body in functions(src):
        kernel = "__global__" in head
        waits = "pdl_wait()" in body or "whiten_block<" in body  # (k_whiten waits inside the block)
        if kernel and not waits:
            continue
        name = re.search(r"(\w+)\s*\([^()]*(?:\([^()]*\)[^()]*)*\)\s*\{$", head).group(1)
        if kernel:
            out += [(name, p) for p in re.findall(r"const[^,()]*__restrict__\s+(\w+)", head) if p not in CONSTANT]
        for arg in re.findall(r"__ldg\(\s*(?:reinterpret_cast<[^>]*>\()?&?([\w.]+)", body):
            if arg not in CONSTANT:
                out.append((name, "__ldg " + arg))
    return out


def test_the_scan_sees_both_forms():
    src = """__global__ void __launch_bounds__(64) k_a(const float *__restrict__ raw, const float *__restrict__ gamma, float *o) {
    if (o) { pdl_wait(); }
    o[0] = raw[0] + __ldg(&raw[1]) + __ldg(gamma + 1);
}
__global__ void k_b(const float *__restrict__ raw, float *o) { o[0] = __ldg(raw); }"""
    assert violations(src) == [("k_a", "raw"), ("k_a", "__ldg raw")]


@pytest.mark.parametrize("path", FILES, ids=os.path.basename)
def test_dependent_launches_read_plain_pointers(path):
    src = re.sub(r"//[^\n]*", "", open(path).read())
    if "pdl_wait" not in src:
        return
    assert violations(src) == []
