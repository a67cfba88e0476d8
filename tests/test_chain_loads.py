"""Kernels launched as links of a chain (programmatic dependent launch) and what they read, checked on the
CPU from the source.

Such a kernel is resident while the launch before it still writes its input.  That is sound only if it
waits before its first access to memory and reads what the launch before wrote by loads that are coherent
and stay behind the wait: chain_load, not __ldg and not a plain load through a const __restrict__ pointer.
"""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1504_07034_gb300", "csrc")
# kernel: its unit, its argument struct with the members that the launch before wrote, and the functions
# that load for it
CHAINED = {
    "march2d_kernel": ("lbrs_march.cuh", "MarchArgs", ("src",), ("march_load2", "march_rows")),
    "fmarch_kernel": ("lbrs_kernels_fmarch.cu", "FMarchArgs", ("src",), ()),
    "step2d_u2_kernel": ("lbrs_kernels_f16.cu", "F16Args", ("Uin", "gin", "scale"), ()),
}


def _read(name):
    with open(os.path.join(CSRC, name)) as f:
        return re.sub(r"//[^\n]*", "", f.read())


def _body(src, head):
    """The braces after the first match of `head`."""
    m = re.search(head, src)
    assert m, head
    start = src.index("{", m.end())
    depth = 0
    for i in range(start, len(src)):
        depth += {"{": 1, "}": -1}.get(src[i], 0)
        if depth == 0:
            return src[start:i + 1]
    raise AssertionError(head)


def test_every_chained_kernel_is_listed():
    found = set()
    for name in os.listdir(CSRC):
        if name.endswith((".cu", ".cuh")):
            found |= set(re.findall(r"launch_in_chain\([^,]*,\s*(\w+)", _read(name))) - {"void"}
    assert found == set(CHAINED)


@pytest.mark.parametrize("kernel", sorted(CHAINED))
def test_chained_kernels_read_behind_the_wait(kernel):
    unit, args, members, helpers = CHAINED[kernel]
    src = _read(unit)
    body = _body(src, rf"\b{kernel}\(")
    bodies = [body] + [_body(src, rf"\b{h}\(") for h in helpers]
    names = "|".join(members)
    load = re.compile(rf"__ldg|\ba\.({names})\s*\[|chain_load|march_rows<")
    first = load.search(body)
    assert first and "chain_begin();" in body[:first.start()]
    for b in bodies:
        if "if constexpr (CHAINED) {" in b:              # the other branch is of launches outside chains
            b = b[:b.index("} else {")]
        assert "__ldg" not in b
        assert not re.search(rf"\ba\.({names})\s*\[|\*\s*a\.({names})\b", b)
    assert any("chain_load(" in b for b in bodies)
    struct = _body(src, rf"struct {args}\b")
    for m in members:
        decl = re.search(rf"[^;{{}}]*\b{m};", struct).group(0)
        assert "__restrict__" not in decl, decl


def test_unchained_loads_belong_to_unchained_launches():
    """march_load2's read-only loads are the recording form's, which is never launched in a chain."""
    march = _read("lbrs_march.cuh")
    calls = re.findall(r"march_load2<([^>]*)>\(a\.src", march)
    assert calls and all(c == "ODD, !RECORD" for c in calls)
    unit = _read("lbrs_kernels_march.cu")
    body = _body(unit, r"cudaError_t launch_k\(")
    assert body.index("chained = chained && !RECORD;") < body.index("launch_in_chain(")


def test_chain_load_keeps_its_place():
    src = _read("lbrs_chain.cuh")
    loads = re.findall(r"chain_load\(const [^{]*\{(.*?)\n\}", src, re.S)
    assert len(loads) == 3
    for body in loads:
        assert re.search(r"asm volatile\(\"ld\.global\.", body) and ".nc" not in body
