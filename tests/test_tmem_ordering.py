"""Tensor-memory ordering, read off the kernel sources: some warps store the twiddles that all warps of
their quadrant load, so between the stores and the first load there must be, in this order, a
tcgen05.fence::before_thread_sync, a CTA barrier and a tcgen05.fence::after_thread_sync, also on the
way of a CTA's first segment group.  (A missing fence is a race that need not show in any output.)"""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1711_10855_gb300", "csrc")
EVENTS = re.compile(r"(?P<store>\btwiddles_to_tmem<)|(?P<before>\btmem_fence_before_sync\(\))"
                    r"|(?P<barrier>\b__syncthreads(?:_and)?\()|(?P<after>\btmem_fence_after_sync\(\))"
                    r"|(?P<load>\b(?:forward_to_tmem|forward_transform|exchange_pass2|exchange_twist_pass2)<)")


def block_end(text, start):
    """Index after the brace block that opens at or after `start`."""
    i = text.index("{", start)
    depth = 0
    for j in range(i, len(text)):
        depth += {"{": 1, "}": -1}.get(text[j], 0)
        if depth == 0:
            return j + 1
    raise AssertionError("unbalanced braces")


def kernels():
    for name in ("fdas_convolve.cu", "fdas_convolve_wide.cu"):
        with open(os.path.join(CSRC, name)) as f:
            text = re.sub(r"//[^\n]*", "", f.read())
        for m in re.finditer(r"__global__\s+void\s+__launch_bounds__\([^)]*\)\s*(\w+)\(", text):
            body = text[m.end():block_end(text, m.end())]
            if "twiddles_to_tmem<" in body:
                yield m.group(1), body


CASES = list(kernels())


def test_every_kernel_is_found():
    assert sorted(n for n, _ in CASES) == ["fdas_convolve_pairs_kernel", "fdas_convolve_tmem_kernel",
                                           "fdas_convolve_wide_kernel", "fdas_segment_spectra_kernel"]


@pytest.mark.parametrize("name,body", CASES, ids=[n for n, _ in CASES])
def test_twiddle_stores_are_ordered_before_the_first_load(name, body):
    # what a CTA does only from its second group on does not order its first
    while (m := re.search(r"if \(a > 0\)\s*\{", body)):
        body = body[:m.start()] + body[block_end(body, m.start()):]
    wanted = ["before", "barrier", "after"]
    for ev in EVENTS.finditer(body, body.index("twiddles_to_tmem<")):
        if ev.lastgroup == "store":
            wanted = ["before", "barrier", "after"]
        elif ev.lastgroup == "load":
            break
        elif wanted and ev.lastgroup == wanted[0]:
            wanted.pop(0)
    assert not wanted, f"{name}: no {wanted} between the twiddle stores and the first load"
