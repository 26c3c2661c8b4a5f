"""Bulk copies that outlive a failed wait.

A bulk copy writes to its CTA's shared memory until it has landed, and a CTA that
leaves earlier gives that memory to the next one.  So where a bounded wait runs out, a
kernel waits once more, bounded too, for the copies (and matrix instructions) that it
has issued.  The path cannot be taken on purpose on a GPU without holding a copy back;
this reads the sources instead: every block that a kernel enters when a wait has
failed has a wait of its own.
"""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2101_02270_gb300", "csrc")
COPY = r"cp\.async\.bulk[\w.:]*\.mbarrier"


def _block(text, at):
    """The braces' content that opens at or after `at`."""
    start = text.index("{", at)
    depth = 0
    for i in range(start, len(text)):
        depth += {"{": 1, "}": -1}.get(text[i], 0)
        if depth == 0:
            return text[start:i + 1]
    raise AssertionError("unbalanced braces")


def _source(name):
    with open(os.path.join(CSRC, name)) as f:
        text = re.sub(r"//[^\n]*", "", f.read())
    return re.sub(r'"(?:[^"\\\n]|\\.)*"', lambda m: m.group(0).replace("{", "(").replace("}", ")"), text)


@pytest.mark.parametrize("name,kernel,failed", [
    ("kernels.cu", "k_dense_update_fixed(", r"if \(__syncthreads_or\(!"),
    ("dense_il.cu", "k_il_gemm(", r"if \(__syncthreads_or\(!"),
    ("dense_im.cu", " update_fma(", r"if \(fail >= 0"),
    ("dense_im.cu", " update_tc(", r"if \(__syncthreads_or\(!ok \|\|"),
    ("gemm_tc.cuh", " k_gemm_tma(", r"if \(s_fail\)"),
])
def test_a_failed_wait_waits_for_what_is_in_flight(name, kernel, failed):
    body = _block(_source(name), _source(name).index(kernel))
    at = re.search(failed, body)
    assert at, "the failure path is no longer where this test looks for it"
    assert re.search(r"wait\(", _block(body, at.start()))


def test_every_source_with_bulk_copies_is_read():
    with_copies = {n for n in os.listdir(CSRC) if n.endswith((".cu", ".cuh")) and re.search(COPY, _source(n))}
    assert with_copies <= {"kernels.cu", "dense_il.cu", "dense_im.cu", "gemm_tc.cuh"}
