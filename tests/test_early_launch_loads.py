"""Kernels that may start before the kernel in front of them on the stream ends
(they call grid_dep_wait) read what that kernel writes with ordinary loads: the
read-only path (const __restrict__ parameters, __ldg) is for data that nothing writes
while the kernel is resident.  What may go through it is constant once a launch can
name it: the model's K and track grid, and the rows C K^t of a session."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_1906_02318_gb300", "csrc")
# row, src: pointers into K, its staged layouts and C K^t, in the kernels that use them
CONSTANT = re.compile(r"(row\b|&?src\b|K \+|&?a\.safety\.track\.blob|"
                      r"reinterpret_cast<const float4\*>\((a\.K|row)\b)")


def _kernels():
    """(name, parameters, body) of every kernel in the sources that waits for the one
    before it."""
    for f in sorted(os.listdir(CSRC)):
        if not f.endswith((".cu", ".cuh")):
            continue
        text = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, f)).read())
        for m in re.finditer(r"__global__", text):
            at = re.search(r"(\w+)\s*\(((?:const __grid_constant__ )?[^()]*)\)\s*\{",
                           text[m.end():])
            if at is None:
                continue
            start = m.end() + at.end()
            depth, i = 1, start
            while depth:
                depth += {"{": 1, "}": -1}.get(text[i], 0)
                i += 1
            if "grid_dep_wait" in text[start:i]:
                yield at.group(1), at.group(2), text[start:i]


KERNELS = list(_kernels())


def test_the_early_launched_kernels_are_found():
    names = {k[0] for k in KERNELS}
    assert {"tick_kernel", "tc_tick_kernel", "factored_kernel", "screen_score", "screen_cost",
            "screen_compact", "train_tiles", "reduce_grad"} <= names


@pytest.mark.parametrize("name,params,body", KERNELS, ids=[k[0] for k in KERNELS])
def test_no_read_only_loads_of_data_another_kernel_writes(name, params, body):
    assert "__restrict__" not in params
    for m in re.finditer(r"__ldg\(", body):
        assert CONSTANT.match(body[m.end():]), body[m.start():m.start() + 60]
