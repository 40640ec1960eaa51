"""Rules of the CUDA sources that no run on a GPU can show to be broken: what
breaks them works for as long as the compiler happens to arrange it so.

1. An aligned barrier (bar.sync, bar.red, barrier.cluster ... .aligned) asks
   that all lanes of a warp execute it together. Every helper that issues one
   brings the warp's lanes together itself, so that it may follow code that
   only some lanes ran (a store by lane 0, a guarded row).
2. A bounded wait counts from when its role begins to wait. Each role of the
   tensor-core kernels first waits for the previous kernel (pdl_wait), so that
   the limit is on the kernel's own work, however long the previous one runs.
"""
import os
import re

import pytest

from paper_2606_13898_gb300 import build

BARRIER = re.compile(r"\b(bar\.(sync|red|arrive)|barrier\.cluster\.(arrive|wait))\b")


def sources():
    return sorted(f for f in os.listdir(build.CSRC) if f.endswith((".cu", ".cuh")))


def read(name):
    with open(os.path.join(build.CSRC, name)) as f:
        return f.read()


def barriers(text):
    """(function, its body up to the barrier) of every barrier in inline assembly."""
    for m in re.finditer(r'"[^"\n]*"', text):
        if BARRIER.search(m.group(0)):
            head = list(re.finditer(r"^__device__ [\w ]*?(\w+)\(", text[:m.start()], re.M))[-1]
            yield head.group(1), text[head.end():m.start()]


@pytest.mark.parametrize("name", sources())
def test_aligned_barriers_converge_their_warp(name):
    for fn, before in barriers(read(name)):
        assert "__syncwarp();" in before, f"{name}: {fn} issues an aligned barrier without __syncwarp()"


def test_the_rule_sees_the_barriers():
    found = {fn for name in sources() for fn, _ in barriers(read(name))}
    assert {"named_bar_sync", "bar_red_or", "cluster_sync", "cluster_arrive_relaxed", "cluster_wait"} <= found, found


@pytest.mark.parametrize("name,roles", [
    ("gemm2_tc.cu", ["TMA producer", "MMA issuer", "epilogue, both CTAs"]),
    ("attn_tc.cu", ["TMA producers", "MMA issuer", "warp 11", "softmax: warpgroup"]),
])
def test_roles_wait_for_the_previous_kernel_before_bounded_waits(name, roles):
    text = read(name)
    kernel = text[text.index("__global__"):]
    starts = [kernel.index("// ---------------- " + r) for r in roles]
    assert starts == sorted(starts)
    shared = "pdl_wait();  // " in kernel[:starts[0]]  # all threads, ahead of the roles
    for r, a, b in zip(roles, starts, starts[1:] + [len(kernel)]):
        role = kernel[a:b]
        first = re.search(r"!mbar_wait\w*\(", role)
        if not shared and first:
            assert "pdl_wait();" in role[:first.start()], f"{name}, {r}: a bounded wait before pdl_wait()"
