"""Counters in shared memory that a whole CTA zeroes and its warps then add to:
in every kernel a block barrier stands between the zeroing and the first add (a
warp that is done early would otherwise add to entries another warp then zeroes,
and the counts come out too small).  Read from the source: such a race shows on a
GPU once in a great many calls."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2511_19457_gb300", "csrc")
BARRIER = re.compile(r"__syncthreads\(\)|named_bar_sync\(")


def _kernels():
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        src = re.sub(r"//[^\n]*", "", open(path).read())
        for part in src.split("__global__")[1:]:
            yield os.path.basename(path), part[:part.find("\n}")]


def _counters():
    for name, body in _kernels():
        for arr in sorted(set(re.findall(r"atomicAdd\(&(s_\w+)\[", body))):
            kernel = re.search(r"(\w+)\(const|(\w+_kernel)\b", body).group(0).split("(")[0]
            yield pytest.param(body, arr, id=f"{name}-{kernel}-{arr}")


@pytest.mark.parametrize("body,arr", list(_counters()))
def test_barrier_between_zeroing_and_adding(body, arr):
    zero = re.search(re.escape(arr) + r"\[[^=;]*\] = 0u;", body)
    assert zero, f"{arr} is added to but never zeroed"
    add = body.find(f"atomicAdd(&{arr}[")
    assert add > zero.end()
    assert BARRIER.search(body, zero.end(), add), f"no block barrier between zeroing {arr} and adding to it"


def test_finds_the_kernels():
    ids = " ".join(p.id for p in _counters())
    for k in ("ln_rows", "attention", "dw3", "igemm", "onetile"):
        assert k in ids, ids
