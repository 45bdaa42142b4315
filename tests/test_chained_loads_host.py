"""Kernels that may begin before the kernel ahead of them has ended (those that call
grid_wait) read what a kernel of the same call wrote through plain pointers: the
read-only path, which const __restrict__ parameters and __ldg take, is for data that is
constant over the kernel's lifetime.  Read from the source: such a kernel's read-only
parameters are the caller's data, which grid_wait gets, or tables written once when the
plan is made."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(__file__), os.pardir, "paper_1712_05834_gb300", "csrc")
CALLERS = {"pos", "w", "vals", "item_off"}
TABLES = {"twg", "modes1d", "modes2d"}


def _kernels():
    for name in sorted(os.listdir(CSRC)):
        if not name.endswith(".cu"):
            continue
        text = open(os.path.join(CSRC, name)).read()
        for m in re.finditer(r"__global__ void[^;{]*?\b(k_\w+)\(([^{;]*?)\)\s*\{\s*grid_wait\(([^)]*)\);", text):
            yield m.group(1), m.group(2), m.group(3)


KERNELS = list(_kernels())


def test_every_waiting_kernel_is_found():
    calls = sum(len(re.findall(r"^\s*grid_wait\(", open(os.path.join(CSRC, f)).read(), re.M))
                for f in os.listdir(CSRC) if f.endswith(".cu"))
    assert calls == len(KERNELS) >= 10, (calls, [k[0] for k in KERNELS])


@pytest.mark.parametrize("kernel,params,waited", KERNELS, ids=[k[0] for k in KERNELS])
def test_read_only_parameters(kernel, params, waited):
    read_only = set(re.findall(r"const\s+\w+(?:\s+\w+)*\s*\*\s*__restrict__\s+(\w+)", params))
    assert read_only <= CALLERS | TABLES, (kernel, read_only - CALLERS - TABLES)
    assert read_only & CALLERS <= set(re.findall(r"\w+", waited)), kernel


def test_explicit_read_only_loads():
    text = open(os.path.join(CSRC, "pk_kernels.cu")).read()
    for arg in re.findall(r"__ldg\(([^;]*)", text):
        assert re.match(r"(reinterpret_cast<const float4 \*>\(pos\)|p|w|vals) \+", arg), arg
