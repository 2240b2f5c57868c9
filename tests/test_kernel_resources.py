"""What ptxas reports for the kernels (the library's own compile, no GPU): local memory, which
the driver reserves for every thread the GPU can hold once a kernel that uses it runs, and the
registers that decide how many threads an SM holds."""
import os
import re

import pytest

from paper_2608_23048_gb300 import _build


@pytest.fixture(scope="module")
def usage():
    """{mangled kernel name: (registers, stack bytes, bytes of spill stores)} per source file."""
    try:
        _build.nvcc()
    except RuntimeError:
        pytest.skip("needs nvcc")
    _build.build(force=not all(os.path.exists(_build.log_of(s)) for s in _build.SOURCES))
    out = {}
    for src in _build.SOURCES:
        with open(_build.log_of(src)) as f:
            text = f.read()
        out[src] = {
            m[1]: (int(m[4]), int(m[2]), int(m[3])) for m in re.finditer(
                r"Compiling entry function '(\w+)'[^\n]*\n[^\n]*\n\s*(\d+) bytes stack frame, (\d+) bytes spill "
                r"stores[^\n]*\n[^\n]*Used (\d+) registers", text)}
    return out


def test_local_memory(usage):
    """The widest patterns' backward keeps 31 steps of 32 weights (3968 B) and ExactGroup's few
    rows of 32 beside them, not a second history."""
    stacks = {name: u[1] for kernels in usage.values() for name, u in kernels.items()}
    assert len(stacks) > 50
    assert max(stacks.values()) <= 5000, max(stacks, key=stacks.get)


def test_exact_kernels(usage):
    """The kernels of the patterns at a tau too small for the WIDE relaxation: 64 registers or
    fewer (eight CTAs of 128 threads an SM), and frames of 16 bytes times an odd number, which
    spread over the sets of the L1."""
    exact = {n: u for n, u in usage["roi_any.cu"].items() if "exact" in n}
    assert len(exact) == 2
    assert all(regs <= 64 and stack % 32 == 16 for regs, stack, _ in exact.values()), exact


def test_4of8_adamw_does_not_spill(usage):
    """4:8 at tau != 1 with the fused optimizer: the order of the sweep's sums and where the
    optimizer's arguments live decide whether the tile loops keep within 168 registers (they
    spilled 8 B alone, 168 and 268 B in runs, which cost up to 15 %)."""
    for name in ("roi_bwd_kernel", "roi_bwd_multi_kernel"):
        kernels = {n: u for n, u in usage["roi_bwd.cu"].items() if name + "ILi4ELi8ELb0ELb0ELb1E" in n}
        assert len(kernels) == 2 and all(u[2] == 0 for u in kernels.values()), kernels
