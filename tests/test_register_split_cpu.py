"""Kernels that hand registers from some warps to others: setmaxnreg.inc waits, without a bound, for registers that the
launch does not hold, and how many it holds is the compiler's choice. So every such kernel is launched only after the
host has asked the runtime for its registers and found the shares covered."""

import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1905_07931_gb300", "csrc")


def _source(path):
    with open(path) as f:
        return re.sub(r"//[^\n]*", "", f.read())


SPLIT = [p for p in sorted(glob.glob(os.path.join(CSRC, "*.cu"))) if "setmaxnreg.inc" in _source(p)]


def test_there_are_such_kernels():
    assert SPLIT


@pytest.mark.parametrize("path", SPLIT, ids=[os.path.basename(p) for p in SPLIT])
def test_host_asks_for_the_registers(path):
    src, helper = _source(path), _source(os.path.join(CSRC, "tc_pair.cuh"))
    own = "cudaFuncGetAttributes" in src and "numRegs" in src
    assert own or ("pair_kernel_ready(" in src and "fa.numRegs * threads >= regs" in helper)


@pytest.mark.parametrize("path", SPLIT, ids=[os.path.basename(p) for p in SPLIT])
def test_shares_cover_every_warp(path):
    """The sum that the host compares with is that of all warps' shares: a warpgroup at the lowered value each for the
    producers, every other warp at its own."""
    src = _source(path)
    vals = {k: int(v) for k, v in re.findall(r"\b(k\w+)\s*=\s*(\d+)\b", src)}
    if "SplitRegs" not in src:
        return      # the other form names the sum where it asks
    pre = "kGs" if "kGsSplitRegs" in src else "kSt"
    total = 128 * vals[pre + "ProdRegs"] + 32 * vals[pre + "EpiWarps"] * vals[pre + "EpiRegs"]
    warps = 4 + vals[pre + "EpiWarps"]
    if pre + "ExpandWarps" in vals:
        total += 32 * vals[pre + "ExpandWarps"] * vals[pre + "ExpandRegs"]
        warps += vals[pre + "ExpandWarps"]
    given = {32 * warps * int(r) for r in re.findall(pre + r"SplitRegs <= k\w+Threads \* (\d+)", src)}
    assert len(given) == 1 and total <= given.pop()
