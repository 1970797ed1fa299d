"""Registers and shared memory of every kernel against the launch that the sources give it
(block sizes and dynamic shared memory are read from the sources), from ptxas's resource report
of an sm_103a compile.  No GPU is needed."""
import os
import re
import sys
from concurrent.futures import ThreadPoolExecutor

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)

from paper_2608_27128_gb300 import build as B   # noqa: E402
from test_build_budgets import _one, _report    # noqa: E402

SRCS = ["twk_audit.cu", "twk_refine.cu", "twk_repair.cu", "twk_prep.cu", "twk_policy.cu"]
SM_REGS, SM_SMEM, BLOCK_SMEM, RESERVED = 65536, 228 * 1024, 227 * 1024, 1024


@pytest.fixture(scope="module")
def reports():
    with ThreadPoolExecutor(len(SRCS)) as ex:
        return dict(zip(SRCS, ex.map(_report, SRCS)))


def _source(name):
    with open(os.path.join(B.CSRC, name)) as f:
        return f.read()


def _const(src, name, **known):
    m = re.search(rf"constexpr (?:int|uint32_t) {name} = ([^;]+);", _source(src))
    return eval(m.group(1), {}, known)   # integer expressions of this repository's sources


def _registers(regs, threads):
    """Registers of a block: a warp's are allotted in steps of 256."""
    return (regs * 32 + 255) // 256 * 256 * (threads // 32)


@pytest.mark.parametrize("d,count,sym", [(d, c, y) for d in (64, 128)
                                         for c, y in ((0, 0), (1, 0), (0, 1))])
def test_audit_gets_the_registers_its_warpgroups_trade(reports, d, count, sym):
    """The warpgroups' shares after setmaxnreg add up to kLaunchRegs per thread: a launch with
    fewer is refused, one with more does not fit."""
    helpers = _const("twk_audit.cu", "kHelperWarps")
    epilogue = _const("twk_audit.cu", "kEpiWarps")
    threads = 32 * (helpers + epilogue)
    regs, _, _ = _one(reports["twk_audit.cu"], rf"audit_kernelILi{d}ELb{count}ELb{sym}E")
    assert regs == _const("twk_audit.cu", "kLaunchRegs")
    assert _registers(regs, threads) <= SM_REGS


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("blocks", [4, 5, 6])
def test_refine_blocks_per_sm(reports, d, blocks):
    threads = _const("twk_refine.cu", "kRefineThreads")
    regs, spill, smem = _one(reports["twk_refine.cu"], rf"refine_kernelILi{d}ELi{blocks}E")
    assert _registers(regs, threads) * (blocks * 256 // threads) <= SM_REGS
    assert smem == 0
    if blocks == 4:
        assert spill == 0


@pytest.mark.parametrize("kernel", ["select_kernelILi1EE", "select_kernelILi2EE",
                                    "select_kernelILi4EE", "select_kernelILi8EE",
                                    "select_kernelILi16EE", "dedup_kernel"])
def test_selections_two_blocks_per_sm(reports, kernel):
    threads = _const("twk_repair.cu", "kT")
    cap, sort_max = _const("twk_repair.cu", "kCap"), _const("twk_repair.cu", "kSortMax")
    walk = _const("twk_repair.cu", "kWalkChunk")
    regs, spill, smem = _one(reports["twk_repair.cu"], kernel)

    def dynamic(n):                       # config_select; launch_repair for the dedup variant
        sides = 2 * cap * 12
        if kernel != "dedup_kernel":
            return sides
        state = -(-((n + 15) // 16 * 4 + walk * 4) // 16) * 16
        return max(sides, state + sort_max * 12)

    assert spill == 0 and 2 * _registers(regs, threads) <= SM_REGS
    assert 2 * (smem + dynamic(16384) + RESERVED) <= SM_SMEM
    assert smem + dynamic(1 << 19) <= BLOCK_SMEM      # the dedup variant's longest unit


@pytest.mark.parametrize("d,key", [(d, k) for d in (64, 128) for k in "tf"])
def test_prep_unit_block(reports, d, key):
    threads = _const("twk_prep.cu", "kUnitThreads")
    regs, spill, _ = _one(reports["twk_prep.cu"], rf"prep_unit_kernelILi{d}E{key}E")
    assert spill == 0 and _registers(regs, threads) <= SM_REGS


def test_policy_select_block(reports):
    threads = _const("twk_policy.cu", "kPT")
    regs, spill, smem = _one(reports["twk_policy.cu"], "policy_select_kernel")
    assert spill == 0 and _registers(regs, threads) <= SM_REGS
    assert smem <= 48 * 1024
