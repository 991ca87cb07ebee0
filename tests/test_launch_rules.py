"""The rules that launches follow, on the host: the inline functions of cfa_internal.h compiled on
their own."""
import ctypes
import os
import re
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CODE = r"""
#include "cfa_internal.h"
uint32_t parts_log2(uint64_t item_bytes, uint64_t bytes, uint32_t part_bytes, uint64_t n_items,
                    uint32_t grid)
{
    const cfa_cut cut = {item_bytes, bytes, part_bytes};
    return cfa_parts_log2(&cut, n_items, grid);
}
uint32_t chain_flags(uint32_t i, uint32_t n, int early) { return cfa_chain_flags(i, n, early); }
"""

KIB, MIB = 1 << 10, 1 << 20
GRID = 456
EARLY, WAIT_FIRST, WAIT_LAST, RELEASE = 1, 2, 4, 8


@pytest.fixture(scope="module")
def rules(tmp_path_factory):
    d = tmp_path_factory.mktemp("rules")
    (d / "rules.c").write_text(CODE)
    subprocess.run(["gcc", "-O1", "-std=c11", "-Wall", "-Werror", "-shared", "-fPIC",
                    "-I", os.path.join(ROOT, "include"),
                    "-I", os.path.join(ROOT, "paper_2607_18957_gb300", "csrc"),
                    str(d / "rules.c"), "-o", str(d / "rules.so")], check=True)
    lib = ctypes.CDLL(str(d / "rules.so"))
    lib.parts_log2.argtypes = [ctypes.c_uint64, ctypes.c_uint64, ctypes.c_uint32,
                               ctypes.c_uint64, ctypes.c_uint32]
    lib.parts_log2.restype = ctypes.c_uint32
    return lib


@pytest.mark.parametrize("item,part", [(256 * KIB, 32 * KIB), (2 * MIB, 64 * KIB),
                                       (64 * MIB, 32 * KIB), (32 * KIB, 32 * KIB)])
@pytest.mark.parametrize("n", [1, 7, 256, 4096, 100_000])
def test_full_items_are_cut_to_the_part_size(rules, item, part, n):
    assert item >> rules.parts_log2(item, n * item, part, n, GRID) == part


@pytest.mark.parametrize("item,part", [(256 * KIB, 32 * KIB), (2 * MIB, 64 * KIB),
                                       (4 * MIB, 64 * KIB), (64 * MIB, 32 * KIB)])
@pytest.mark.parametrize("n", [1, 300, 457, 16_000, 1 << 20, 1 << 24, (1 << 31) - 1])
@pytest.mark.parametrize("mean", [16, 8 * KIB, 24 * KIB, 33 * KIB, 100 * KIB, 3 * MIB])
def test_visits_stay_near_the_parts_that_hold_bytes(rules, item, part, n, mean):
    """Items of any size are visited at most once, or once per CTA, or half as often again as there
    are parts with bytes in them; and never 2^31 times or more."""
    visits = n << rules.parts_log2(item, n * mean, part, n, GRID)
    assert visits < 1 << 31
    assert visits <= max(n, GRID, n * mean // part * 3 // 2)


def test_no_cut_without_a_part_size(rules):
    assert rules.parts_log2(64 * MIB, 1 << 40, 0, 1 << 14, GRID) == 0


@pytest.mark.parametrize("early", [0, 1])
@pytest.mark.parametrize("n", [1, 2, 3, 9])
def test_a_call_releases_its_own_kernels_only(rules, n, early):
    """The last kernel of a call never releases its dependents, which are the caller's kernels; a
    kernel that starts early without waiting first follows one that releases; and it waits at its
    end, so that what follows on the stream follows every kernel of the call."""
    flags = [rules.chain_flags(i, n, early) for i in range(n)]
    assert not flags[-1] & RELEASE
    assert flags[0] & (EARLY | WAIT_FIRST) == (EARLY | WAIT_FIRST if early else 0)
    assert not flags[0] & WAIT_LAST
    for before, f in zip(flags, flags[1:]):
        assert before & RELEASE
        assert f & EARLY and f & WAIT_LAST and not f & WAIT_FIRST


def test_kernels_that_start_early_read_with_coherent_loads():
    """A kernel launched early is resident while the one before it writes its source: non-coherent
    loads, for memory that nobody writes while a kernel runs, are for a plan's own descriptors."""
    csrc = os.path.join(ROOT, "paper_2607_18957_gb300", "csrc")
    for name in sorted(os.listdir(csrc)):
        if not name.endswith((".cu", ".cuh")):
            continue
        text = re.sub(r"/\*.*?\*/", "", open(os.path.join(csrc, name)).read(), flags=re.S)
        assert "global.nc" not in text, name
        if name == "cfa_bulk.cu":  # the descriptors, in bulk_fetch
            fetch = text.index("bulk_fetch(")
            text = text[:fetch] + text[text.index("return b;", fetch):]
        assert "__ldg" not in text, name
