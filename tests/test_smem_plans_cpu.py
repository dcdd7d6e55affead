"""Host-side checks of the shared-memory sizes the launchers ask for: no kernel
may carve up more than it is given.  The sizes come from the library itself, the
kernels' plans from the header the kernels are compiled from; nothing here
touches a GPU."""
import ctypes
import os
import subprocess

import pytest

from paper_0909_4039_gb300 import _build

SRC = r"""
#include "teuk_internal.cuh"
using namespace teuk;
extern "C" long long split_plan(int rows, int N, int tsize) { return split_smem_plan(rows, N, tsize).total; }
extern "C" long long pair_plan(int tr, int N, int ks) { return (long long)pair_smem_bytes(tr, N, ks); }
extern "C" long long lone_size(int prec, int tr, int N, int ks)
{
    if (prec == TEUK_FP32)
        return ks == 1 ? split_smem_bytes<float>(tr, N) : (ks == 2 ? split2_smem_bytes<float>(tr, N) : split3_smem_bytes<float>(tr, N));
    return ks == 1 ? split_smem_bytes<double>(tr, N) : (ks == 2 ? split2_smem_bytes<double>(tr, N) : split3_smem_bytes<double>(tr, N));
}
extern "C" long long pipe_size(int tr, int N, int tsize) { return pipe_smem_plan(tr + 4, N, tsize).total; }
extern "C" int runs_pair(int tr, int N, int ks) { return pair_runs(tr, N, ks); }
extern "C" int eligible(int N) { return pair_eligible(N); }
extern "C" int segment(int N) { return implicit_seg(N); }
extern "C" long long batch_size(int prec, int tr, int N, int ks, int paired)
{
    return (long long)batch_tile_bytes(prec, tr, N, ks, paired != 0);
}
"""
LIMIT = 227 * 1024


@pytest.fixture(scope="module")
def plans(tmp_path_factory):
    lib = _build.build()
    d = tmp_path_factory.mktemp("plans")
    src, so = os.path.join(d, "plans.cu"), os.path.join(d, "plans.so")
    with open(src, "w") as f:
        f.write(SRC)
    subprocess.run([_build.nvcc(), *_build.ARCH, "-std=c++17", "-Xcompiler", "-fPIC", "-shared", "-I", _build.CSRC, "-I",
                    _build.INCLUDE, src, "-o", so, lib, "-Xlinker", "-rpath=" + os.path.dirname(lib)], check=True)
    p = ctypes.CDLL(so)
    for n in ("split_plan", "pair_plan", "batch_size", "lone_size", "pipe_size"):
        getattr(p, n).restype = ctypes.c_longlong
    return p


def _row_copy(N, tsize, ks, seg):
    # tiles that sample their own steps copy the extraction row (two planes)
    return 4 * N * tsize if ks > 1 and tsize == 4 and seg == 4 else 0


@pytest.mark.parametrize("ks", [1, 2])
@pytest.mark.parametrize("N", [16, 63, 64, 127, 128, *range(129, 257), 257, 300, 512])
def test_batch_tiles_hold_the_plan_of_their_kernel(plans, N, ks):
    """Every width, height and precision: a batch tile's size holds the plan of
    the kernel that runs it.  A width that runs on packed pairs alone runs
    k_split_batch in a batch with a width that does not (129 .. 256, no multiple
    of 4): its tile then holds that kernel's plan, with its paired theta table."""
    for prec, tsize in ((0, 8), (1, 4)):
        for paired in (False, True):
            if paired and not (tsize == 4 and plans.eligible(N)):
                continue
            for tr in range(1, 255):
                size = plans.batch_size(prec, tr, N, ks, paired)
                first = plans.split_plan(tr + 2, N, tsize)
                if paired:
                    full = plans.pair_plan(tr, N, ks)
                else:
                    full = plans.split_plan(tr + 2 * ks, N, tsize) + _row_copy(N, tsize, ks, plans.segment(N))
                if min(first, full) > LIMIT:
                    break
                assert size >= max(first, full), (N, ks, tr, prec, paired)


@pytest.mark.parametrize("N", range(129, 257))
def test_fp32_tile_heights_are_those_of_plain_rows(plans, N):
    """FP32 rows of 129 to 256 points take every height at which a tile of plain
    rows fits: two state planes, the step table's entries of 20 fields at nodes
    and half nodes, the theta table of 8 fields and, for more steps a launch or
    the pipelined kernel, two rows beside them (each section on 16 bytes).  A pair
    tile's rows are longer; where it does not fit, the scalar kernel runs."""
    def up(x):
        return -(-x // 16) * 16

    def plain(R, positions):
        return 2 * up(8 * R * N) + up(positions * 20 * 4) + up(8 * 4 * N)

    for ks in (1, 2, 3):
        for tr in range(1, 255):
            R = tr + 2 * ks
            need = plain(R, 2 * R - 1) + (2 * 8 * N if ks > 1 else 0)
            if need > LIMIT - 1400:   # (a kernel's own static part)
                break
            size = plans.lone_size(1, tr, N, ks)
            # the plan of the kernel that runs, and of a first step's at this height
            full = plans.pair_plan(tr, N, ks) if plans.runs_pair(tr, N, ks) else plans.split_plan(R, N, 4)
            assert max(full, plans.split_plan(tr + 2, N, 4)) <= size <= LIMIT - 1400, (N, ks, tr)
            if ks < 3:
                assert plans.batch_size(1, tr, N, ks, 0) <= LIMIT - 1400, (N, ks, tr)
    for tr in range(1, 255):
        R = tr + 4
        need = up(8 * 4 * N) + 2 * up(8 * N) + 2 * (2 * up(8 * R * N) + up(2 * R * 20 * 4) + up(4 * (R + 8)))
        assert need > LIMIT - 1400 or plans.pipe_size(tr, N, 4) <= LIMIT - 1400, (N, tr)
