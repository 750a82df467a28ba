"""The choice of kernel variant and scratch size (csrc/plan.cuh), compiled for
the host and run over the accepted shapes with an occupancy made up from the
shared memory and a register limit: every shape fits in a block's shared
memory, and the per-warp scratch always holds what the kernel writes there, a
tick's ranking (a key and two byte indices per instance, padded to four
instances) and, in the loop of few replicas with several instances per lane,
the list of a window's formations (8 bytes per instance)."""
import ctypes
import os
import shutil
import subprocess

import pytest

from paper_2608_16336_gb300 import _build

SRC = r"""
#include <initializer_list>
#include "plan.cuh"
using namespace mt;
struct Res { int fits, c, sms, many, set_bits, scratch; long long smem; };
// an SM of 228 KB of which every block takes 1 KB more, and reg_blocks blocks by
// registers (0: what the kernels' registers allow); more than 227 KB for a block is an error, as it is for the driver
extern "C" Res plan(int R, int N, int K, int T, int Bmax, int sms, int reg_blocks) {
    Plan p;
    const int f = choose_plan(R, N, Bmax, make_layout(N, K, T), sms, 232448, [&](const Plan &q) {
        const int n = q.smem > 232448 ? -1 : (int)(233472 / (q.smem + 1024));
        const int regs = reg_blocks > 0 ? reg_blocks : !q.many ? (q.c <= 2 ? 6 : 4) : q.c == 1 ? 8 : q.c == 2 ? 10 : 6;
        return n < regs ? n : regs;
    }, p);
    return Res{f, p.c, p.sms, p.many, p.set_bits, (int)p.scratch, (long long)p.smem};
}
// shapes and replica counts whose scratch is too small; the last one in *at
extern "C" int too_small(int N, int sms, int *at) {
    int bad = 0;
    for (int K = 1; K <= 16; ++K)
        for (int T : {1, 16, 64})
            for (int B : {1, 5, 6, 64})
                for (int reg_blocks : {4, 5, 6, 8, 10})
                    for (int k = 1; k <= 10; ++k)
                        for (int odd = 0; odd < 2; ++odd) {
                            const int R = 2 * sms * k + odd;
                            const Res p = plan(R, N, K, T, B, sms, reg_blocks);
                            const int np = (N + 3) / 4 * 4, rank = 4 * np + 2 * np;
                            const int list = !p.many && p.c > 1 ? 8 * N : 0;
                            const int scratch = (int)p.scratch;
                            if (scratch < rank || scratch < list || (p.c > 1 && scratch < 1 << p.set_bits)) {
                                ++bad;
                                at[0] = R; at[1] = N; at[2] = K; at[3] = T; at[4] = B;
                            }
                        }
    return bad;
}
// shapes without a plan that fits in a block's shared memory
extern "C" int refused(int N, int *at) {
    int bad = 0;
    for (int K = 1; K <= 16; ++K)
        for (int T = 1; T <= 64; ++T)
            for (int B = 1; B <= 64; ++B)
                for (int R : {1, 700, 8192}) {
                    const Res p = plan(R, N, K, T, B, 152, 4);
                    if (p.fits < 1 || p.smem > 232448) {
                        ++bad;
                        at[0] = R; at[1] = N; at[2] = K; at[3] = T; at[4] = B;
                    }
                }
    return bad;
}
"""


class Res(ctypes.Structure):
    _fields_ = [(n, ctypes.c_int) for n in ("fits", "c", "sms", "many", "set_bits", "scratch")] + [("smem", ctypes.c_longlong)]


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    d = tmp_path_factory.mktemp("plan")
    (d / "plan.cpp").write_text(SRC)
    so = str(d / "plan.so")
    subprocess.run([cxx, "-std=c++17", "-O2", "-Wall", "-Werror", "-shared", "-fPIC", "-x", "c++", "-I",
                    os.path.join(_build.CSRC), str(d / "plan.cpp"), "-o", so], check=True)
    L = ctypes.CDLL(so)
    L.plan.restype = Res
    return L


@pytest.mark.parametrize("sms", [152, 148, 1])
def test_scratch_holds_its_uses(lib, sms):
    at = (ctypes.c_int * 5)()
    for n in range(1, 257):
        assert lib.too_small(n, sms, at) == 0, "R, N, K, T, Bmax = %s" % list(at)


def test_every_accepted_shape_has_a_plan(lib):
    at = (ctypes.c_int * 5)()
    for n in range(1, 257):
        assert lib.refused(n, at) == 0, "R, N, K, T, Bmax = %s" % list(at)


def test_one_instance_per_lane_keeps_its_residency(lib):
    """24 instances with 4 tiers and a batch of 64: four blocks per SM as long as the
    scratch holds the ranking alone, so that 1,024 replicas are all resident."""
    p = lib.plan(1024, 24, 4, 16, 64, 152, 6)
    assert (p.c, p.sms, p.many, p.fits) == (1, 1, 0, 4)


@pytest.mark.parametrize("n,k,replicas,many", [
    (64, 4, 1824, 0), (64, 4, 1825, 1), (64, 4, 2736, 1), (64, 4, 2737, 0), (64, 4, 3648, 0), (64, 4, 3649, 1),
    (64, 4, 8192, 1), (64, 10, 16384, 1), (64, 16, 1520, 0), (64, 16, 2432, 0), (64, 16, 16384, 0), (40, 4, 1825, 1), (32, 4, 1824, 0), (32, 4, 1825, 1),
    (32, 4, 2433, 0), (32, 10, 3840, 1), (1, 4, 1824, 0), (8, 4, 1064, 0), (8, 4, 1065, 1), (16, 4, 1520, 0),
    (16, 4, 1521, 1), (24, 4, 8192, 0), (100, 4, 1216, 0), (100, 4, 1217, 1), (100, 4, 1520, 1), (100, 4, 1824, 1),
    (100, 4, 2048, 0), (100, 4, 2433, 1), (128, 10, 8192, 0), (129, 4, 8192, 0)])
def test_main_loop(lib, n, k, replicas, many):
    """The variant whose waves take less time, on either side of the replica counts that
    fill a wave of 152 SMs; with records in shared memory, of the lines drawn there."""
    p = lib.plan(replicas, n, k, 16, 64, 152, 0)
    assert p.many == many


@pytest.mark.parametrize("k,replicas,scratch", [(4, 2736, 2048), (4, 3952, 2048), (4, 3953, 1024), (4, 16384, 1024), (3, 16384, 2048),
                                                (5, 16384, 1024), (8, 16384, 2048)])
def test_small_scratch_only_where_it_holds_more_blocks(lib, k, replicas, scratch):
    p = lib.plan(replicas, 64, k, 16, 64, 152, 0)
    assert p.many == 1 and p.scratch == scratch

