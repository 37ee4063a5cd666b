"""Layout of the cluster schedule (csrc/cluster_plan.h), checked on the CPU: everything fits and is aligned."""
import ctypes
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2512_08537_b200", "csrc")

SRC = """
#include "cluster_plan.h"
extern "C" {
int rows(int W, int64_t t) { return cluster_rows(W, t); }
int units(int W, int C, int r) { return cluster_units(W, C, r); }
int smem() { return CL_SMEM - 1024; }
int min_stages() { return CL_MIN_STAGES; }
int direct() { return CL_DIRECT_BYTES; }
void layout(int W, int C, int r, int u, int* o) {
    const ClusterLayout l(W, C, r, u);
    const int v[] = {l.bufs, l.stages, (int)l.stage, (int)l.act, (int)l.u, (int)l.a, (int)l.xb, (int)l.x, (int)l.stats, (int)l.part,
                     (int)l.total};
    for (int i = 0; i < 11; ++i) o[i] = v[i];
}
size_t bytes(int K, int64_t t, int L, int W) { return mods_bytes(K, t, L, W); }
int64_t survivors(size_t b, int K, int L, int W) { return mods_survivors(b, K, L, W); }
int stride(int S) { return mods_stride(S); }
}
"""


@pytest.fixture(scope="module")
def plan(tmp_path_factory):
    d = tmp_path_factory.mktemp("cluster")
    (d / "p.cpp").write_text(SRC)
    subprocess.check_call(["g++", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, str(d / "p.cpp"), "-o", str(d / "p.so")])
    lib = ctypes.CDLL(str(d / "p.so"))
    i, z, q = ctypes.c_int, ctypes.c_size_t, ctypes.c_int64
    for name, args, res in (("rows", [i, q], i), ("bytes", [i, q, i, i], z), ("survivors", [z, i, i, i], q)):
        getattr(lib, name).argtypes, getattr(lib, name).restype = args, res
    return lib


@pytest.mark.parametrize("W", range(256, 4097, 256))
def test_layout(plan, W):
    for tokens in (1, 64, 65, 1 << 20):
        rows = plan.rows(W, tokens)
        assert (rows == 0) == (W > 2048)
        if not rows:
            continue
        assert W % rows == 0 and W // rows <= 16 and rows % 32 == 0 and rows >= 64
        for C in (16, 48, 64):
            most = plan.units(W, C, rows)
            assert 1 <= most <= 4
            for units in range(1, most + 1):
                o = (ctypes.c_int * 11)()
                plan.layout(W, C, rows, units, o)
                bufs, stages, stage, act, u, a, xb, x, stats, part, total = o
                N = 16 * units
                assert total <= plan.smem() and stages >= plan.min_stages()
                assert stage % 1024 == 0 and u == stages * stage and (W // 64 * 64 * rows * 2) % stage == 0
                assert all(v % 16 == 0 for v in (act, u, a, xb, x, stats, part))
                # regions in order, none into the next; the products read 128 rows of a slice of `rows`
                assert act == N * W * 2 and a == u + (bufs - 1) * act and xb == a + act and x == xb + N * 128
                assert stats == x + N * C * 4 and part == stats + N * (W // rows) * 8 and total == part + N * rows // 32 * 8 + (
                    N * (4 - rows // 32) * 8)
                assert u + 128 * 128 <= plan.smem()
                assert bufs == 2 or act > plan.direct()       # direct copies need a buffer each for u and a


@pytest.mark.parametrize("W,L", [(256, 1), (1024, 3), (2048, 64)])
def test_modulation_buffer(plan, W, L):
    for K_max in (1, 4, 64):
        for tokens in (1, 7, 8, 65, 1 << 20):
            b = plan.bytes(K_max, tokens, L, W)
            assert b <= 256 << 20
            for K in (1, K_max):
                S = min(plan.survivors(b, K, L, W), tokens)
                assert plan.stride(S) * K * (3 * L + 2) * W * 4 <= b
                if plan.stride(min(tokens, 1 << 24)) * K_max * (3 * L + 2) * W * 4 <= 256 << 20:
                    assert S == tokens
