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
int chain(int W, int r, int K, int L) { return chain_beside_clusters(W, r, K, L); }
int64_t round_(int W, int c, int u, int K, int L) { return cluster_survivors(W, c, u, K, L); }
}
"""


@pytest.fixture(scope="module")
def plan(tmp_path_factory):
    d = tmp_path_factory.mktemp("cluster")
    (d / "p.cpp").write_text(SRC)
    subprocess.check_call(["g++", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, str(d / "p.cpp"), "-o", str(d / "p.so")])
    lib = ctypes.CDLL(str(d / "p.so"))
    i, z, q = ctypes.c_int, ctypes.c_size_t, ctypes.c_int64
    for name, args, res in (("rows", [i, q], i), ("round_", [i] * 5, q), ("bytes", [i, q, i, i], z), ("survivors", [z, i, i, i], q)):
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


# us of a call on a B200, W, columns a CTA, blocks, steps, tokens, chain, clusters
CHAIN_OR_CLUSTERS = [
    (512, 128, 12, 1, 1, 112, 97), (768, 128, 12, 1, 4, 124, 131), (768, 128, 12, 1, 14, 135, 131), (768, 128, 12, 1, 24, 142, 133), (768, 128, 6, 1, 14, 86, 81), (768, 128, 12, 4, 12, 417, 379),
    (768, 64, 12, 1, 12, 138, 125), (1024, 128, 3, 1, 8, 66, 72), (1024, 128, 3, 2, 4, 95, 102), (1024, 128, 3, 4, 1, 152, 166),
    (1024, 128, 3, 4, 24, 184, 167), (1024, 128, 3, 8, 1, 274, 298), (1024, 128, 3, 8, 12, 313, 299), (1024, 128, 12, 4, 8, 458, 490),
    (1024, 128, 12, 4, 24, 515, 490), (1024, 128, 12, 8, 4, 828, 920), (1024, 128, 12, 8, 20, 962, 921), (1024, 128, 1, 4, 8, 109, 101),
    (1024, 64, 3, 2, 8, 94, 100), (1024, 64, 3, 2, 20, 109, 101), (1024, 64, 12, 2, 16, 285, 262), (1024, 64, 12, 8, 4, 837, 878),
    (1280, 128, 3, 8, 4, 353, 387), (1280, 128, 3, 8, 24, 411, 391), (1280, 128, 12, 4, 16, 580, 619), (1280, 128, 1, 4, 24, 131, 119),
    (1536, 96, 3, 8, 8, 417, 450), (1536, 96, 3, 4, 28, 258, 248), (1536, 96, 12, 4, 28, 713, 736), (1536, 96, 1, 8, 20, 259, 233),
    (2048, 128, 1, 8, 12, 273, 316), (2048, 128, 12, 8, 32, 1717, 1981), (1792, 128, 3, 4, 32, 302, 311)]
# W, clusters, units, blocks, steps, tokens, tiles, clusters
TILES_OR_CLUSTERS = [
    (256, 74, 4, 3, 1, 3552, 89, 79), (256, 74, 4, 3, 1, 4736, 94, 106), (256, 74, 4, 12, 1, 4736, 233, 210), (256, 74, 4, 2, 2, 4440, 120, 129),
    (512, 33, 4, 3, 1, 1584, 104, 84), (512, 33, 4, 3, 1, 2112, 106, 113), (512, 33, 4, 4, 1, 1980, 125, 131), (512, 33, 4, 5, 1, 2112, 144, 152),
    (512, 33, 4, 1, 2, 2112, 103, 108), (512, 33, 4, 2, 2, 1848, 147, 137), (512, 33, 4, 1, 4, 2112, 179, 174), (768, 22, 4, 3, 1, 1408, 121, 131),
    (1024, 15, 4, 3, 1, 720, 133, 124), (1024, 15, 4, 3, 1, 748, 122, 132), (1024, 15, 4, 4, 1, 748, 155, 159), (1024, 15, 4, 3, 1, 960, 130, 143), (1024, 15, 4, 3, 4, 960, 445, 390), (1280, 11, 3, 4, 1, 528, 193, 174),
    (1536, 7, 2, 1, 1, 224, 84, 66)]


def test_the_schedule_that_was_measured_faster(plan):
    """Where two schedules differ by 2 % and more, the rules take the faster one."""
    for W, rows, L, K, tokens, chain, clusters in CHAIN_OR_CLUSTERS:
        assert (tokens <= plan.chain(W, rows, K, L)) == (chain < clusters), (W, rows, L, K, tokens)
    for W, n, units, L, K, tokens, tiles, clusters in TILES_OR_CLUSTERS:
        assert (tokens <= plan.round_(W, n, units, K, L)) == (clusters < tiles), (W, L, K, tokens)


@pytest.mark.parametrize("W", range(256, 2049, 256))
def test_rules_are_monotonic_and_bounded(plan, W):
    for L in range(1, 65):
        for rows in (64, 96, 128):
            limits = [plan.chain(W, rows, K, L) for K in range(1, 65)]
            assert limits == sorted(limits, reverse=True) and 0 <= limits[-1] and limits[0] <= 32
        for K in (1, 2, 3, 4, 64):
            assert 33 * 64 * 12 // 16 <= plan.round_(W, 33, 4, K, L) <= 33 * 64
