"""Buffers of the few-token schedule (csrc/chain_plan.h), checked on the CPU: bounded, and large enough for every call."""
import ctypes
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2512_08537_b200", "csrc")
LIMIT = 128 << 20

SRC = """
#include "chain_plan.h"
extern "C" {
size_t mods(int K, int64_t t, int L, int W) { return chain_mods_bytes(K, t, L, W); }
size_t xch(int K, int64_t t, int L, int W, int C) { return chain_xch_bytes(K, t, L, W, C); }
int survivors(size_t m, size_t x, int K, int L, int W, int C) { return chain_survivors(m, x, K, L, W, C); }
size_t need_mods(int S, int K, int L, int W) { return (size_t)K * S * mods_floats_per_token_step(L, W) * 4; }
size_t need_xch(int S, int K, int L, int W, int C) { return ChainLayout(S, K, L, W, C).total; }
}
"""


@pytest.fixture(scope="module")
def plan(tmp_path_factory):
    d = tmp_path_factory.mktemp("chain")
    (d / "p.cpp").write_text(SRC)
    subprocess.check_call(["g++", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, str(d / "p.cpp"), "-o", str(d / "p.so")])
    lib = ctypes.CDLL(str(d / "p.so"))
    i, z = ctypes.c_int, ctypes.c_size_t
    for name, args, res in (("mods", [i, ctypes.c_int64, i, i], z), ("xch", [i, ctypes.c_int64, i, i, i], z),
                            ("survivors", [z, z, i, i, i, i], i), ("need_mods", [i] * 4, z), ("need_xch", [i] * 5, z)):
        getattr(lib, name).argtypes, getattr(lib, name).restype = args, res
    return lib


@pytest.mark.parametrize("W", [256, 1024, 1536, 2048])
@pytest.mark.parametrize("L", [1, 3, 12, 64])
def test_bounded_and_sufficient(plan, W, L):
    for K_max in (1, 2, 4, 8, 63, 64):
        for max_tokens in (1, 7, 8, 9, 63, 64, 65, 1 << 20):
            for C in (16, 64):
                m, x = plan.mods(K_max, max_tokens, L, W), plan.xch(K_max, max_tokens, L, W, C)
                assert m <= LIMIT and x <= LIMIT
                for K in {1, 2, 4, K_max}:
                    if K > K_max:
                        continue
                    S = plan.survivors(m, x, K, L, W, C)
                    assert 0 <= S <= 64
                    if S:
                        assert plan.need_mods(S, K, L, W) <= m and plan.need_xch(S, K, L, W, C) <= x
                    # and as many as fit: one more would not (or the head never has as many)
                    if S < min(64, max_tokens):
                        assert plan.need_mods(S + 1, K, L, W) > m or plan.need_xch(S + 1, K, L, W, C) > x


def test_the_usual_heads_keep_all_their_tokens(plan):
    for W, L, C in ((256, 2, 16), (1024, 3, 16), (1536, 6, 16), (1536, 12, 64)):
        m, x = plan.mods(4, 32768, L, W), plan.xch(4, 32768, L, W, C)
        assert [plan.survivors(m, x, K, L, W, C) for K in (1, 2, 4)] == [64, 64, 64]
    # many steps of a deep head: fewer
    m, x = plan.mods(64, 64, 12, 512), plan.xch(64, 64, 12, 512, 16)
    assert plan.survivors(m, x, 64, 12, 512, 16) == 26
