"""How the block-prefix gate deals draft blocks to CTAs (csrc/gate_plan.h), checked on the CPU."""
import ctypes
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2512_08537_b200", "csrc")
MAX_BLOCKS = 4096         # capacity of the count scratch
MAX_ROWS = 24576          # row entropies that a CTA's shared memory holds


@pytest.fixture(scope="module")
def plan(tmp_path_factory):
    d = tmp_path_factory.mktemp("plan")
    (d / "p.cpp").write_text('#include "gate_plan.h"\nextern "C" void plan(int64_t nb, int64_t rows, int64_t round, int64_t want, '
                             'int64_t cap, int64_t* out) { auto p = ardiff::plan_draft_blocks(nb, rows, round, want, cap); '
                             'out[0] = p.blocks_per_cta; out[1] = p.grid; }\n')
    subprocess.check_call(["g++", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, str(d / "p.cpp"), "-o", str(d / "p.so")])
    fn = ctypes.CDLL(str(d / "p.so")).plan
    fn.argtypes = [ctypes.c_int64] * 5 + [ctypes.c_void_p]

    def call(nb, rows, want, round_=16, cap=MAX_BLOCKS):
        out = (ctypes.c_int64 * 2)()
        fn(nb, rows, round_, want, cap, out)
        return out[0], out[1]
    return call


def one_wave(nb, rows, want, cap=MAX_BLOCKS):
    """Every CTA of one wave the same number of draft blocks: what serves a shape at all."""
    want = min(want, cap)
    bpc = min(max(-(-nb // want), 1), max(MAX_ROWS // rows, 1))
    return rows <= MAX_ROWS and -(-nb // bpc) <= cap


@pytest.mark.parametrize("want", [1, 148, 296, 592, 1184, 2048, 2049, 2368, 4096, 4736])
def test_no_shape_that_one_wave_serves_is_turned_away(plan, want):
    edges = {1, 2, 147, want - 1, want, want + 1, 2 * want - 1, 2 * want, 2 * want + 1, 3 * want, MAX_BLOCKS - 1, MAX_BLOCKS,
             MAX_BLOCKS + 1, 4400, 4736, 2 * MAX_BLOCKS, 2 * MAX_BLOCKS + 1, 100000, 2 ** 30}
    for nb in sorted(e for e in edges if e > 0):
        for rows in (1, 8, 15, 16, 17, 128, 2048, 4096, 12288, 12289, MAX_ROWS, MAX_ROWS + 1):
            bpc, grid = plan(nb, rows, want)
            assert (grid > 0) == one_wave(nb, rows, want), (nb, rows, want)
            if grid:
                assert grid <= MAX_BLOCKS and bpc * rows <= MAX_ROWS
                assert (grid - 1) * bpc < nb <= grid * bpc            # every draft block, no empty CTA


@pytest.mark.parametrize("round_", [8, 16, 32, 64])
def test_a_second_wave_of_ctas_only_for_draft_blocks_of_two_rounds_of_rows(plan, round_):
    """A CTA costs its start: draft blocks that occupy the warps of a CTA for less than two rounds share CTAs, so that the
    CTAs are one wave; larger ones get a CTA each up to two waves."""
    want = 444
    for nb in (1, want - 1, want, want + 1, 600, 2 * want, 2 * want + 1, 3 * want + 1):
        for rows in (1, round_ // 2, 2 * round_ - 1):
            assert plan(nb, rows, want, round_)[1] <= want
        for rows in (2 * round_, 2 * round_ + 1, 8 * round_):
            bpc, grid = plan(nb, rows, want, round_)
            assert (bpc, grid) == (1, nb) if nb <= 2 * want else grid <= want
