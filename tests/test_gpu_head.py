"""GPU parity of the K-step head against the fp64 oracle, through the C ABI.

Agreement bar: per token, max |out - oracle| <= 2e-2 * RMS(oracle row) (bf16 GEMM operands, fp32
accumulation on the GPU; no rounding in the oracle). The same bar is applied to the velocity
(out - noise) on one-step runs, where the noise no longer props up the RMS. On the full-size
workloads, where several hundred tokens are compared, a token that misses the bar is looked up in
the CPU rounding model (gpu_util.assert_head_parity): it may pass only if bf16 rounding alone
already puts it there.
"""
import numpy as np
import pytest
import torch

import oracle
import rounding_model
import synth
import paper_2512_08537_b200 as ardiff
from gpu_util import assert_head_parity, dev_bf16, dev_f32, require_cuda

pytestmark = pytest.mark.gpu

REL_TOL = 2e-2
SENTINEL = -777.0


def make_head(wl, weights, max_tokens=None, K_max=None):
    return ardiff.Head(wl.C, wl.Dc, wl.W, wl.L, wl.F, wl.K if K_max is None else K_max,
                       wl.n if max_tokens is None else max_tokens, weights)


def run_head(head, cond_bits, noise, t, idx_np, n_rows=None):
    dev = require_cuda()
    cond = dev_bf16(cond_bits)
    nz = dev_f32(noise)
    idx = torch.from_numpy(np.ascontiguousarray(idx_np, dtype=np.int32)).to(dev)
    if idx.numel() == 0:
        idx = torch.zeros(1, dtype=torch.int32, device=dev)
    count = torch.tensor([len(idx_np)], dtype=torch.int32, device=dev)
    out = torch.full(noise.shape, SENTINEL, dtype=torch.float32, device=dev)
    head.ardiff_head_sample(cond, nz, t, idx, count, out)
    st = head.status()
    assert st == 0, ardiff.strerror(st)
    return out.cpu().numpy()


def assert_parity(got, want, rows, what="out"):
    err = np.abs(got[rows].astype(np.float64) - want[rows]).max(axis=1)
    rms = np.sqrt((want[rows] ** 2).mean(axis=1))
    worst = float((err / rms).max())
    assert worst <= REL_TOL, f"{what}: worst max|err|/rms = {worst:.3e}"
    return worst


def sample_tokens(idx, extra=96, seed=0):
    """First tile, a middle tile, the last (ragged) tile, and some random survivors."""
    S = len(idx)
    pos = set(range(min(S, 128)))
    pos |= set(range(max(0, (S // 256) * 128), min(S, (S // 256) * 128 + 64)))
    pos |= set(range(max(0, S - (S % 128 or 128)), S))
    rng = np.random.default_rng(seed)
    pos |= set(int(p) for p in rng.integers(0, S, size=extra))
    return np.array(sorted(pos), dtype=np.int64)


def test_cfg1_all_tokens_gate_then_head():
    dev = require_cuda()
    wl = synth.workload("cfg1")
    feat_bits = synth.features(wl)
    H = oracle.entropy(feat_bits)
    tau = float(np.median(H))
    _, mask_o, idx_o, count_o = oracle.gate(feat_bits, tau)
    w, cond_bits, noise, t = synth.head_weights(wl), synth.cond(wl), synth.noise(wl), synth.t_sched(wl.K)
    want = oracle.head_sample(w, cond_bits, noise, t, idx_o)
    head = make_head(wl, w)
    mask, idx, count, _ = ardiff.ardiff_entropy_gate(dev_bf16(feat_bits), tau)
    out = torch.full(noise.shape, SENTINEL, dtype=torch.float32, device=dev)
    head.ardiff_head_sample(dev_bf16(cond_bits), dev_f32(noise), t, idx, count, out)
    assert head.status() == 0
    got = out.cpu().numpy()
    assert int(count.item()) == count_o
    assert_parity(got, want, idx_o)
    dropped = np.flatnonzero(mask_o == 0)
    assert np.all(got[dropped] == SENTINEL)          # rows of filtered tokens are never written
    head.close()


@pytest.mark.parametrize("std", [0.02, None])
@pytest.mark.parametrize("count", [1, 64, 127, 128, 129, 300])
def test_small_head_ragged_counts(std, count):
    wl = synth.workload("cfg1", n=320)
    w, cond_bits, noise, t = synth.head_weights(wl, std=std), synth.cond(wl), synth.noise(wl), synth.t_sched(wl.K)
    idx = np.random.default_rng(count).permutation(wl.n)[:count].astype(np.int32)   # any order
    want = oracle.head_sample(w, cond_bits, noise, t, idx)
    head = make_head(wl, w)
    got = run_head(head, cond_bits, noise, t, idx)
    assert_parity(got, want, idx)
    rest = np.setdiff1d(np.arange(wl.n), idx)
    assert np.all(got[rest] == SENTINEL)
    head.close()


# Where the schedules change is what ardiff_head_few_limits says. The counts of the tests that were written before the clusters
# came in stay (512 / 513 here, 64 / 65 at every width, 26 / 27 with 64 steps of 12 blocks, 900 tokens in the test of the waits: all
# of them the clusters' now), whatever their docstrings say of the schedule; each has one behind it that takes its counts from the
# limits, or asserts on them, and so reaches the schedule it names.
@pytest.mark.parametrize("count", [512, 513, 3072, 3073, 23808, 23809, 26112, 26113])
def test_item_width_boundaries(count):
    """The last token count of each item width and the first of the next one (W = 512 on 148 SMs: 64 output columns
    per item up to 2 pairs of token tiles, 128 up to 12, then 256), of a group of the usual size (93 pairs), and of a lone
    group (102). Tolerance: the agreement bar of this file."""
    wl = synth.workload("cfg1", n=count + 5, W=512, L=2, K=2)
    w, cond_bits, noise, t = synth.head_weights(wl, std=None), synth.cond(wl), synth.noise(wl), synth.t_sched(wl.K)
    idx = np.random.default_rng(count).permutation(wl.n)[:count].astype(np.int32)
    rows = idx[sample_tokens(idx)]
    want = oracle.head_sample(w, cond_bits, noise, t, rows)
    head = make_head(wl, w)
    got = run_head(head, cond_bits, noise, t, idx)
    assert_parity(got, want, rows)
    assert np.all(got[np.setdiff1d(np.arange(wl.n), idx)] == SENTINEL)
    head.close()


@pytest.mark.parametrize("count", [104, 105, 1024, 1025, 6144, 6145])
def test_item_widths_where_the_modulations_hold_few_tokens(count):
    """64 steps of 12 blocks, W = 256: 256 MB of modulations are those of 104 survivors, so that the tiles begin there, with items
    of 64 columns up to 4 pairs of token tiles, then 128 up to 24, then 256. Tolerance: the agreement bar of this file."""
    wl = synth.workload("cfg1", n=6150, W=256, L=12, K=64)
    w, cond_bits, noise, t = synth.head_weights(wl, std=None), synth.cond(wl), synth.noise(wl), synth.t_sched(wl.K)
    idx = np.random.default_rng(count).permutation(wl.n)[:count].astype(np.int32)
    rows = idx[np.unique(np.concatenate([[0, 63, 64, count // 2, count - 1], np.random.default_rng(2).integers(0, count, 16)]))]
    want = oracle.head_sample(w, cond_bits, noise, t, rows)
    head = make_head(wl, w)
    assert head.few_limits(wl.K) == (0, 104)
    got = run_head(head, cond_bits, noise, t, idx)
    assert_parity(got, want, rows)
    assert np.all(got[np.setdiff1d(np.arange(wl.n), idx)] == SENTINEL)
    head.close()


@pytest.mark.parametrize("W", [256, 512, 768, 1024, 1280, 1536, 1792, 2048, 2304])
def test_few_tokens_at_every_width(W):
    """Up to 64 survivors the chain of layers leaves the tile schedule (one instance per W / 256 up to 8): one token, a
    ragged token tile, a second pass, the last count it takes and the first that it does not; the same call twice gives
    the same bits. Tolerance: the agreement bar of this file."""
    wl = synth.workload("cfg1", n=80, W=W, L=2, K=3, C=32 if W % 512 else 64, Dc=192)
    w, cond_bits, noise, t = synth.head_weights(wl, std=None), synth.cond(wl), synth.noise(wl), synth.t_sched(wl.K)
    order = np.random.default_rng(W).permutation(wl.n).astype(np.int32)
    want = oracle.head_sample(w, cond_bits, noise, t, order[:65])
    head = make_head(wl, w)
    for count in (1, 9, 33, 64, 65):
        idx = order[:count]
        got = run_head(head, cond_bits, noise, t, idx)
        assert_parity(got, want, idx, f"{count} tokens")
        assert np.all(got[np.setdiff1d(np.arange(wl.n), idx)] == SENTINEL)
        assert np.array_equal(run_head(head, cond_bits, noise, t, idx), got)
    head.close()


@pytest.mark.parametrize("n", [64, 80])
@pytest.mark.parametrize("W", [256, 512, 768, 1024, 1280, 1536, 1792, 2048, 2304])
def test_few_tokens_at_the_limits_of_every_width(W, n):
    """One token, the chain where it serves some (its last count and the first of the clusters), ragged token tiles, and up to
    the 64 tokens of heads that split a layer over as many CTAs as a cluster may have (n = 64: 64 columns each up to W = 1024);
    no such schedule above W = 2048. The same call twice gives the same bits. Tolerance: the agreement bar of this file."""
    wl = synth.workload("cfg1", n=n, W=W, L=2, K=3, C=32 if W % 512 else 64, Dc=192)
    w, cond_bits, noise, t = synth.head_weights(wl, std=None), synth.cond(wl), synth.noise(wl), synth.t_sched(wl.K)
    order = np.random.default_rng(W).permutation(wl.n).astype(np.int32)
    want = oracle.head_sample(w, cond_bits, noise, t, order[:65])
    head = make_head(wl, w)
    chain, clusters = head.few_limits(wl.K)
    assert (chain > 0) == (1024 <= W <= 2048) and (clusters >= 64) == (W <= 2048)
    for count in sorted({1, 9, 33, 64, min(n, 65), chain or 2, chain + 1}):
        idx = order[:count]
        got = run_head(head, cond_bits, noise, t, idx)
        assert_parity(got, want, idx, f"{count} tokens")
        assert np.all(got[np.setdiff1d(np.arange(wl.n), idx)] == SENTINEL)
        assert np.array_equal(run_head(head, cond_bits, noise, t, idx), got)
    head.close()


@pytest.mark.parametrize("L", [1, 3, 12])
def test_the_chain_at_its_narrowest_width(L):
    """W = 768, where the chain serves calls of one step only: one token, its last count and the first of the clusters. Tolerance:
    the agreement bar of this file."""
    wl = synth.workload("cfg1", n=80, W=768, L=L, K=2, C=32, Dc=192)
    w, cond_bits, noise, t = synth.head_weights(wl, std=None), synth.cond(wl), synth.noise(wl), synth.t_sched(1)
    order = np.random.default_rng(L).permutation(wl.n).astype(np.int32)
    head = make_head(wl, w)
    chain, clusters = head.few_limits(1)
    assert 1 < chain < 32 and clusters >= 80 and head.few_limits(2)[0] == 0
    want = oracle.head_sample(w, cond_bits, noise, t, order[:chain + 1])
    for count in (1, chain, chain + 1):
        got = run_head(head, cond_bits, noise, t, order[:count])
        assert_parity(got, want, order[:count], f"{count} tokens")
        assert np.array_equal(run_head(head, cond_bits, noise, t, order[:count]), got)
    head.close()


@pytest.mark.parametrize("W,counts", [(256, (80, 81, 2112, 4224, 4225, 4737)), (512, (129, 1600, 2112, 2113)),
                                      (768, (100, 337, 1300)), (1024, (240, 241, 481, 720, 721)),
                                      (1280, (32, 33, 177, 353, 529)), (1536, (32, 33, 112, 113, 224, 225)),
                                      (1792, (33, 112, 225)), (2048, (32, 33, 112, 113, 224, 225))])
def test_token_groups_of_the_clusters(W, counts):
    """Clusters of W / 128 CTAs take groups of 16, 32, 48 or 64 tokens: counts on both sides of where the group grows, where the
    values go through L2 instead of directly, and of the last that fits (on 148 SMs); a ragged last group; fresh noise; the
    same call twice gives the same bits. Tolerance: the agreement bar of this file."""
    dev = require_cuda()
    wl = synth.workload("cfg1", n=max(counts) + 3, W=W, L=2, K=2, C=48 if W % 512 else 16, Dc=128)
    w, cond_bits, noise = synth.head_weights(wl, std=None), synth.cond(wl), synth.noise(wl)
    t_in = np.array([0.9, 0.4], np.float32)
    coef = np.array([[0.4, 0.7, 0.5], [0.2, 1.0, 0.1]], np.float32)
    z = np.random.default_rng(9).standard_normal((2, wl.n, wl.C)).astype(np.float32)
    order = np.random.default_rng(W).permutation(wl.n).astype(np.int32)
    pos = np.unique(np.concatenate([[0, 15, 16, 31, 47, 63], np.array(counts) - 1, np.random.default_rng(1).integers(0, max(counts), 24)]))
    want = np.zeros((wl.n, wl.C))
    want[order[pos]] = oracle.head_sample_coef(w, cond_bits, noise, t_in, coef, order[pos], step_noise=z)[order[pos]]
    head = make_head(wl, w)
    cond, noise_d, z_d = dev_bf16(cond_bits), dev_f32(noise), torch.from_numpy(z).to(dev)
    for count in counts:
        outs = []
        for _ in range(2):
            out = torch.full(noise.shape, SENTINEL, dtype=torch.float32, device=dev)
            head.ardiff_head_sample_coef(cond, noise_d, t_in, coef, torch.from_numpy(order[:count].copy()).to(dev),
                                         torch.tensor([count], dtype=torch.int32, device=dev), out, step_noise=z_d)
            assert head.status() == 0
            outs.append(out.cpu().numpy())
        rows = order[pos[pos < count]]
        assert_parity(outs[0], want, rows, f"{count} tokens")
        assert np.array_equal(outs[0], outs[1])
        assert np.all(outs[0][order[count:]] == SENTINEL) and not np.any(outs[0][order[:count]] == SENTINEL)
    head.close()


@pytest.mark.parametrize("W,n,counts", [(256, 4740, (1184, 3552, 3553)), (512, 2116, (528, 529)), (768, 1412, (337,)),
                                        (1024, 964, (720, 721)), (1280, 532, (353,)), (1536, 228, (112,)), (1792, 228, (112, 113)),
                                        (2048, 228, (112,))])
def test_token_groups_up_to_the_limit_of_the_clusters(W, n, counts):
    """Clusters of W / 128 CTAs (W / 96 at 1536) take groups of 16, 32, 48 or 64 tokens: counts on both sides of where the group
    grows, where the values go through L2 instead of directly, the last that they serve and the first that they do not; a
    ragged last group; fresh noise; the same call twice gives the same bits. Tolerance: the agreement bar of this file."""
    dev = require_cuda()
    wl = synth.workload("cfg1", n=n, W=W, L=2, K=2, C=48 if W % 512 else 16, Dc=128)
    w, cond_bits, noise = synth.head_weights(wl, std=None), synth.cond(wl), synth.noise(wl)
    t_in = np.array([0.9, 0.4], np.float32)
    coef = np.array([[0.4, 0.7, 0.5], [0.2, 1.0, 0.1]], np.float32)
    z = np.random.default_rng(9).standard_normal((2, wl.n, wl.C)).astype(np.float32)
    order = np.random.default_rng(W).permutation(wl.n).astype(np.int32)
    head = make_head(wl, w)
    chain, last = head.few_limits(wl.K)
    assert chain <= 32 and max(counts) <= last < n
    counts = counts + (last, last + 1)
    pos = np.unique(np.concatenate([[0, 15, 16, 31, 47, 63], np.array(counts) - 1, np.random.default_rng(1).integers(0, max(counts), 24)]))
    want = np.zeros((wl.n, wl.C))
    want[order[pos]] = oracle.head_sample_coef(w, cond_bits, noise, t_in, coef, order[pos], step_noise=z)[order[pos]]
    cond, noise_d, z_d = dev_bf16(cond_bits), dev_f32(noise), torch.from_numpy(z).to(dev)
    for count in counts:
        outs = []
        for _ in range(2):
            out = torch.full(noise.shape, SENTINEL, dtype=torch.float32, device=dev)
            head.ardiff_head_sample_coef(cond, noise_d, t_in, coef, torch.from_numpy(order[:count].copy()).to(dev),
                                         torch.tensor([count], dtype=torch.int32, device=dev), out, step_noise=z_d)
            assert head.status() == 0
            outs.append(out.cpu().numpy())
        rows = order[pos[pos < count]]
        assert_parity(outs[0], want, rows, f"{count} tokens")
        assert np.array_equal(outs[0], outs[1])
        assert np.all(outs[0][order[count:]] == SENTINEL) and not np.any(outs[0][order[:count]] == SENTINEL)
    head.close()


def test_few_token_limit_set_by_the_buffers():
    """64 steps of 12 blocks: the few-token buffers (128 MB of modulations) hold 26 survivors. The last count that they serve
    and the first that they do not. Tolerance: the agreement bar of this file."""
    wl = synth.workload("cfg1", n=40, W=512, L=12, K=64)
    w, cond_bits, noise, t = synth.head_weights(wl, std=None), synth.cond(wl), synth.noise(wl), synth.t_sched(wl.K)
    order = np.random.default_rng(26).permutation(wl.n).astype(np.int32)
    rows = order[[0, 7, 25, 26]]
    want = oracle.head_sample(w, cond_bits, noise, t, rows)
    head = make_head(wl, w)
    for count in (26, 27):
        got = run_head(head, cond_bits, noise, t, order[:count])
        assert_parity(got, want, rows[:3] if count == 26 else rows, f"{count} tokens")
        assert np.all(got[np.setdiff1d(np.arange(wl.n), order[:count])] == SENTINEL)
    head.close()


def test_few_token_limit_set_by_the_modulations():
    """64 steps of 12 blocks: the modulations (at most 256 MB) are those of 48 survivors. The last count that the clusters serve
    and the first that they do not. Tolerance: the agreement bar of this file."""
    wl = synth.workload("cfg1", n=64, W=512, L=12, K=64)
    w, cond_bits, noise, t = synth.head_weights(wl, std=None), synth.cond(wl), synth.noise(wl), synth.t_sched(wl.K)
    order = np.random.default_rng(26).permutation(wl.n).astype(np.int32)
    rows = order[[0, 7, 47, 48]]
    want = oracle.head_sample(w, cond_bits, noise, t, rows)
    head = make_head(wl, w)
    assert head.few_limits(64) == (0, 48) and head.few_limits(32)[1] >= 64
    for count in (48, 49):
        got = run_head(head, cond_bits, noise, t, order[:count])
        assert_parity(got, want, rows[:3] if count == 48 else rows, f"{count} tokens")
        assert np.all(got[np.setdiff1d(np.arange(wl.n), order[:count])] == SENTINEL)
    head.close()


def test_head_without_room_for_the_few_token_buffers():
    """The few-token schedule's buffers are an accelerator: a device that has room for the rest of a head, but not for them,
    still gets the head, and calls of few tokens take the schedule of larger ones. (The memory is held by one ordinary
    allocation; nothing runs out but the library's own request.)"""
    dev = require_cuda()
    wl = synth.workload("cfg1", n=64, W=512, L=12, K=64)
    w, cond_bits, noise = synth.head_weights(wl, std=None), synth.cond(wl), synth.noise(wl)
    t = synth.t_sched(2)
    idx = np.arange(0, wl.n, 5).astype(np.int32)
    want = oracle.head_sample(w, cond_bits, noise, t, idx)
    head = make_head(wl, w)                          # (kernels loaded; what a whole head takes)
    run_head(head, cond_bits, noise, t, idx)
    with_buffers = torch.cuda.mem_get_info()[0]
    head.close()
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    free = torch.cuda.mem_get_info()[0]
    taken = free - with_buffers
    assert taken > 250 << 20                         # weights and scratch about 100 MB, the buffers 128 MB and more
    held = torch.empty(free - taken + (120 << 20), dtype=torch.uint8, device=dev)
    try:
        head = make_head(wl, w)
        got = run_head(head, cond_bits, noise, t, idx)
        assert_parity(got, want, idx)
        head.close()
    finally:
        del held
        torch.cuda.empty_cache()


def test_head_without_room_takes_the_tiles():
    """The few-token schedule's buffers are an accelerator: a device that has room for the rest of a head, but not for them,
    still gets the head, and calls of few tokens take the schedule of larger ones. (The memory is held by one ordinary
    allocation; nothing runs out but the library's own request.)"""
    dev = require_cuda()
    wl = synth.workload("cfg1", n=64, W=512, L=12, K=64)
    w, cond_bits, noise = synth.head_weights(wl, std=None), synth.cond(wl), synth.noise(wl)
    t = synth.t_sched(2)
    idx = np.arange(0, wl.n, 5).astype(np.int32)
    want = oracle.head_sample(w, cond_bits, noise, t, idx)
    torch.cuda.empty_cache()                         # (what earlier tests left in torch's cache is not this head's)
    head = make_head(wl, w)                          # (kernels loaded; what a whole head takes)
    run_head(head, cond_bits, noise, t, idx)
    with_buffers = torch.cuda.mem_get_info()[0]
    head.close()
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    free = torch.cuda.mem_get_info()[0]
    taken = free - with_buffers
    assert taken > 250 << 20                         # weights and scratch about 100 MB, the buffers 128 MB and more
    held = torch.empty(free - taken + (120 << 20), dtype=torch.uint8, device=dev)
    try:
        head = make_head(wl, w)
        assert head.few_limits(2) == (0, 0)
        got = run_head(head, cond_bits, noise, t, idx)
        assert_parity(got, want, idx)
        head.close()
    finally:
        del held
        torch.cuda.empty_cache()


def test_a_head_for_large_batches_holds_no_modulation_buffer_beside_its_workspace():
    """W = 1024, 3 blocks, 4 steps, 16384 tokens: weights, two groups of 47 pairs of token tiles of every activation, and 64 MB
    for the rest (exchange buffers, tables, allocation granularity); the modulations of one round of clusters are 173 MB."""
    wl = synth.workload("cfg2")
    w = synth.head_weights(wl)
    make_head(wl, w).close()                         # (kernels loaded)
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    free = torch.cuda.mem_get_info()[0]
    head = make_head(wl, w)
    taken = free - torch.cuda.mem_get_info()[0]
    head.close()
    R = 4 * 47 * 128
    weights = 2 * wl.W * (wl.W * (5 * wl.L + 3) + wl.Dc + wl.C + 64 + wl.F)
    scratch = R * (2 * wl.Dc + 2 * 64 + 4 * wl.C + wl.W * (2 * wl.K + 4 * 2 + 4) + 2 * 8 * wl.W // 64)
    assert taken <= weights + scratch + (64 << 20), (taken >> 20, weights >> 20, scratch >> 20)


@pytest.mark.parametrize("W,few", [(512, 300), (1536, 20)])
def test_schedules_that_share_memory_leave_nothing_to_one_another(W, few):
    """Modulations of few tokens and the activations of the tile schedule lie in the same memory: calls of either kind between
    calls of the other give the bits of a head that has only ever run theirs. (W = 512: clusters, 1536: the chain.)"""
    wl = synth.workload("cfg1", n=2600, W=W, L=2, K=2)
    w, cond_bits, noise, t = synth.head_weights(wl, std=None), synth.cond(wl), synth.noise(wl), synth.t_sched(wl.K)
    order = np.random.default_rng(5).permutation(wl.n).astype(np.int32)
    head = make_head(wl, w)
    got = {}
    for count in (few, 2590, few, 2470, few + 7, 2590, few):
        out = run_head(head, cond_bits, noise, t, order[:count])
        assert count not in got or np.array_equal(got[count], out)
        got[count] = out
    for count, out in got.items():
        fresh = make_head(wl, w)
        assert np.array_equal(run_head(fresh, cond_bits, noise, t, order[:count]), out)
        fresh.close()
    head.close()


def test_few_tokens_with_fresh_noise_and_after_a_stall():
    """The sampler form with step noise on few tokens, before and after a call whose conditioning never completes."""
    dev = require_cuda()
    wl = synth.workload("cfg1", n=50, W=512, K=2)
    w, cond_bits, noise = synth.head_weights(wl, std=None), synth.cond(wl), synth.noise(wl)
    idx_np = np.random.default_rng(3).permutation(wl.n)[:41].astype(np.int32)
    t_in = np.array([0.95, 0.5], np.float32)
    coef = np.array([[0.3, 0.7, 0.7], [0.0, 1.0, 0.1]], np.float32)
    z = np.random.default_rng(8).standard_normal((2, wl.n, wl.C)).astype(np.float32)
    want = oracle.head_sample_coef(w, cond_bits, noise, t_in, coef, idx_np, step_noise=z)
    head = make_head(wl, w)
    idx = torch.from_numpy(idx_np).to(dev)
    count = torch.tensor([len(idx_np)], dtype=torch.int32, device=dev)
    clean = None
    for stall in (False, True, False):
        if stall:
            head.inject_stall(0, 3000)
        out = torch.full(noise.shape, SENTINEL, dtype=torch.float32, device=dev)
        head.ardiff_head_sample_coef(dev_bf16(cond_bits), dev_f32(noise), t_in, coef, idx, count, out,
                                     step_noise=torch.from_numpy(z).to(dev))
        assert head.status() == (ardiff.ARDIFF_ERR_TIMEOUT if stall else 0)
        if not stall:
            got = out.cpu().numpy()
            assert_parity(got, want, idx_np)
            assert clean is None or np.array_equal(got, clean)
            clean = got
    head.close()


@pytest.mark.parametrize("std", [0.02, None])
def test_velocity_parity_one_step(std):
    wl = synth.workload("cfg1", n=256, K=1)
    w, cond_bits, noise, t = synth.head_weights(wl, std=std), synth.cond(wl), synth.noise(wl), synth.t_sched(1)
    idx = np.arange(wl.n, dtype=np.int32)
    want = oracle.head_sample(w, cond_bits, noise, t, idx)
    head = make_head(wl, w)
    got = run_head(head, cond_bits, noise, t, idx)
    assert_parity(got - noise, want - noise, idx, "velocity")
    head.close()


def test_k0_copies_noise_and_count0_writes_nothing():
    wl = synth.workload("cfg1", n=200)
    w, cond_bits, noise = synth.head_weights(wl), synth.cond(wl), synth.noise(wl)
    head = make_head(wl, w)
    idx = np.arange(0, 200, 3, dtype=np.int32)
    got = run_head(head, cond_bits, noise, synth.t_sched(0), idx)
    assert np.array_equal(got[idx], noise[idx])
    assert np.all(got[np.setdiff1d(np.arange(200), idx)] == SENTINEL)
    got0 = run_head(head, cond_bits, noise, synth.t_sched(4), np.zeros(0, np.int32))
    assert np.all(got0 == SENTINEL)
    head.close()


def test_nonuniform_schedule_and_k_sweep():
    wl = synth.workload("cfg1", n=192, K=8)
    w, cond_bits, noise = synth.head_weights(wl, std=None), synth.cond(wl), synth.noise(wl)
    head = make_head(wl, w, K_max=8)
    idx = np.arange(wl.n, dtype=np.int32)
    for K in (1, 2, 3, 8):
        t = np.sort(np.random.default_rng(K).uniform(0.0, 1.0, size=K + 1)).astype(np.float32)
        want = oracle.head_sample(w, cond_bits, noise, t, idx)
        got = run_head(head, cond_bits, noise, t, idx)
        assert_parity(got, want, idx, f"K={K}")
    # reversed time direction
    t = np.array([1.0, 0.5, 0.0], np.float32)
    assert_parity(run_head(head, cond_bits, noise, t, idx), oracle.head_sample(w, cond_bits, noise, t, idx), idx)
    head.close()


def test_two_calls_on_one_head_give_identical_results():
    wl = synth.workload("cfg1", n=300)
    w, cond_bits, noise, t = synth.head_weights(wl), synth.cond(wl), synth.noise(wl), synth.t_sched(wl.K)
    head = make_head(wl, w)
    idx = np.arange(wl.n, dtype=np.int32)
    a = run_head(head, cond_bits, noise, t, idx)
    b = run_head(head, cond_bits, noise, t, idx)
    assert np.array_equal(a, b)
    head.close()


@pytest.mark.parametrize("name,runs,K", [("cfg2", 12, 4), ("cfg3", 4, 2)])
def test_full_size_runs_are_bit_identical(name, runs, K):
    """The kernel's arithmetic has a fixed order, so equal inputs must give equal bits however the
    items of the many CTAs interleave. A tile read before its producer's writes were visible (an
    ordering bug between CTAs) shows up here as a run that differs; the cache flush and the
    varying survivor counts in between change the timing from run to run."""
    dev = require_cuda()
    wl = synth.workload(name, K=K)
    w, t = synth.head_weights(wl), synth.t_sched(wl.K)
    cond, noise = dev_bf16(synth.cond(wl)), dev_f32(synth.noise(wl))
    head = make_head(wl, w)
    S = int(round(wl.n * (1 - wl.filter_q)))
    idx = torch.randperm(wl.n, device=dev, generator=torch.Generator(device=dev).manual_seed(3))[:S]
    idx = idx.sort().values.to(torch.int32).contiguous()
    count = torch.tensor([S], dtype=torch.int32, device=dev)
    flush = torch.empty(256 << 20, dtype=torch.uint8, device=dev)
    ref = None
    for r in range(runs):
        if r % 3 == 1:                                  # a different, smaller run in between
            c2 = torch.tensor([S // 2 + 7 * r], dtype=torch.int32, device=dev)
            scratch = torch.empty((wl.n, wl.C), dtype=torch.float32, device=dev)
            head.ardiff_head_sample(cond, noise, t, idx, c2, scratch)
        flush.fill_(r)
        out = torch.full((wl.n, wl.C), SENTINEL, dtype=torch.float32, device=dev)
        head.ardiff_head_sample(cond, noise, t, idx, count, out)
        assert head.status() == 0
        if ref is None:
            ref = out
        else:
            assert torch.equal(out, ref), f"run {r} differs from run 0"
    assert bool(torch.isfinite(ref[idx.long()]).all())
    head.close()


@pytest.mark.parametrize("W,n,few", [(1536, 300, (17, 23)), (256, 2000, (300, 1100)), (1024, 900, (200, 470)),
                                     (1024, 960, (700, 941)), (2048, 300, (100, 220))])
def test_few_token_runs_are_bit_identical(W, n, few):
    """The same for the chain (first) and the clusters (values copied between shared memories, and through L2): a flush, another
    call of the head and a busy second stream between and beside the runs."""
    dev = require_cuda()
    wl = synth.workload("cfg1", n=n, W=W, L=3, K=4, Dc=256)
    w, t = synth.head_weights(wl, std=None), synth.t_sched(wl.K)
    cond, noise = dev_bf16(synth.cond(wl)), dev_f32(synth.noise(wl))
    head = make_head(wl, w)
    chain, clusters = head.few_limits(wl.K)
    assert max(few) <= (chain if W == 1536 else clusters) and (W == 1536 or min(few) > chain)
    idx = torch.randperm(n, device=dev, generator=torch.Generator(device=dev).manual_seed(3)).to(torch.int32)
    counts = [torch.tensor([c], dtype=torch.int32, device=dev) for c in few]
    flush = torch.empty(256 << 20, dtype=torch.uint8, device=dev)
    busy = torch.randn(1 << 22, device=dev)
    side = torch.cuda.Stream(device=dev)
    ref = [None, None]
    for r in range(24):
        if r % 3 == 0:
            flush.fill_(r)
        if r % 4 == 1:
            side.wait_stream(torch.cuda.current_stream())
            with torch.cuda.stream(side):
                for _ in range(r):
                    busy = busy * 1.0001
        k = int(r % 5 in (1, 3))
        out = torch.full((n, wl.C), SENTINEL, dtype=torch.float32, device=dev)
        head.ardiff_head_sample(cond, noise, t, idx, counts[k], out)
        assert head.status() == 0
        if ref[k] is None:
            ref[k] = out
        assert torch.equal(out, ref[k]), f"run {r} with {few[k]} tokens differs"
    torch.cuda.synchronize()
    head.close()


@pytest.mark.parametrize("name,extra,K", [("cfg2", 160, None), ("cfg3", 48, None), ("cfg4", 32, None),
                                          ("cfg3", 24, 1), ("cfg3", 12, 8)])
def test_workload_configs_sampled_tokens(name, extra, K):
    """Full-size gate -> head run; the oracle checks one token of every token tile, the first, a middle
    and the last (ragged) token tile and random survivors one by one (tokens are independent). cfg 3
    also runs at the other step counts its workload names (K = 1 and 8)."""
    dev = require_cuda()
    wl = synth.workload(name) if K is None else synth.workload(name, K=K)
    feat_bits = synth.features(wl)
    H = oracle.entropy(feat_bits)
    Hs = np.sort(H)
    k = int(round(wl.filter_q * wl.n))
    tau = 0.5 * (Hs[k - 1] + Hs[k])
    w, cond_bits, noise, t = synth.head_weights(wl), synth.cond(wl), synth.noise(wl), synth.t_sched(wl.K)
    head = make_head(wl, w)
    mask, idx, count, _ = ardiff.ardiff_entropy_gate(dev_bf16(feat_bits), tau)
    out = torch.full(noise.shape, SENTINEL, dtype=torch.float32, device=dev)
    head.ardiff_head_sample(dev_bf16(cond_bits), dev_f32(noise), t, idx, count, out)
    assert head.status() == 0
    S = int(count.item())
    idx_h = idx.cpu().numpy()[:S]
    got = out.cpu().numpy()
    # Oracle-checked, element by element: one random token of EVERY token tile (an error confined to some
    # tiles, a group boundary or a scratch-slot reuse cannot hide), plus the whole first, one middle and the
    # last (ragged) tile and some random survivors. At the other step counts of cfg 3 the whole tiles are
    # thinned to keep the oracle's share of the run to seconds.
    rng = np.random.default_rng(11)
    tiles = (S + 127) // 128
    per_tile = np.minimum(np.arange(tiles) * 128 + rng.integers(0, 128, size=tiles), S - 1)
    whole = sample_tokens(idx_h, extra=extra)
    if K is not None:
        whole = whole[::4]
    pos = np.unique(np.concatenate([per_tile, whole]))
    toks = idx_h[pos]
    want = oracle.head_sample(w, cond_bits, noise, t, toks)

    def floor(rows):        # what bf16 rounding alone costs these tokens (CPU model, fp64)
        exact = rounding_model.head(w, cond_bits, noise, t, rows, rounded=())
        return rounding_model.error_ratio(rounding_model.head(w, cond_bits, noise, t, rows), exact)

    assert_head_parity(got, want, toks, name, model=floor)
    # properties that hold for every token: written iff kept, finite
    kept = np.zeros(wl.n, bool)
    kept[idx_h] = True
    assert np.all(got[~kept] == SENTINEL)
    assert np.all(np.isfinite(got[kept])) and not np.any(got[kept] == SENTINEL)
    head.close()


def test_two_heads_on_two_streams():
    """Two heads of different shapes, driven from two streams without any ordering between them: every
    launch needs the whole GPU (cooperative launch), so the launches take turns; both results must
    match what each head gives alone."""
    dev = require_cuda()
    wa, wb = synth.workload("cfg1", n=700), synth.workload("cfg1", n=900, W=512, L=3, seed=77)
    outs = {}
    heads = {}
    for key, wl in (("a", wa), ("b", wb)):
        w, t = synth.head_weights(wl), synth.t_sched(wl.K)
        head = make_head(wl, w)
        cond, noise = dev_bf16(synth.cond(wl)), dev_f32(synth.noise(wl))
        idx = torch.arange(wl.n, dtype=torch.int32, device=dev)
        count = torch.tensor([wl.n], dtype=torch.int32, device=dev)
        alone = torch.empty((wl.n, wl.C), dtype=torch.float32, device=dev)
        head.ardiff_head_sample(cond, noise, t, idx, count, alone)
        heads[key] = (head, cond, noise, t, idx, count, alone, wl)
    torch.cuda.synchronize()
    streams = {k: torch.cuda.Stream(device=dev) for k in heads}
    for rep in range(4):
        for key, (head, cond, noise, t, idx, count, alone, wl) in heads.items():
            out = torch.full((wl.n, wl.C), SENTINEL, dtype=torch.float32, device=dev)
            head.ardiff_head_sample(cond, noise, t, idx, count, out, stream=streams[key])
            outs[(key, rep)] = out
    torch.cuda.synchronize()
    for (key, rep), out in outs.items():
        head, *_, alone, wl = heads[key]
        assert head.status() == 0
        assert torch.equal(out, alone), (key, rep)
    for head, *_ in heads.values():
        head.close()


@pytest.mark.parametrize("na,nb", [(4900, 2300), (4900, 900)])
def test_two_heads_on_two_streams_with_tiles(na, nb):
    """The same with tiles, and with one head of tiles beside one of clusters."""
    dev = require_cuda()
    wa, wb = synth.workload("cfg1", n=na), synth.workload("cfg1", n=nb, W=512, L=3, seed=77)
    outs = {}
    heads = {}
    for key, wl in (("a", wa), ("b", wb)):
        w, t = synth.head_weights(wl), synth.t_sched(wl.K)
        head = make_head(wl, w)
        cond, noise = dev_bf16(synth.cond(wl)), dev_f32(synth.noise(wl))
        idx = torch.arange(wl.n, dtype=torch.int32, device=dev)
        count = torch.tensor([wl.n], dtype=torch.int32, device=dev)
        alone = torch.empty((wl.n, wl.C), dtype=torch.float32, device=dev)
        head.ardiff_head_sample(cond, noise, t, idx, count, alone)
        heads[key] = (head, cond, noise, t, idx, count, alone, wl)
        assert (head.few_limits(wl.K)[1] < wl.n) == (wl.n > 1000)
    torch.cuda.synchronize()
    streams = {k: torch.cuda.Stream(device=dev) for k in heads}
    for rep in range(4):
        for key, (head, cond, noise, t, idx, count, alone, wl) in heads.items():
            out = torch.full((wl.n, wl.C), SENTINEL, dtype=torch.float32, device=dev)
            head.ardiff_head_sample(cond, noise, t, idx, count, out, stream=streams[key])
            outs[(key, rep)] = out
    torch.cuda.synchronize()
    for (key, rep), out in outs.items():
        head, *_, alone, wl = heads[key]
        assert head.status() == 0
        assert torch.equal(out, alone), (key, rep)
    for head, *_ in heads.values():
        head.close()


def test_bad_arguments_are_rejected():
    require_cuda()
    wl = synth.workload("cfg1")
    w = synth.head_weights(wl)
    with pytest.raises(ardiff.ArdiffError):
        ardiff.Head(wl.C, wl.Dc, 250, wl.L, wl.F, 4, 64, w)          # W not a multiple of 256
    with pytest.raises(ardiff.ArdiffError):
        ardiff.Head(8, wl.Dc, wl.W, wl.L, wl.F, 4, 64, w)            # C too small
    head = make_head(wl, w)
    lib = ardiff.lib()
    buf = torch.zeros(1 << 16, dtype=torch.uint8, device="cuda")
    p = buf.data_ptr()
    t = synth.t_sched(4)
    assert lib.ardiff_head_sample(head._h, p, p, t.ctypes.data, 5, p, p, p, None) == ardiff.ARDIFF_ERR_SHAPE
    assert lib.ardiff_head_sample(head._h, p, p, t.ctypes.data, 4, None, p, p, None) == ardiff.ARDIFF_ERR_NULL
    assert lib.ardiff_head_sample(head._h, p + 2, p, t.ctypes.data, 4, p, p, p, None) == ardiff.ARDIFF_ERR_ALIGN
    head.close()


def ddim_coef(abar):
    """Deterministic eps-prediction steps along abar[0] -> abar[1] -> ... (coefficients of x and eps)."""
    abar = np.asarray(abar, np.float64)
    ax = np.sqrt(abar[1:] / abar[:-1])
    av = np.sqrt(1 - abar[1:]) - ax * np.sqrt(1 - abar[:-1])
    return np.stack([ax, av, np.zeros_like(ax)], axis=1).astype(np.float32)


@pytest.mark.parametrize("sampler", ["euler", "ddim", "x0_renoise"])
def test_linear_sampler_steps(sampler):
    """Other samplers on the same head: every step is x <- ax x + av v + an z_k."""
    dev = require_cuda()
    wl = synth.workload("cfg1", n=300, K=4)
    # all three on the harder 1/sqrt(fan_in) weights (every layer keeps unit scale, nothing damps an error)
    w = synth.head_weights(wl, std=None)
    cond_bits, noise = synth.cond(wl), synth.noise(wl)
    idx_np = np.random.default_rng(7).permutation(wl.n)[:211].astype(np.int32)
    z = None
    if sampler == "euler":
        t = np.array([0.0, 0.2, 0.5, 0.9, 1.0], np.float32)
        t_in = t[:-1]
        coef = np.stack([np.ones(4), t[1:].astype(np.float64) - t[:-1].astype(np.float64), np.zeros(4)], 1).astype(np.float32)
    elif sampler == "ddim":
        t_in = np.array([0.95, 0.7, 0.45, 0.2], np.float32)
        coef = ddim_coef([0.05, 0.3, 0.6, 0.85, 0.999])
    else:
        # two-step consistency sampling: predict x0, re-noise to abar = 0.5, predict x0 again. The output
        # is the head's last raw prediction (ax = 0 discards the state), so nothing props up its RMS.
        t_in = np.array([0.95, 0.5], np.float32)
        abn = np.array([0.5, 1.0])
        coef = np.stack([np.zeros(2), np.sqrt(abn), np.sqrt(1 - abn)], 1).astype(np.float32)
        z = np.random.default_rng(8).standard_normal((2, wl.n, wl.C)).astype(np.float32)
    want = oracle.head_sample_coef(w, cond_bits, noise, t_in, coef, idx_np, step_noise=z)
    head = make_head(wl, w)
    idx = torch.from_numpy(idx_np).to(dev)
    count = torch.tensor([len(idx_np)], dtype=torch.int32, device=dev)
    out = torch.full(noise.shape, SENTINEL, dtype=torch.float32, device=dev)
    head.ardiff_head_sample_coef(dev_bf16(cond_bits), dev_f32(noise), t_in, coef, idx, count, out,
                                 step_noise=None if z is None else torch.from_numpy(z).to(dev))
    assert head.status() == 0
    got = out.cpu().numpy()
    assert_parity(got, want, idx_np, sampler)
    assert np.all(got[np.setdiff1d(np.arange(wl.n), idx_np)] == SENTINEL)
    if sampler == "euler":                 # the Euler entry point is this call with the Euler coefficients
        got2 = run_head(head, cond_bits, noise, np.array([0.0, 0.2, 0.5, 0.9, 1.0], np.float32), idx_np)
        assert np.array_equal(got2[idx_np], got[idx_np])
    head.close()


@pytest.mark.parametrize("shape", [dict(W=4096, L=1, K=1, C=32, Dc=64, n=130),
                                   dict(W=2048, L=2, K=2, C=64, Dc=128, n=300),
                                   dict(W=256, L=5, K=3, C=48, Dc=1024, n=257),
                                   dict(W=512, L=1, K=64, C=16, Dc=64, n=40),
                                   dict(W=256, L=64, K=1, C=16, Dc=64, n=130),
                                   dict(W=512, L=2, K=2, C=16, Dc=128, F=1024, n=200),
                                   dict(W=256, L=2, K=3, C=32, Dc=64, F=2, n=129)])
def test_extreme_shapes(shape):
    """Widest head (16 column tiles, 32 LayerNorm partials per row), the largest token dim, an odd number
    of blocks (gate buffers alternate by block parity), the largest step count, the deepest head (64 blocks),
    the largest and the smallest time-embedding size."""
    n = shape.pop("n")
    wl = synth.workload("cfg1", n=n, **shape)
    w, cond_bits, noise, t = synth.head_weights(wl), synth.cond(wl), synth.noise(wl), synth.t_sched(wl.K)
    idx = np.arange(n, dtype=np.int32)
    want = oracle.head_sample(w, cond_bits, noise, t, idx)
    head = make_head(wl, w)
    got = run_head(head, cond_bits, noise, t, idx)
    assert_parity(got, want, idx, str(shape))
    head.close()


@pytest.mark.parametrize("shape", [dict(W=256, L=5, K=3, C=48, Dc=1024, n=4800), dict(W=512, L=1, K=64, C=16, Dc=64, n=420),
                                   dict(W=256, L=64, K=1, C=16, Dc=64, n=1500), dict(W=512, L=2, K=2, C=16, Dc=128, F=1024, n=2200)])
def test_extreme_shapes_beyond_the_clusters(shape):
    """The same with more tokens than the clusters serve: an odd number of blocks, the largest step count, the deepest head, the
    largest time embedding with the tiles. The oracle takes some tokens of the first, a middle and the last token tile."""
    shape = dict(shape)
    n = shape.pop("n")
    wl = synth.workload("cfg1", n=n, **shape)
    w, cond_bits, noise, t = synth.head_weights(wl), synth.cond(wl), synth.noise(wl), synth.t_sched(wl.K)
    idx = np.arange(n, dtype=np.int32)
    rows = sample_tokens(idx, extra=16)[::5]
    want = oracle.head_sample(w, cond_bits, noise, t, rows)
    head = make_head(wl, w)
    assert head.few_limits(wl.K)[1] < n
    assert_parity(run_head(head, cond_bits, noise, t, idx), want, rows, str(shape))
    head.close()


def test_bounded_wait_runs_out_reports_timeout_and_the_head_recovers():
    """The self-test hook makes one tile's dependency wait unsatisfiable and shortens the wait limit to 3 ms:
    the kernel must come back by itself (no fault, no trap, no endless spin), the status word must say
    TIMEOUT, and the very next call on the same head must give the bits of an undisturbed run."""
    wl = synth.workload("cfg1", n=900)
    w, cond_bits, noise, t = synth.head_weights(wl), synth.cond(wl), synth.noise(wl), synth.t_sched(wl.K)
    idx = np.arange(wl.n, dtype=np.int32)
    head = make_head(wl, w)
    clean = run_head(head, cond_bits, noise, t, idx)
    for tile in (0, 3, 7):                                # first, an odd (partner CTA) and the last, ragged tile
        head.inject_stall(tile, 3000)
        dev = require_cuda()
        out = torch.zeros(noise.shape, dtype=torch.float32, device=dev)
        head.ardiff_head_sample(dev_bf16(cond_bits), dev_f32(noise), t, torch.from_numpy(idx).to(dev),
                                torch.tensor([wl.n], dtype=torch.int32, device=dev), out)
        assert head.status() == ardiff.ARDIFF_ERR_TIMEOUT
        assert head.status() == 0                         # reading the status clears it
        assert np.array_equal(run_head(head, cond_bits, noise, t, idx), clean)
    head.inject_stall(4000, 3000)                         # a tile this call does not have: no effect
    assert np.array_equal(run_head(head, cond_bits, noise, t, idx), clean)
    fresh = make_head(wl, w)
    assert np.array_equal(run_head(fresh, cond_bits, noise, t, idx), clean)
    with pytest.raises(ardiff.ArdiffError):
        head.inject_stall(0, 5)                           # limit below 100 us
    fresh.close()
    head.close()


def test_a_wait_of_the_tile_schedule_runs_out():
    """The same with more tokens than the clusters serve: waits of gathers, products, epilogues and of the drained rings. The first
    tile, an odd one (partner CTA) and the last."""
    dev = require_cuda()
    wl = synth.workload("cfg1", n=5000)
    w, cond_bits, noise, t = synth.head_weights(wl), synth.cond(wl), synth.noise(wl), synth.t_sched(wl.K)
    idx = np.arange(wl.n, dtype=np.int32)
    head = make_head(wl, w)
    assert head.few_limits(wl.K)[1] < wl.n
    clean = run_head(head, cond_bits, noise, t, idx)
    for tile in (0, 3, 39):
        head.inject_stall(tile, 3000)
        out = torch.zeros(noise.shape, dtype=torch.float32, device=dev)
        head.ardiff_head_sample(dev_bf16(cond_bits), dev_f32(noise), t, torch.from_numpy(idx).to(dev),
                                torch.tensor([wl.n], dtype=torch.int32, device=dev), out)
        assert head.status() == ardiff.ARDIFF_ERR_TIMEOUT
        assert head.status() == 0
        assert np.array_equal(run_head(head, cond_bits, noise, t, idx), clean)
    head.close()


@pytest.mark.parametrize("W,n", [(256, 500), (1024, 64), (1024, 500), (1536, 200), (2048, 200)])
def test_a_wait_inside_the_clusters_runs_out(W, n):
    """One CTA of the first, or of a later, cluster stops between two layers (values copied between shared memories at the first two
    sizes, through L2 at the others): its peers' waits end at the limit, the status says TIMEOUT, and the next call gives the
    bits of an undisturbed run. A cluster that the call does not need: no effect."""
    dev = require_cuda()
    wl = synth.workload("cfg1", n=n, W=W, L=2, K=2, Dc=128)
    w, cond_bits, noise, t = synth.head_weights(wl), synth.cond(wl), synth.noise(wl), synth.t_sched(wl.K)
    idx = np.arange(n, dtype=np.int32)
    head = make_head(wl, w)
    chain, clusters = head.few_limits(wl.K)
    assert chain < n <= clusters
    clean = run_head(head, cond_bits, noise, t, idx)
    for cluster in (0, 3):
        head.inject_cluster_stall(cluster, 3000)
        out = torch.zeros(noise.shape, dtype=torch.float32, device=dev)
        head.ardiff_head_sample(dev_bf16(cond_bits), dev_f32(noise), t, torch.from_numpy(idx).to(dev),
                                torch.tensor([n], dtype=torch.int32, device=dev), out)
        assert head.status() == ardiff.ARDIFF_ERR_TIMEOUT
        assert np.array_equal(run_head(head, cond_bits, noise, t, idx), clean)
    head.inject_cluster_stall(400, 3000)
    assert np.array_equal(run_head(head, cond_bits, noise, t, idx), clean)
    head.close()


def test_more_survivors_than_the_head_was_created_for():
    """*count above max_tokens: the head runs the first max_tokens survivors, leaves every other row
    untouched and flags the call with ARDIFF_ERR_SHAPE in its status word; the next call is clean."""
    dev = require_cuda()
    wl = synth.workload("cfg1", n=400)
    w, cond_bits, noise, t = synth.head_weights(wl), synth.cond(wl), synth.noise(wl), synth.t_sched(wl.K)
    head = make_head(wl, w, max_tokens=256)
    idx_np = np.random.default_rng(2).permutation(wl.n)[:300].astype(np.int32)
    want = oracle.head_sample(w, cond_bits, noise, t, idx_np[:256])
    idx = torch.from_numpy(idx_np).to(dev)
    count = torch.tensor([300], dtype=torch.int32, device=dev)
    out = torch.full(noise.shape, SENTINEL, dtype=torch.float32, device=dev)
    head.ardiff_head_sample(dev_bf16(cond_bits), dev_f32(noise), t, idx, count, out)
    assert head.status() == ardiff.ARDIFF_ERR_SHAPE
    got = out.cpu().numpy()
    assert_parity(got, want, idx_np[:256])
    assert np.all(got[np.setdiff1d(np.arange(wl.n), idx_np[:256])] == SENTINEL)
    assert np.array_equal(run_head(head, cond_bits, noise, t, idx_np[:200])[idx_np[:200]], got[idx_np[:200]])
    head.close()


def test_persisting_l2_is_set_aside_while_a_head_exists_and_put_back_after():
    # include/ardiff.h, ardiff_head_create: the context's persisting-L2 limit covers one token group's fp32
    # residual stream while heads exist on the device, and returns to what it was with the last of them
    rt = pytest.importorskip("cuda.bindings.runtime")
    require_cuda()

    def limit():
        err, v = rt.cudaDeviceGetLimit(rt.cudaLimit.cudaLimitPersistingL2CacheSize)
        assert int(err) == 0
        return int(v)

    err, max_size = rt.cudaDeviceGetAttribute(rt.cudaDeviceAttr.cudaDevAttrMaxPersistingL2CacheSize, 0)
    assert int(err) == 0
    if max_size <= 0:
        pytest.skip("device has no persisting L2")
    wl = synth.workload("cfg1")
    weights = synth.head_weights(wl)
    before = limit()
    h1 = make_head(wl, weights)
    during = limit()
    group_h_bytes = 2 * 128 * wl.W * 4          # cfg1: one pair of token tiles per group
    assert during >= min(group_h_bytes, max_size) and during >= before
    h2 = make_head(wl, weights)
    h1.close()
    assert limit() == during
    h2.close()
    assert limit() == before
