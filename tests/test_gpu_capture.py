"""Gate and head calls inside a stream capture after one call outside it.

One call of an entry point on a device loads all its row kernels (which takes device memory): calls of any other width and
number of rows take none and may be captured. Each case runs in a fresh process, where no kernel has been loaded before that call.
"""
import subprocess
import sys
import textwrap

import pytest

from conftest import ROOT
from gpu_util import require_cuda

pytestmark = pytest.mark.gpu

CHILD = """
    import sys
    import torch
    import paper_2512_08537_b200 as ardiff
    kind, first = sys.argv[1], int(sys.argv[2])
    dev = torch.device("cuda:0")
    shapes = [(n, d) for d in (8, 40, 64, 100, 128, 200, 256, 300, 512, 700, 768, 777, 1000, 1024, 1500, 2048, 2500, 3072, 4096,
                               4099, 5120, 6000, 6144, 7001, 8192, 8200, 9001, 16384) for n in (50, 6000)]
    gen = torch.Generator(device=dev).manual_seed(1)
    x = torch.randn(6000 * 16384, device=dev, generator=gen).to(torch.bfloat16)
    mask = torch.zeros(6000, dtype=torch.uint8, device=dev)
    idx = torch.zeros(6000, dtype=torch.int32, device=dev)
    count = torch.zeros(1, dtype=torch.int32, device=dev)
    keep = []
    def call(n, d):
        feat = x[: n * d].view(n, d)
        if kind == "noalloc":
            ardiff.ardiff_entropy_gate_noalloc(feat, 2.0, mask[:n], idx[:n], count)
        elif kind == "gate":
            ardiff.ardiff_entropy_gate(feat, 2.0, mask[:n], idx[:n], count)
        else:
            keep.append(ardiff.ardiff_entropy_gate_blocks(feat, 1, 5, 2.0))
    call(64, first)
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    free = torch.cuda.mem_get_info()[0]
    if kind != "blocks":                      # (the block form's wrapper allocates its outputs)
        for n, d in shapes:
            call(n, d)
        torch.cuda.synchronize()
    lost = free - torch.cuda.mem_get_info()[0]
    side = torch.cuda.Stream()
    for n, d in shapes:
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=side):
            call(n, d)
        graph.replay()
        torch.cuda.synchronize()
    print("captured", len(shapes), "driver bytes", lost)
    assert lost <= 0, lost
"""


@pytest.mark.parametrize("kind", ["noalloc", "gate", "blocks"])
@pytest.mark.parametrize("first", [256, 777])
def test_any_width_can_be_captured_after_one_call(kind, first):
    require_cuda()
    r = subprocess.run([sys.executable, "-c", textwrap.dedent(CHILD), kind, str(first)], cwd=ROOT, timeout=300,
                       capture_output=True, text=True)
    print(r.stdout[-500:])
    assert r.returncode == 0, r.stdout[-1000:] + r.stderr[-1500:]


@pytest.mark.parametrize("W,counts", [(256, (300, 33, 4900)), (1536, (20, 200, 1000)), (2304, (60, 700))])
def test_a_captured_head_call_follows_the_count(W, counts):
    """One captured head call, its launches over the one before included, replayed with the count of every schedule in turn
    (clusters, chain at W = 1536, tiles): the bits of eager calls, and again after them."""
    import numpy as np
    import torch
    import synth
    import paper_2512_08537_b200 as ardiff
    dev = require_cuda()
    wl = synth.workload("cfg1", n=max(counts), W=W, L=2, K=2, Dc=128)
    head = ardiff.Head(wl.C, wl.Dc, wl.W, wl.L, wl.F, wl.K, wl.n, synth.head_weights(wl))
    chain, clusters = head.few_limits(wl.K)
    assert clusters < max(counts) and (W > 2048 or sorted(counts)[-2] > chain) and (W != 1536 or min(counts) <= chain)
    gen = torch.Generator(device=dev).manual_seed(2)
    cond = torch.randn((wl.n, wl.Dc), device=dev, generator=gen).to(torch.bfloat16)
    noise = torch.randn((wl.n, wl.C), device=dev, generator=gen)
    idx = torch.randperm(wl.n, device=dev, generator=gen).to(torch.int32)
    count, out, t = torch.zeros(1, dtype=torch.int32, device=dev), torch.zeros_like(noise), synth.t_sched(wl.K)

    def run(call, c):
        count.fill_(c)
        out.fill_(-5.0)
        call()
        assert head.status() == 0
        return out.cpu().numpy()

    def eager():
        head.ardiff_head_sample(cond, noise, t, idx, count, out)

    want = {c: run(eager, c) for c in counts}
    graph, side = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph, stream=side):
        eager()
    for c in counts + counts[::-1]:
        assert np.array_equal(run(graph.replay, c), want[c]), c
    assert np.array_equal(run(eager, counts[0]), want[counts[0]])
    del graph
    head.close()
