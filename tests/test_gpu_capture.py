"""Gate calls inside a stream capture after one call outside it.

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
