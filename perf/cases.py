"""What is timed of this framework: passes through its public calls at the sizes they are used at.

A case is a dict of plain values; `listed()` names the fixed ones, `draw()` gives more of the same ranges. `prepare()`
makes what a program holds before the call (device tensors, a head with its weights, a host-buffer pipeline) and
`run()` makes one pass. Shapes are those of the repository's workload table and benchmark, or lie between them:

  tiny   token dim 16, conditioning  256, width  256,  2 blocks
  class  token dim 16, conditioning  768, width 1024,  3 blocks   (class-conditional 16x16 latent grids)
  deep   token dim 16, conditioning 1024, width 1536,  6 blocks
  text   token dim 64, conditioning 5120, width 1536, 12 blocks   (text-conditioned 32x32 latent grids)

Kinds of pass:
  path       entropy gate, compaction, K Euler steps of the head over the survivors (device tensors)
  sampler    the same with a re-noising x0-prediction sampler (per-step coefficients and fresh noise)
  gate       entropy gate and compaction alone, entropies asked for
  blocks     block-prefix gate over attention-map rows, then the accepted length of every draft block
  calibrate  threshold statistics of one batch, and the threshold of a pool of entropies gathered before
  host       batches in pinned host memory through the host-buffer pipeline (copies included)
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2512_08537_b200 as ardiff

TIME_FEATURES = 256
HEADS = {
    "tiny": dict(C=16, Dc=256, W=256, L=2),
    "class": dict(C=16, Dc=768, W=1024, L=3),
    "deep": dict(C=16, Dc=1024, W=1536, L=6),
    "text": dict(C=64, Dc=5120, W=1536, L=12),
}
# the most that one drawn pass may cost: the survivors of the largest listed head pass, the rows of the largest gate pass
MAX_FLOPS = 27.2e12
MAX_BYTES = 10.7e9


def listed():
    return [
        # the smallest call: one short draft of the smallest head; launches and latency are all there is
        dict(name="path_64_tiny", kind="path", n=64, d=256, **HEADS["tiny"], K=4, drop=0.5, heavy=False),
        # speculative decoding of five prompts, a draft block of 8 tokens each, with the largest head
        dict(name="path_40_text", kind="path", n=40, d=5120, **HEADS["text"], K=4, drop=0.3, heavy=True),
        # a handful of images in flight, ragged: what a lightly loaded server sees
        dict(name="path_1000_class", kind="path", n=1000, d=768, **HEADS["class"], K=4, drop=0.3, heavy=False),
        # batch 64 of 16x16 grids
        dict(name="path_16384_class", kind="path", n=16384, d=768, **HEADS["class"], K=4, drop=0.3, heavy=False),
        # batch 32 of 32x32 grids with the largest head: the flagship batch
        dict(name="path_32768_text", kind="path", n=32768, d=5120, **HEADS["text"], K=4, drop=0.3, heavy=True),
        # two-step consistency sampling with re-noising, odd batch
        dict(name="sampler_9001_deep", kind="sampler", n=9001, d=1024, **HEADS["deep"], K=2, drop=0.4, heavy=False),
        # the gate's stress size: a million wide rows, the largest read
        dict(name="gate_1048576_5120", kind="gate", n=1 << 20, d=5120, drop=0.5, heavy=True),
        # a feature width that is no multiple of 8, so rows start at any even address
        dict(name="gate_65536_777", kind="gate", n=65536, d=777, drop=0.4, heavy=True),
        # attention-map rows (16 per token, 1024 keys) in draft blocks of 8, then the accepted lengths
        dict(name="blocks_4096x16x1024", kind="blocks", n=4096, rows=16, d=1024, gamma=8, drop=0.05, heavy=False),
        # threshold calibration on codebook-sized rows and a pool of a million entropies
        dict(name="calibrate_8192_16384", kind="calibrate", n=8192, d=16384, pool=1 << 20, heavy=True),
        # one batch from host memory, blocking
        dict(name="host_16384_class", kind="host", n=16384, d=768, **HEADS["class"], K=4, drop=0.3, heavy=False,
             slots=1, batches=1),
        # a stream of small batches from host memory, overlapped over three staging slots
        dict(name="host_6x2048_class", kind="host", n=2048, d=768, **HEADS["class"], K=4, drop=0.3, heavy=False,
             slots=3, batches=6),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _width(rng, lo, hi):
    """A row width: mostly a multiple of 8 (vectorisable rows), a quarter of the time any number."""
    d = _log(rng, lo, hi)
    return d if rng.random() < 0.25 else max(8, d // 8 * 8)


def _head(rng):
    if rng.random() < 0.5:
        return dict(HEADS[rng.choice(sorted(HEADS))])
    return dict(C=rng.choice([16, 32, 48, 64]), Dc=64 * _log(rng, 4, 80), W=256 * rng.randint(1, 8),
                L=rng.randint(1, 12))


def draw(rng):
    kind = rng.choice(["path", "path", "path", "sampler", "gate", "gate", "blocks", "calibrate", "host"])
    heavy = rng.random() < 0.5
    if kind in ("path", "sampler", "host"):
        c = dict(kind=kind, n=_log(rng, 8, 65536), d=_width(rng, 256, 5120), **_head(rng), K=rng.choice([1, 2, 4, 8]),
                 drop=rng.choice([0.0, 0.1, 0.3, 0.4, 0.5, 0.9]), heavy=heavy)
        if kind == "host":
            c["slots"] = rng.choice([1, 3])
            c["batches"] = 1 if c["slots"] == 1 else rng.randint(3, 8)
            c["n"] = min(c["n"], 16384)
        per_token = _survivors(c) / c["n"] * _flops_per_token(c) * c.get("batches", 1)
        c["n"] = max(8, min(c["n"], int(MAX_FLOPS / per_token)))
        return c
    if kind == "gate":
        c = dict(kind=kind, n=_log(rng, 64, 1 << 20), d=_width(rng, 64, 16384),
                 drop=rng.choice([0.0, 0.1, 0.5, 0.9, 0.99]), heavy=heavy)
        c["n"] = max(1, min(c["n"], int(MAX_BYTES / (2 * c["d"] + 9))))
        return c
    if kind == "blocks":
        c = dict(kind=kind, n=_log(rng, 64, 65536), rows=_log(rng, 1, 32), d=_width(rng, 64, 4096),
                 gamma=rng.randint(2, 16), drop=rng.choice([0.02, 0.05, 0.1]), heavy=heavy)
        c["n"] = max(16, min(c["n"], int(MAX_BYTES / (2 * c["d"] * c["rows"] + 30))))
        return c
    c = dict(kind=kind, n=_log(rng, 64, 65536), d=_width(rng, 256, 16384), pool=_log(rng, 1024, 1 << 20), heavy=heavy)
    c["n"] = max(64, min(c["n"], int(MAX_BYTES / 4 / (2 * c["d"] + 9))))
    return c


# ---- inputs -------------------------------------------------------------------------------------
def _features(n, d, heavy, gen):
    """bf16 [n, d]: flat N(0,1) rows mixed 70 : 30 with peaked ones (one channel at 20 |x|), or heavy-tailed
    (Student-t, 3 degrees of freedom) rows mixed 70 : 30 with peaked ones."""
    dev = gen.device
    feat = torch.empty((n, d), dtype=torch.bfloat16, device=dev)
    step = max(1, (1 << 26) // d)
    for r0 in range(0, n, step):
        m = min(step, n - r0)
        x = torch.randn((m, d), device=dev, generator=gen)
        peaked = torch.rand((m, 1), device=dev, generator=gen) < 0.3
        if heavy:
            chi = torch.randn((m, d), device=dev, generator=gen).square_()
            chi -= 2.0 * torch.rand((m, d), device=dev, generator=gen).clamp_(min=1e-30).log_()
            x = torch.where(peaked, x, x / (chi / 3.0).sqrt_())
        col = torch.randint(0, d, (m, 1), device=dev, generator=gen)
        at = x.gather(1, col)
        x.scatter_(1, col, torch.where(peaked, 20.0 * at.abs(), at))
        feat[r0:r0 + m] = x
    return feat


def _entropies(feat, rows_per_token=1):
    """Indicator of up to 4096 tokens of the batch in fp64 (mean over each token's rows), ascending."""
    n, d = feat.shape[0] // rows_per_token, feat.shape[1]
    m = max(1, min(n, 4096, (1 << 24) // (d * rows_per_token)))
    tok = torch.arange(m, device=feat.device) * n // m
    rows = (tok[:, None] * rows_per_token + torch.arange(rows_per_token, device=feat.device)).reshape(-1)
    lp = torch.log_softmax(feat[rows].double(), dim=1)
    h = -(lp.exp() * lp).sum(dim=1).reshape(m, rows_per_token).mean(dim=1)
    return h.sort().values.cpu().numpy()


def _threshold(h, drop):
    """The threshold that drops about this share: the middle of the widest gap near the quantile, so that no token's
    decision hangs on the last bit of its entropy."""
    if drop <= 0.0:
        return -1.0
    k = min(max(1, int(round(drop * len(h)))), len(h) - 1)
    w = len(h) // 25
    lo, hi = max(0, k - 1 - w), min(len(h) - 1, k + w)
    if hi <= lo:
        return float(h[0]) - 1e-3
    g = lo + int(np.argmax(np.diff(h[lo:hi + 1])))
    return 0.5 * float(h[g] + h[g + 1])


def _weights(case, gen):
    """bf16 bit patterns of a head's parameters, N(0, 0.02), as host arrays (what a checkpoint loads into)."""
    C, Dc, W, L, F = case["C"], case["Dc"], case["W"], case["L"], TIME_FEATURES
    shapes = {"Wc": (W, Dc), "bc": (W,), "Wt1": (W, F), "bt1": (W,), "Wt2": (W, W), "bt2": (W,), "Win": (W, C),
              "bin": (W,), "Wmod": (L, 3 * W, W), "bmod": (L, 3 * W), "W1": (L, W, W), "b1": (L, W), "W2": (L, W, W),
              "b2": (L, W), "Wfm": (2 * W, W), "bfm": (2 * W,), "Wout": (C, W), "bout": (C,)}
    out = {}
    for name, shape in shapes.items():
        w = torch.empty(shape, device=gen.device).normal_(0.0, 0.02, generator=gen).to(torch.bfloat16)
        out[name] = w.view(torch.int16).cpu().numpy().view(np.uint16)
    return out


class _State:
    pass


def _inputs(case, seed):
    """The state of a pass without its handles, and the head's weights (None where the path has no head)."""
    dev = torch.device("cuda")
    gen = torch.Generator(device=dev).manual_seed(seed)
    s, kind, n = _State(), case["kind"], case["n"]
    s.kind = kind
    if kind == "host":
        return s, _host_inputs(s, case, gen)
    s.feat = _features(n * case.get("rows", 1), case["d"], case["heavy"], gen)
    if kind == "calibrate":
        s.pool = torch.empty(case["pool"], device=dev).uniform_(0.0, math.log(case["d"]), generator=gen)
        return s, None
    s.tau = _threshold(_entropies(s.feat, case.get("rows", 1)), case["drop"])
    if kind == "blocks":
        s.rows, s.gamma = case["rows"], case["gamma"]
        s.r = torch.rand(n, device=dev, generator=gen)
        s.ratio = 0.5 + torch.rand(n, device=dev, generator=gen)
        return s, None
    s.mask = torch.zeros(n, dtype=torch.uint8, device=dev)
    s.idx = torch.zeros(n, dtype=torch.int32, device=dev)
    s.count = torch.zeros(1, dtype=torch.int32, device=dev)
    if kind == "gate":
        s.entropy = torch.zeros(n, device=dev)
        return s, None
    K = case["K"]
    s.cond = torch.randn((n, case["Dc"]), device=dev, generator=gen).to(torch.bfloat16)
    s.noise = torch.randn((n, case["C"]), device=dev, generator=gen)
    s.out = torch.zeros((n, case["C"]), device=dev)       # rows of dropped tokens are left as they are
    weights = _weights(case, gen)
    if kind == "path":
        s.t = np.arange(K + 1, dtype=np.float32) / K
    else:
        # predict x0, re-noise to the next level, ... ; the last step returns the prediction
        s.t = 1.0 - np.arange(K, dtype=np.float32) / K
        keep = (np.arange(K) + 1.0) / K
        s.coef = np.stack([np.zeros(K), np.sqrt(keep), np.sqrt(1.0 - keep)], axis=1).astype(np.float32)
        s.step_noise = torch.randn((K, n, case["C"]), device=dev, generator=gen)
    return s, weights


def _host_inputs(s, case, gen):
    n, K = case["n"], case["K"]
    s.slots, s.batches = case["slots"], []
    for _ in range(case["batches"]):
        feat = _features(n, case["d"], case["heavy"], gen)
        tau = _threshold(_entropies(feat), case["drop"])
        cond = torch.randn((n, case["Dc"]), device=gen.device, generator=gen).to(torch.bfloat16)
        noise = torch.randn((n, case["C"]), device=gen.device, generator=gen)
        s.batches.append(dict(feat=feat.cpu().pin_memory(), cond=cond.cpu().pin_memory(),
                              noise=noise.cpu().pin_memory(), tau=tau, out=torch.zeros((n, case["C"])).pin_memory(),
                              mask=torch.zeros(n, dtype=torch.uint8).pin_memory()))
    s.t = np.arange(K + 1, dtype=np.float32) / K
    return _weights(case, gen)


def prepare(case, seed):
    s, weights = _inputs(case, seed)
    if weights is not None:
        s.head = ardiff.Head(case["C"], case["Dc"], case["W"], case["L"], TIME_FEATURES, case["K"], case["n"], weights)
    if s.kind == "host":
        s.pipe = ardiff.Pipeline(s.head, case["n"], case["d"], slots=s.slots)
    return s


# ---- one pass -----------------------------------------------------------------------------------
def run(s):
    if s.kind == "host":
        return _run_host(s)
    if s.kind == "calibrate":
        mask, idx, count, entropy, tau3 = ardiff.ardiff_entropy_gate_stats(s.feat, want_entropy=True)
        return [mask, idx, count, entropy, tau3, ardiff.ardiff_tau_calibrate(s.pool)]
    if s.kind == "blocks":
        # the ids behind *count in idx are unspecified and idx is fresh on every call: the mask says the same
        mask, idx, count, block_len, _, indicator = ardiff.ardiff_entropy_gate_blocks(
            s.feat, s.rows, s.gamma, s.tau, want_token_entropy=True)
        return [mask, count, block_len, indicator, ardiff.ardiff_accept_prefix(s.r, s.ratio, s.gamma, block_len)]
    if s.kind == "gate":
        ardiff.ardiff_entropy_gate(s.feat, s.tau, s.mask, s.idx, s.count, s.entropy)
        return [s.mask, s.idx, s.count, s.entropy]
    ardiff.ardiff_entropy_gate(s.feat, s.tau, s.mask, s.idx, s.count)
    if s.kind == "path":
        s.head.ardiff_head_sample(s.cond, s.noise, s.t, s.idx, s.count, s.out)
    else:
        s.head.ardiff_head_sample_coef(s.cond, s.noise, s.t, s.coef, s.idx, s.count, s.out, step_noise=s.step_noise)
    return [s.mask, s.idx, s.count, s.out]


def _run_host(s):
    if s.slots == 1:
        b = s.batches[0]
        kept = s.pipe.ardiff_pipeline_run_host(b["feat"], b["cond"], b["noise"], b["tau"], s.t, b["out"], b["mask"])
        return [b["out"], b["mask"], kept]
    kept = []
    for i, b in enumerate(s.batches):
        if i >= s.slots:
            kept.append(s.pipe.ardiff_pipeline_wait(i % s.slots))
        s.pipe.ardiff_pipeline_submit(i % s.slots, b["feat"], b["cond"], b["noise"], b["tau"], s.t, b["out"], b["mask"])
    for i in range(len(s.batches) - min(s.slots, len(s.batches)), len(s.batches)):
        kept.append(s.pipe.ardiff_pipeline_wait(i % s.slots))
    return [kept] + [[b["out"], b["mask"]] for b in s.batches]


# ---- the same in 64 bits -------------------------------------------------------------------------
def _row_entropies(feat):
    """Row entropies in fp64, whole batches in slices."""
    n, d = feat.shape
    step = max(1, (1 << 27) // d)
    h = torch.empty(n, dtype=torch.float64, device="cuda")
    for r0 in range(0, n, step):
        lp = torch.log_softmax(feat[r0:r0 + step].cuda().double(), dim=1)
        h[r0:r0 + step] = -(lp.exp() * lp).sum(dim=1)
    return h


def _threshold_statistics(h):
    mean, std = h.double().mean(), h.double().std(unbiased=False)
    return torch.stack([mean, std, 0.3 * mean - 0.1 * std])


def _head64(case, weights, cond, noise, t, coef, step_noise):
    """The head's sampler steps over the given rows: noise, one (ax, av, an) per step, fresh noise or None."""
    def bf16(name):
        return torch.from_numpy(weights[name].view(np.int16)).cuda().view(torch.bfloat16)

    w = {name: bf16(name) for name in weights}
    linear = lambda x, a, b: torch.nn.functional.linear(x, a.double(), b.double())
    silu, W, F = torch.nn.functional.silu, case["W"], TIME_FEATURES
    ln = lambda x: torch.nn.functional.layer_norm(x, (W,), eps=1e-6)
    freq = torch.exp(-math.log(10000.0) * torch.arange(F // 2, dtype=torch.float64, device="cuda") / (F // 2))
    c = linear(cond.cuda().double(), w["Wc"], w["bc"])
    x = noise.cuda().double()
    for k in range(len(coef)):
        arg = 1000.0 * float(t[k]) * freq
        temb = linear(silu(linear(torch.cat([arg.cos(), arg.sin()]), w["Wt1"], w["bt1"])), w["Wt2"], w["bt2"])
        s = silu(c + temb)
        h = linear(x, w["Win"], w["bin"])
        for b in range(case["L"]):
            shift, scale, gate = linear(s, w["Wmod"][b], w["bmod"][b]).chunk(3, dim=1)
            u = ln(h) * (1.0 + scale) + shift
            h = h + gate * linear(silu(linear(u, w["W1"][b], w["b1"][b])), w["W2"][b], w["b2"][b])
        shift, scale = linear(s, w["Wfm"], w["bfm"]).chunk(2, dim=1)
        v = linear(ln(h) * (1.0 + scale) + shift, w["Wout"], w["bout"])
        ax, av, an = (float(a) for a in coef[k])
        x = ax * x + av * v
        if step_noise is not None:
            x = x + an * step_noise[k].cuda().double()
    return x


def exact(case, seed):
    """What run() returns, in fp64 torch; None in the place of masks, ids, counts and lengths."""
    s, weights = _inputs(case, seed)
    kind = case["kind"]
    if kind == "gate":
        return [None, None, None, _row_entropies(s.feat)]
    if kind == "calibrate":
        h = _row_entropies(s.feat)
        return [None, None, None, h, _threshold_statistics(h), _threshold_statistics(s.pool)]
    if kind == "blocks":
        return [None, None, None, _row_entropies(s.feat).reshape(-1, s.rows).mean(dim=1), None]
    if kind == "sampler":
        coef, batches = s.coef.astype(np.float64), [s.__dict__]
    else:
        t = s.t.astype(np.float64)
        coef = np.stack([np.ones(case["K"]), np.diff(t), np.zeros(case["K"])], axis=1)
        batches = s.batches if kind == "host" else [s.__dict__]
    outs = []
    for b in batches:
        keep = (_row_entropies(b["feat"]) >= b["tau"]).nonzero()[:, 0]
        at = keep.to(b["cond"].device)
        out = torch.zeros((case["n"], case["C"]), dtype=torch.float64, device="cuda")
        fresh = s.step_noise[:, at] if kind == "sampler" else None
        out[keep] = _head64(case, weights, b["cond"][at], b["noise"][at], s.t, coef, fresh)
        outs.append(out)
    if kind != "host":
        return [None, None, None, outs[0]]
    return [outs[0], None, None] if s.slots == 1 else [None] + [[out, None] for out in outs]


# ---- what a pass cannot do without ---------------------------------------------------------------
def _survivors(case):
    return case["n"] * (1.0 - case["drop"])


def _flops_per_token(case):
    C, Dc, W, L, K = (case[k] for k in ("C", "Dc", "W", "L", "K"))
    return 2.0 * Dc * W + K * (10.0 * L * W * W + 4.0 * W * W + 4.0 * C * W)


def work(case):
    kind, n, d = case["kind"], case["n"], case["d"]
    rows = n * case.get("rows", 1)
    if kind == "gate":
        return {"bytes": rows * (2.0 * d + 4) + 5.0 * n + 4, "flops": 0.0}     # row and entropy; mask and id
    if kind == "blocks":
        # rows, their entropies; mask, id, indicator, two draws per token; two lengths per draft block
        return {"bytes": rows * (2.0 * d + 4) + 17.0 * n + 8.0 * math.ceil(n / case["gamma"]) + 4, "flops": 0.0}
    if kind == "calibrate":
        return {"bytes": rows * (2.0 * d + 4) + 5.0 * n + 4.0 * case["pool"] + 52, "flops": 0.0}
    C, Dc, W, L, K = (case[k] for k in ("C", "Dc", "W", "L", "K"))
    S, reps = _survivors(case), case.get("batches", 1)
    weights = 2.0 * (W * (Dc + TIME_FEATURES + W + C) + L * 5.0 * W * W + 2.0 * W * W + C * W + (5.0 * L + 6) * W + C)
    per_batch = n * (2.0 * d + 5) + 4 + S * (2.0 * Dc + 8.0 * C)
    if kind == "sampler":
        per_batch += K * S * 4.0 * C
    if kind == "host":
        per_batch += (n - S) * (2.0 * Dc + 8.0 * C)        # whole batches cross the bus, dropped rows included
    return {"bytes": weights + reps * per_batch, "flops": reps * S * _flops_per_token(case)}


def tolerance(case):
    """Four times what these passes differ by from the same arithmetic in 64 bits.

    Heads (bf16 operands, fp32 accumulation): Euler passes were off by 1.0e-3 to 2.0e-3 of the output's norm at K >= 2 and
    by 3.8e-3 at K = 1, the x0-prediction sampler, whose output is the raw prediction, by up to 5.9e-3; single values
    by four times that. Entropies (fp32 sums of up to 16384 terms): up to 2.5e-7 of the norm, 2.5e-6 in one value."""
    if case["kind"] in ("path", "host"):
        rel = 8e-3 if case["K"] > 1 else 1.5e-2
        return {"rel": rel, "max": 5 * rel}
    if case["kind"] == "sampler":
        return {"rel": 2.4e-2, "max": 0.12}
    return {"rel": 1e-6, "max": 1e-5}
