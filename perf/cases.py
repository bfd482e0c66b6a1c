"""The work a user of this library has it do, as cases that can be timed and compared.

A pass is one forward call through the public entry points on new inputs: a DiT block, or a stack of
blocks (one denoising step), under the chunking its caller chose or its byte budget asks for.  The
arena reuses the slots of the block input and of the timestep embedding, so a pass starts by
putting them there, as every caller has to.  There is no backward direction.

Fields of a case:
  batch, s_text, grid_t, grid_h, grid_w, hidden, heads, ffn, n_blocks   the request template
  budget_mib   > 0: the activation budget the chunk counts are searched for
  chunks       "": from the budget; else explicit counts of the three phases, "CA,CB,CC"
  per_phase    budget search with one count per phase (the default of BlockSession) or one for all
  serialize    budget search that may split a phase into sub-batches
  call         "forward"  BlockSession.set_inputs and .forward, tensors on the device
               "graph"    the same forward, recorded once by BlockSession.capture and replayed
               "host"     Plan.forward_host: page-locked host buffers in and out
               "shard"    BlockSession.forward_sharded of shard 1 of 4; the keys and values of the
                          other shards are copied in from a buffer at the gather point of each block
"""
from __future__ import annotations

import math

import torch

from paper_2607_11136_b200 import binding as xb
from paper_2607_11136_b200.session import BlockSession
from xema_inputs import Template, weight_shapes

DEVICE = "cuda:0"
TEMB_DIM = 512
SHARD, SHARDS = 1, 4
MIB = 1 << 20
LARGEST_FLOPS = 2.7e14       # just under the largest listed case (42 blocks of 17 776 tokens)


def _case(name, batch, s_text, grid, hidden, heads, n_blocks=1, budget_mib=0.0, chunks="", per_phase=True,
          serialize=False, call="forward", ffn=0):
    case = {"name": name} if name else {}
    case.update(batch=batch, s_text=s_text, grid_t=grid[0], grid_h=grid[1], grid_w=grid[2], hidden=hidden, heads=heads,
                ffn=ffn or 4 * hidden, n_blocks=n_blocks, budget_mib=float(budget_mib), chunks=chunks,
                per_phase=per_phase, serialize=serialize, call=call)
    return case


def listed():
    return [
        # The smallest template, one block: a preview-sized latent, where launches and host time count.
        _case("tiny block", 1, 32, (4, 8, 8), 512, 8, chunks="1,1,1"),
        # A shallow model's whole step on a 256 x 256 image, recorded once and replayed per step: what a
        # latency-minded caller does with launch-bound work.
        _case("small step, graph", 1, 77, (1, 16, 16), 1024, 16, n_blocks=8, chunks="1,1,1", call="graph"),
        # One 512 x 512 image of a medium model, head_dim 64.
        _case("medium image block", 1, 77, (1, 32, 32), 1536, 24, chunks="1,1,1"),
        # Three requests of an odd image size in one batch, head_dim 128, row-chunked: every tile is ragged.
        _case("ragged batch of 3", 3, 77, (1, 37, 53), 2048, 16, chunks="2,3,3"),
        # Flux-style 1024 x 1024 image block, head_dim 128; its budget does not bind.
        _case("flux block", 1, 512, (1, 64, 64), 3072, 24, budget_mib=24 * 1024),
        # Four such requests served together at 0.9 of the unsplit peak: the feed-forward runs as two sub-batches.
        _case("flux block, batch 4", 4, 512, (1, 64, 64), 3072, 24, budget_mib=680, serialize=True),
        # CogVideoX-shaped block at the headline budget: per-phase chunks (1, 1, 2).
        _case("video block 640 MiB", 1, 226, (13, 30, 45), 3072, 48, budget_mib=640),
        # The same block where one chunk count serves all phases (the paper's plain chunking): four chunks.
        _case("video block uniform", 1, 226, (13, 30, 45), 3072, 48, budget_mib=576, per_phase=False),
        # The same block served end to end: latent in from the host, result back to the host.
        _case("video block from host", 1, 226, (13, 30, 45), 3072, 48, budget_mib=640, call="host"),
        # One GPU's share of that block under sequence parallelism of degree 4.
        _case("video block shard", 1, 226, (13, 30, 45), 3072, 48, chunks="1,1,1", call="shard"),
        # A 1080p x 49 frame block under a 4 GiB budget: attention is five sixths of the work.
        _case("long video block", 1, 226, (13, 68, 120), 3072, 48, budget_mib=4096),
        # A full denoising step: 42 stacked blocks.
        _case("video step, 42 blocks", 1, 226, (13, 30, 45), 3072, 48, n_blocks=42, budget_mib=640),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """A template between the listed ones: tokens over three decades, any legal width, either head
    size, one to four requests, one or several blocks, chunked or not, any of the calls."""
    while True:
        head_dim = rng.choice((64, 128))
        hidden = 256 * rng.randint(2, 12)
        batch = rng.choice((1, 1, 1, 2, 3, 4))
        tokens = _log_int(rng, 250, 30000)
        s_text = min(rng.choice((0, 32, 77, 226, 512)), tokens // 3)
        grid_t = rng.choice((1, 1, 4, 7, 13)) if tokens > 2000 else 1
        side = max(4.0, math.sqrt((tokens - s_text) / grid_t))
        grid_h = max(4, int(round(side * rng.uniform(0.7, 1.2))))
        grid_w = max(4, int(round((tokens - s_text) / (grid_t * grid_h))))
        n_blocks = rng.choice((1, 1, 2, 8)) if tokens < 4000 else rng.choice((1, 1, 2))
        counts = (1, 1, 1, 2, 3, 4) if tokens < 4000 else (1, 1, 1, 2, 4, 8)
        chunks = ",".join(str(rng.choice(counts)) for _ in range(3))
        call = rng.choice(("forward", "forward", "forward", "graph", "host", "shard"))
        case = _case("", batch, s_text, (grid_t, grid_h, grid_w), hidden, hidden // head_dim, n_blocks=n_blocks,
                     chunks=chunks, call=call)
        if work(case)["flops"] <= LARGEST_FLOPS:
            return case


def _template(case):
    return Template(case.get("name", "drawn"), case["batch"], case["s_text"], case["grid_t"], case["grid_h"],
                    case["grid_w"], case["hidden"], case["heads"], case["hidden"] // case["heads"], case["ffn"],
                    temb_dim=TEMB_DIM, n_blocks=case["n_blocks"])


def _normal(gen, shape, scale=1.0, mean=0.0):
    return (torch.randn(shape, device=DEVICE, generator=gen, dtype=torch.float32) * scale + mean).to(torch.bfloat16)


class _State:
    """What a user's program holds between calls: a bound session and its own input (and, for the
    host call, output) buffers."""


def prepare(case, seed):
    t = _template(case)
    gen = torch.Generator(device=DEVICE).manual_seed(seed)
    s = _State()
    s.call = case["call"]
    # parameters N(0, 0.02^2), the two RMSNorm gains around 1; activations N(0, 1)
    weights = [{name: _normal(gen, shape, 0.02, 1.0 if name in ("g_q", "g_k") else 0.0)
                for name, shape in weight_shapes(t).items()} for _ in range(t.n_blocks)]
    kw = {}
    if case["chunks"]:
        kw["chunks"] = tuple(int(c) for c in case["chunks"].split(","))
    else:
        kw.update(budget_bytes=int(case["budget_mib"] * MIB), per_phase=case["per_phase"], serialize=case["serialize"])
    if s.call == "shard":
        kw["shard"] = (SHARD, SHARDS)
    s.session = BlockSession(t, weights, device=DEVICE, **kw)
    s.x = _normal(gen, (t.batch, s.session.seq, t.hidden)).view(torch.int16)
    s.temb = _normal(gen, (t.batch, t.temb_dim)).view(torch.int16)
    if s.call == "graph":
        s.session.set_inputs(s.x, s.temb)
        s.graph = s.session.capture()
    elif s.call == "host":
        s.x, s.temb = s.x.cpu().pin_memory(), s.temb.cpu().pin_memory()
        s.out = torch.empty_like(s.x).pin_memory()
    elif s.call == "shard":
        # what the other shards would send: keys as an RMSNorm leaves them, and values
        kv = torch.randn((t.batch, t.seq, 2, t.heads, t.head_dim), device=DEVICE, generator=gen)
        kv[:, :, 0] *= torch.rsqrt(kv[:, :, 0].square().mean(dim=-1, keepdim=True))
        s.kv = kv.to(torch.bfloat16).view(torch.int16).view(t.batch, t.seq, 2 * t.hidden)
        s.own = (s.session.plan.row0, s.session.plan.row0 + s.session.plan.rows)
    return s


def run(s):
    sess = s.session
    stream = torch.cuda.current_stream()
    if s.call == "host":
        sess.plan.forward_host(s.x.data_ptr(), s.temb.data_ptr(), s.out.data_ptr(), stream.cuda_stream)
        return s.out.view(torch.bfloat16)
    sess.set_inputs(s.x, s.temb, non_blocking=True)
    if s.call == "graph":
        s.graph.replay()
    elif s.call == "shard":
        def exchange(block):
            kv = sess.kv(block)
            kv[:, :s.own[0]].copy_(s.kv[:, :s.own[0]])
            kv[:, s.own[1]:].copy_(s.kv[:, s.own[1]:])
        sess.forward_sharded(exchange, stream)
    else:
        sess.forward(stream)
    return sess.hid_out().view(torch.bfloat16)


def work(case):
    B, D, F, L = case["batch"], case["hidden"], case["ffn"], case["n_blocks"]
    S = case["s_text"] + case["grid_t"] * case["grid_h"] * case["grid_w"]
    rows = (SHARD + 1) * S // SHARDS - SHARD * S // SHARDS if case["call"] == "shard" else S
    head_dim = D // case["heads"]
    flops = L * B * (2.0 * rows * D * (3 * D + D + 2 * F) + 4.0 * rows * S * D + 2.0 * 6 * D * TEMB_DIM)
    params = 6 * D * TEMB_DIM + 6 * D + 4 * D * D + 4 * D + 2 * head_dim + 2 * D * F + F + D
    nbytes = 2.0 * L * params + 2 * 2.0 * B * rows * D + 2.0 * B * TEMB_DIM + 4.0 * rows * head_dim
    if case["call"] == "shard":
        nbytes += L * 2.0 * B * (S - rows) * 2 * D
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    # Measured against float32 torch versions that round to bf16 at the same places: relative error
    # up to 1.3e-3 and largest difference up to 1.2e-2 after one block, 2.9e-3 and 2.3e-2 after 8,
    # 1.1e-2 and 8.6e-2 after 42 (a last-bit difference is carried on from block to block).  About
    # four times that; the growth is close to the square root of the number of blocks.
    n = math.sqrt(case["n_blocks"])
    return {"rel": min(5e-3 * n, 3e-2), "max": min(5e-2 * n, 0.35)}
