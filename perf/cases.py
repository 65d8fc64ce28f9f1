"""Workloads of the adapter-over-cache trainer, as a user's program runs them.

Every case goes through the package's public calls (PacContext, quantize_absmax,
dequantize_absmax).  A case is a dict of plain values:

    call    what one pass does (see run()):
              "step"        train_step (waits for the loss) + adam_step
              "async"       train_step_async with the loss in page-locked host memory
              "dev_loss"    train_step_dev_loss + adam_step (one rank of data-parallel training)
              "epoch"       train_epoch: `steps` minibatches of a host permutation
              "epoch_dev"   train_epoch_dev: the same with ids and losses on the device
              "eval"        eval_logits of one batch
              "gather"      gather of one batch's slabs
              "codec"       quantize_absmax and dequantize_absmax of one weight vector
    dtype   of the cache, "bf16" or "f32"
    cache   "device", or "host" (page-locked host memory, reloaded per minibatch)
    head    "cls" (mean-pool classifier) or "lm" (frozen LM head)
    body    "relu" or "identity" (point-wise adapters) or "transformer" (`heads`, ffn width 4r)
    N, L, S, d, r, n_out, B, steps     sizes as in pac.h; B is the minibatch of one step

Caches are larger than L2 and every pass takes other minibatches, as an epoch does.  The training state
is that of a run under way: W_up is not zero and the moments are warm.
"""
import math

import numpy as np
import torch

import paper_2408_10746_b200 as pac


def _case(name, call, dtype, N, L, S, d, r, n_out, B, *, cache="device", head="cls", body="relu", heads=0, steps=1):
    return {"name": name, "call": call, "dtype": dtype, "cache": cache, "head": head, "body": body, "heads": heads,
            "N": N, "L": L, "S": S, "d": d, "r": r, "n_out": n_out, "B": B, "steps": steps}


def listed():
    return [
        # the plainest training loop on the smallest configuration: one blocking call per minibatch
        _case("step_tiny_fp32", "step", "f32", 256, 4, 32, 256, 16, 2, 8),
        # T5-Base-shaped encoder cache, minibatches chosen on the host one at a time, nothing waited for
        _case("async_t5_base", "async", "bf16", 512, 12, 128, 768, 64, 3, 32),
        # BART-Large-shaped cache, a stretch of an epoch whose permutation is on the device
        _case("epoch_bart_large", "epoch_dev", "bf16", 256, 24, 128, 1024, 64, 2, 32, steps=4),
        # T5-Large-shaped cache: long sequences, wide adapters, the largest classifier step
        _case("epoch_t5_large", "epoch_dev", "bf16", 256, 24, 256, 1024, 128, 5, 64, steps=4),
        # LLaMA-7B-shaped decoder stack with its frozen LM head, one rank's step
        _case("lm_llama_7b", "dev_loss", "bf16", 32, 32, 512, 4096, 64, 32000, 16, head="lm"),
        # 500 short samples of 30 tokens (the storage-cost example of the paper), ragged everywhere, host permutation
        _case("epoch_short_ragged", "epoch", "bf16", 500, 12, 30, 768, 64, 2, 20, steps=5),
        # an fp32 cache of an ordinary size, one rank's step: full-precision products
        _case("step_f32_t5_base", "dev_loss", "f32", 128, 12, 128, 768, 64, 3, 16),
        # transformer-body adapters (the paper's "lightweight version of the backbone")
        _case("transformer_t5_base", "async", "bf16", 128, 12, 128, 768, 64, 3, 16, body="transformer", heads=4),
        # validation pass: forward only, the last and smaller batch of a split
        _case("eval_t5_base", "eval", "bf16", 512, 12, 128, 768, 64, 3, 27),
        # the cached states themselves for another consumer
        _case("gather_t5_large", "gather", "bf16", 128, 24, 256, 1024, 128, 5, 32),
        # block-wise INT8 of one 4096 x 11008 weight matrix and back, block 64
        {"name": "codec_block64", "call": "codec", "n": 4096 * 11008, "block": 64},
        # a cache that stays in host memory, one stretch of an epoch
        _case("host_cache_t5_base", "epoch", "bf16", 128, 12, 128, 768, 64, 3, 32, cache="host", steps=4),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["cls", "cls", "cls", "f32", "f32", "transformer", "lm", "eval", "eval", "gather", "codec", "codec", "host"])
    if kind == "codec":
        block = rng.choice([32, 64, 64, 100, 128, 256, 1000, 1024, 2048, 4096])
        n = _log_int(rng, 1 << 14, 1 << 26)
        return {"call": "codec", "n": n if rng.random() < 0.3 else n // block * block + block, "block": block}
    if kind == "lm":
        L, S, d, r = rng.randint(4, 32), rng.randint(20, 512), 64 * rng.randint(4, 64), 16 * rng.randint(1, 4)
        B = max(1, min(16, _log_int(rng, 128, 8192) // S))
        N = max(2 * B, min(512, (1 << 30) // (L * S * d)))
        return _pick(_case("", rng.choice(["dev_loss", "async"]), "bf16", N, L, S, d, r, 8 * rng.randint(1000, 4000), B, head="lm"))
    # classifier shapes: batch x tokens x layers x width bounded by the largest listed step
    L, S = rng.randint(2, 24), _log_int(rng, 12, 300)
    d = rng.choice([8 * rng.randint(16, 128), 64 * rng.randint(2, 16), 768, 1024, rng.randint(100, 1000)])
    r = rng.choice([16, 16 * rng.randint(1, 8), 32, 64, 64, 128, rng.randint(8, 100)])
    top = 64 * 24 * 256 * 1024
    if kind in ("f32", "transformer"):
        top = 16 * 12 * 128 * 768
    B = max(1, min(64, _log_int(rng, 1, 96), top // (L * S * d)))
    while B * L * S * d > top or (kind != "cls" and B * L * S * r > 2 * 64 * 24 * 256 * 16):
        S = max(8, S // 2)
    N = max(2 * B, min(512, (1 << 28) // (L * S * d)))
    n_out, body = rng.randint(2, 8), "identity" if rng.random() < 0.15 else "relu"
    if kind == "transformer":
        heads = rng.choice([2, 4, 8])
        r = heads * max(2, min(96 // heads, r // heads))
        S = min(S, 256)
        return _pick(_case("", rng.choice(["async", "dev_loss"]), rng.choice(["bf16", "bf16", "f32"]), N, L, S, d, r, n_out, B,
                           body="transformer", heads=heads))
    if kind == "host":
        B = min(B, 32, max(1, (1 << 25) // (L * S * d)))
        return _pick(_case("", "epoch", "bf16", 4 * B, L, S, d, r, n_out, B, cache="host", body=body, steps=rng.randint(2, 4)))
    if kind in ("eval", "gather"):
        return _pick(_case("", kind, rng.choice(["bf16", "bf16", "f32"]) if B * L * S * d <= top // 8 else "bf16", N, L, S, d, r, n_out, B, body=body))
    call = rng.choice(["step", "async", "dev_loss", "epoch", "epoch_dev"])
    return _pick(_case("", call, "f32" if kind == "f32" else "bf16", N, L, S, d, r, n_out, B, body=body,
                       steps=rng.randint(2, 4) if call.startswith("epoch") else 1))


def _pick(case):
    """A drawn case has no name of its own."""
    return {k: v for k, v in case.items() if k != "name"}


_STREAM = None


def _stream():
    """One stream for every context, as a program with one training stream has it."""
    global _STREAM
    if _STREAM is None:
        _STREAM = torch.cuda.Stream()
    return _STREAM


def _normal(gen, *shape, dtype=torch.float32):
    return torch.randn(*shape, generator=gen, device="cuda", dtype=dtype)


def prepare(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    if case["call"] == "codec":
        # weights of a trained layer: Gaussian, a few large entries
        x = _normal(gen, case["n"]).mul_(0.02)
        x[::997] *= 8.0
        return {"case": case, "x": x}
    N, L, S, d, r, n_out, B = (case[k] for k in ("N", "L", "S", "d", "r", "n_out", "B"))
    # hidden states: Gaussian, the standard deviation grows with depth (Section VI's models are not available here)
    growth = (1.0 + 0.1 * torch.arange(L, device="cuda")).view(1, L, 1, 1)
    cache = torch.empty(N, L, S, d, device="cuda", dtype=torch.bfloat16 if case["dtype"] == "bf16" else torch.float32)
    for n0 in range(0, N, 16):
        part = cache[n0:n0 + 16]
        part.copy_(_normal(gen, *part.shape, dtype=cache.dtype).mul_(growth.to(cache.dtype)))
    lm = case["head"] == "lm"
    labels = torch.randint(0, n_out, (N, S) if lm else (N,), generator=gen, device="cuda", dtype=torch.int32)
    head = _normal(gen, n_out, d, dtype=torch.bfloat16).mul_(1.0 / (math.sqrt(d) * (1.0 + 0.1 * (L - 1)))) if lm else None
    if case["cache"] == "host":
        host = torch.empty(cache.shape, dtype=cache.dtype, pin_memory=True)
        host.copy_(cache)
        cache, labels = host, labels.cpu().pin_memory()
    torch.cuda.synchronize()
    ctx = pac.PacContext(0, _stream().cuda_stream)
    (ctx.cache_register_host if case["cache"] == "host" else ctx.cache_register)(cache, labels)
    more = {}
    if case["body"] == "transformer":
        more = {"body": pac.PAC_BODY_TRANSFORMER, "n_heads": case["heads"], "ffn_width": 4 * r}
    ctx.adapter_init(r=r, n_out=n_out, max_batch=B, act=pac.PAC_ACT_IDENTITY if case["body"] == "identity" else pac.PAC_ACT_RELU,
                     head=pac.PAC_HEAD_FROZEN_LM if lm else pac.PAC_HEAD_MEANPOOL_CLS, lm_head=head, seed=seed, **more)
    params, grads = ctx.device_buffers()
    params.owner = grads.owner = ctx          # views of the context's memory: they must not outlive it
    n = params.numel()
    up = L * d * r + L
    params[up - L:up] += 0.05 * _normal(gen, L)
    params[up:up + r * d] = 0.02 * _normal(gen, r * d)
    torch.cuda.synchronize()
    ctx.params_changed()
    rng = np.random.default_rng(seed)
    m = rng.standard_normal(n, dtype=np.float32) * np.float32(1e-4)
    v = rng.random(n, dtype=np.float32) * np.float32(1e-6) + np.float32(5e-7)
    ctx.set_opt_state(m, v, 200)
    ctx.sync()
    # one shuffled epoch after the other; enough of them that no pass repeats another's minibatches soon
    per_pass = B * case["steps"]
    perm = np.concatenate([rng.permutation(N) for _ in range(max(1, -(-4 * per_pass // N)))]).astype(np.int32)
    passes = max(1, perm.size // per_pass)
    state = {"case": case, "ctx": ctx, "hp": pac.AdamW(), "params": params, "grads": grads, "at": 0,
             "ids": [np.ascontiguousarray(perm[i * per_pass:(i + 1) * per_pass]) for i in range(passes)]}
    if case["call"] == "eval":
        state["out"] = torch.empty((B, S, n_out) if lm else (B, n_out), device="cuda")
    elif case["call"] == "gather":
        state["out"] = torch.empty(L, B, S, d, device="cuda", dtype=cache.dtype)
    elif case["call"] == "async":
        state["loss"] = torch.zeros(1).pin_memory()
    elif case["call"] == "dev_loss":
        state["loss"] = torch.zeros(1, device="cuda")
    elif case["call"] == "epoch_dev":
        state["ids"] = [torch.from_numpy(i).cuda() for i in state["ids"]]
        state["loss"] = torch.zeros(case["steps"], device="cuda")
    return state


def run(state):
    case = state["case"]
    call = case["call"]
    if call == "codec":
        q, c = pac.quantize_absmax(state["x"], case["block"])
        return q, c, pac.dequantize_absmax(q, c, case["block"])
    ctx, hp = state["ctx"], state["hp"]
    ids = state["ids"][state["at"] % len(state["ids"])]
    state["at"] += 1
    if call == "eval":
        return ctx.eval_logits(ids, state["out"])
    if call == "gather":
        return ctx.gather(ids, state["out"])
    if call == "step":
        loss = ctx.train_step(ids)
        ctx.adam_step(hp)
    elif call == "async":
        loss = state["loss"]
        ctx.train_step_async(ids, hp, loss.data_ptr())
    elif call == "dev_loss":
        loss = state["loss"]
        ctx.train_step_dev_loss(ids, loss.data_ptr())
        ctx.adam_step(hp)
    elif call == "epoch":
        loss = ctx.train_epoch(ids, case["B"], hp)
    else:
        loss = state["loss"]
        ctx.train_epoch_dev(ids, case["B"], hp, loss)
    return {"loss": loss, "params": state["params"], "grads": state["grads"]}


def work(case):
    """Each input once and each output once; the adapter stack's own products, no padding and no recomputation."""
    if case["call"] == "codec":
        n, blocks = case["n"], -(-case["n"] // case["block"])
        return {"bytes": (4 + 1) * n + 4 * blocks + (1 + 4) * n + 4 * blocks, "flops": 4 * n}
    L, S, d, r, n_out, B, steps = (case[k] for k in ("L", "S", "d", "r", "n_out", "B", "steps"))
    e = 2 if case["dtype"] == "bf16" else 4
    M, slabs = B * S, B * L * S * d * e
    if case["call"] == "gather":
        return {"bytes": 2 * slabs, "flops": 0}
    lm = case["head"] == "lm"
    n = L * d * r + L + r * d + (0 if lm else d * n_out + n_out)
    fwd = 2 * M * L * d * r
    if lm:
        fwd += 2 * M * d * n_out + 2 * M * d * r
    if case["body"] == "transformer":
        n += L * (4 * r * r + 8 * r * r + 9 * r)
        fwd += L * (2 * M * (4 * r * r + 8 * r * r) + 4 * M * S * r)
    if case["call"] == "eval":
        return {"bytes": slabs + 4 * n + 4 * (M if lm else B) * n_out + (2 * n_out * d if lm else 0), "flops": fwd}
    bwd = 2 * M * L * d * r
    if lm:
        bwd += 2 * M * d * n_out + 2 * 2 * M * d * r
    if case["body"] == "transformer":
        bwd += L * (4 * M * (4 * r * r + 8 * r * r) + 8 * M * S * r)
    # parameters and both moments in and out, gradients out
    return {"bytes": steps * (slabs + 28 * n + (2 * n_out * d if lm else 0)), "flops": steps * (fwd + bwd)}


def tolerance(case):
    """What another correct implementation would show.  The codec's arithmetic is defined operation by operation and a
    gather copies: nothing may differ.  bf16 caches: products of bf16 operands.  fp32 products differ by about 1e-6, but
    a ReLU whose argument is within that of zero may open on one side only and moves single gradient elements by a
    token's share: with n gated elements about n * 1e-6 of them, of relative weight 1 / sqrt(n) each, do so."""
    if case["call"] in ("codec", "gather"):
        return "exact"
    full = case["dtype"] == "f32" or case["body"] == "transformer"
    if not full:
        return {"rel": 1e-2, "max": 0.4}
    if case["call"] == "eval":
        return {"rel": 2e-5, "max": 2e-4}
    gated = case["B"] * case["S"] * case["L"] * case["r"] * (5 if case["body"] == "transformer" else 1)
    if case["body"] == "identity" or gated < 100000:
        return {"rel": 1e-4, "max": 1e-2}
    return {"rel": 2e-3, "max": 0.2}
