"""Ids as arguments of a step's own kernels, up to 160 of them, and as stored ids above: same losses, gradients and parameters bit for bit as with ids on the device, and
logits of the samples that were asked for, row by row against the oracle (1e-4 for fp32 precision, 2e-2 for bf16 products, of a row's norm: another sample's row is another row)."""
import numpy as np
import pytest
import torch

import pac_inputs as pi
import paper_2408_10746_b200 as pac
from oracle import pac_oracle as po
from oracle import tbody_oracle as tb
from tests.common import Case
from tests.test_tbody_gpu import random_flat

pytestmark = pytest.mark.gpu

SPEC = pi.CacheSpec("arg_ids", N=400, L=2, S=4, d=64, dtype="bf16", r=16, n_out=3, B=8)


@pytest.fixture(scope="module")
def case():
    return Case(SPEC)


def same_everywhere(make, N, B, batches):
    """Every call with host ids against an epoch of one step with device ids, step by step; the first context stays open."""
    hp = pac.AdamW(lr=1e-3)
    ids = [np.array([(11 * i + 5 + s) % N for i in range(B)], dtype=np.int32) for s in range(batches)]
    dev, calls = make(), [make() for _ in range(4)]
    loss, pinned = torch.zeros(1, dtype=torch.float32, device="cuda"), torch.zeros(1).pin_memory()
    for i in ids:
        dev.train_epoch_dev(torch.from_numpy(i).cuda(), B, hp, loss)
        dev.sync()
        want, grads, params = float(loss), dev.get_grads(), dev.get_params()
        got = [calls[0].train_step(i)]
        calls[0].adam_step(hp)
        calls[1].train_step_async(i, hp, pinned.data_ptr())
        calls[1].sync()
        got.append(float(pinned))
        calls[2].train_step_dev_loss(i, loss.data_ptr())
        calls[2].adam_step(hp)
        calls[2].sync()
        got.append(float(loss))
        got.append(float(calls[3].train_epoch(i, B, hp)[0]))
        for c, g in zip(calls, got):
            assert g == want
            assert np.array_equal(c.get_grads(), grads) and np.array_equal(c.get_params(), params)
    for c in calls[1:] + [dev]:
        c.close()
    return calls[0]


def rows_match(ctx, B, n_out, ids, ref, tol):
    out = torch.empty((B, n_out), device="cuda")
    ctx.eval_logits(ids, out)
    ctx.sync()
    out = out.cpu().numpy().astype(np.float64)
    for b in range(B):
        assert np.linalg.norm(out[b] - ref[b]) < tol * np.linalg.norm(ref[b]), b


@pytest.mark.parametrize("B", [1, 33, 159, 160, 161])
def test_every_call_with_host_ids_equals_device_ids(case, B):
    ctx = same_everywhere(lambda: case.context(max_batch=B), SPEC.N, B, 3)
    ids = [(11 * i + 8) % SPEC.N for i in range(B)]
    P = case.oracle_params(ctx.get_params())
    rows_match(ctx, B, SPEC.n_out, ids, po.eval_logits(P, case.H(ids).astype(np.float32), 0), 2e-2)
    with pytest.raises(pac.PacError) as e:
        ctx.train_step([SPEC.N] * B)
    assert e.value.status_name == "PAC_ERR_SAMPLE_ID_RANGE"
    ctx.close()


def spec(name, **kw):
    return pi.CacheSpec(name, **{**dict(N=24, L=3, S=65, d=128, dtype="bf16", r=96, n_out=3, B=4), **kw})


# The other kernels that take ids as an argument or leave their copy
ROUTES = [
    (spec("chain_forward", B=3), 4, "tensor+chain_forward"),                        # an odd number of tiles: a CTA each
    (spec("chain_forward_in_pairs"), 4, "tensor+chain_forward"),
    (spec("head_matrix_ahead", r=64, S=140), 0, "tensor"),
    (spec("gates_alone", r=128, S=129, B=8), 0, "tensor"),
    (spec("fp32_products", dtype="f32", r=20, d=100), 0, "simt"),
    (spec("fp32_products_of_a_bf16_cache", r=20, d=101), 0, "simt"),
    (spec("fp32_products_several_waves", dtype="f32", r=16, L=24, S=128, B=16, d=256), 0, "simt"),
]


@pytest.mark.parametrize("sp,path,name", ROUTES, ids=[r[0].name for r in ROUTES])
def test_every_route_takes_host_ids(sp, path, name):
    case = Case(sp)
    start = pi.random_params(sp, 3)

    def make():
        c = case.context(kernel_path=path)
        assert c.kernel_path() == name
        c.set_params(start)
        return c
    ctx = same_everywhere(make, sp.N, sp.B, 3)
    ids = [(7 * i + 2) % sp.N for i in range(sp.B)]
    P = case.oracle_params(ctx.get_params())
    rows_match(ctx, sp.B, sp.n_out, ids, po.eval_logits(P, case.H(ids).astype(np.float32), 0), 1e-4 if name == "simt" else 2e-2)
    ctx.close()


@pytest.mark.parametrize("sp", [spec("transformer_fused", dtype="f32", r=16, S=20), spec("transformer_per_operation", dtype="f32", r=196, S=20, L=2)], ids=lambda s: s.name)
def test_transformer_bodies_take_host_ids(sp):
    heads, f = 2, 24
    start = random_flat(sp, f, 3)
    cache, labels = pi.cache_full(sp, 0, "cuda"), pi.labels(sp, 0, "cuda")

    def make():
        c = pac.PacContext(0)
        c.cache_register(cache, labels)
        c.adapter_init(r=sp.r, n_out=sp.n_out, max_batch=sp.B, body=pac.PAC_BODY_TRANSFORMER, n_heads=heads, ffn_width=f)
        c.set_params(start)
        return c
    ctx = same_everywhere(make, sp.N, sp.B, 3)
    ids = [(7 * i + 2) % sp.N for i in range(sp.B)]
    P, T = tb.unflatten(ctx.get_params(), sp.L, sp.d, sp.r, sp.n_out, f)
    rows_match(ctx, sp.B, sp.n_out, ids, tb.eval_logits(P, T, pi.cache_samples(sp, 0, ids, "cpu").float().numpy(), heads), 1e-4)
    ctx.close()
