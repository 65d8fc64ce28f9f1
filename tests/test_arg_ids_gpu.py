"""Ids as arguments of a step's own kernels, up to 160 of them, and as stored ids above: same losses, gradients and logits bit for bit as with ids on the device."""
import numpy as np
import pytest
import torch

import pac_inputs as pi
import paper_2408_10746_b200 as pac
from tests.common import Case

pytestmark = pytest.mark.gpu

SPEC = pi.CacheSpec("arg_ids", N=400, L=2, S=4, d=64, dtype="bf16", r=16, n_out=3, B=8)


@pytest.fixture(scope="module")
def case():
    return Case(SPEC)


@pytest.mark.parametrize("B", [1, 33, 159, 160, 161])
def test_every_call_with_host_ids_equals_device_ids(case, B):
    hp = pac.AdamW(lr=1e-3)
    ids = [np.array([(11 * i + 5 + s) % SPEC.N for i in range(B)], dtype=np.int32) for s in range(3)]
    dev, calls = case.context(max_batch=B), [case.context(max_batch=B) for _ in range(4)]
    want, loss = [], torch.zeros(1, dtype=torch.float32, device="cuda")
    pinned = torch.zeros(1).pin_memory()
    for i in ids:
        dev.train_epoch_dev(torch.from_numpy(i).cuda(), B, hp, loss)
        dev.sync()
        want.append((float(loss), dev.get_grads(), dev.get_params()))
    for s, i in enumerate(ids):
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
            assert g == want[s][0]
            assert np.array_equal(c.get_grads(), want[s][1]) and np.array_equal(c.get_params(), want[s][2])
    out = torch.empty((B, SPEC.n_out), device="cuda")
    calls[0].eval_logits(ids[0], out)
    calls[0].sync()
    for j in (0, B - 1):
        one = torch.empty((1, SPEC.n_out), device="cuda")
        calls[0].eval_logits(ids[0][j:j + 1], one)
        calls[0].sync()
        assert torch.allclose(out[j], one[0], rtol=1e-5, atol=1e-6)
    for c in calls + [dev]:
        c.close()
    with pytest.raises(Exception):
        case.context(max_batch=B).train_step([SPEC.N] * B)
