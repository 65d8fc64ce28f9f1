"""Ids that travel as a kernel argument and, above 512, as a copy: same samples, same losses as with ids that are on the device."""
import numpy as np
import pytest
import torch

import pac_inputs as pi
import paper_2408_10746_b200 as pac
from tests.common import Case

pytestmark = pytest.mark.gpu

SPEC = pi.CacheSpec("ids", N=600, L=2, S=4, d=64, dtype="bf16", r=16, n_out=3, B=8)


@pytest.fixture(scope="module")
def case():
    return Case(SPEC)


@pytest.mark.parametrize("B", [1, 31, 511, 512, 513, 600])
def test_gather_takes_every_id(case, B):
    ctx = case.context(max_batch=600)
    for shift in (0, 3):                                    # the second call's ids follow while the first call still runs
        ids = [(7 * i + shift) % SPEC.N for i in range(B)]
        out = torch.empty((SPEC.L, B, SPEC.S, SPEC.d), dtype=torch.bfloat16, device="cuda")
        ctx.gather(ids, out)
        ctx.sync()
        assert torch.equal(out, case.cache[torch.tensor(ids, device="cuda")].transpose(0, 1))
    ctx.close()


@pytest.mark.parametrize("n,B", [(2, 1), (512, 64), (513, 57), (1024, 512), (1026, 513)])
def test_epoch_equals_epoch_with_device_ids(case, n, B):
    perm = np.array([(11 * i + 5) % SPEC.N for i in range(n)], dtype=np.int32)
    hp = pac.AdamW(lr=1e-3)
    host, dev = case.context(max_batch=B), case.context(max_batch=B)
    losses = torch.zeros(n // B, dtype=torch.float32, device="cuda")
    for _ in range(2):
        mine = host.train_epoch(perm, B, hp)
        dev.train_epoch_dev(torch.from_numpy(perm).cuda(), B, hp, losses)
        dev.sync()
        assert np.array_equal(mine, losses.cpu().numpy())
    assert np.array_equal(host.get_params(), dev.get_params())
    assert host.train_step(perm[:B]) == dev.train_step(perm[:B])
    host.close(); dev.close()


@pytest.mark.parametrize("pinned", [True, False], ids=["pinned", "pageable"])
@pytest.mark.parametrize("ids", [[5], [3, 9], [9, 3], [4, 4, 4], [599, 0, 598, 1, 2, 2, 300], list(range(20)), list(range(20, 0, -1))], ids=str)
def test_samples_from_host_memory_land_in_their_rows(case, ids, pinned):
    """Two samples of a batch may travel as the rows of one copy: ascending, descending, repeated and odd ones."""
    cache, labels = case.cache.cpu(), case.labels.cpu()
    if pinned:
        cache, labels = cache.pin_memory(), labels.pin_memory()
    ctx = pac.PacContext(0)
    ctx.cache_register_host(cache, labels)
    ctx.adapter_init(r=SPEC.r, n_out=SPEC.n_out, max_batch=20, seed=1)
    out = torch.empty((SPEC.L, len(ids), SPEC.S, SPEC.d), dtype=torch.bfloat16, device="cuda")
    ctx.gather(ids, out)
    ctx.sync()
    assert torch.equal(out, case.cache[torch.tensor(ids, device="cuda")].transpose(0, 1))
    ctx.close()
