"""Decaps' mismatch flags do not outlive a call: the derivation clears them,
one store per item, in its kernel for few items (up to 8 per SM, four to a
CTA) and in the one for many, in lwe_decaps and lwe_decaps_multi.  A call that
rejects every item is followed by one whose items are all valid, and by one
with fewer items."""
import numpy as np
import pytest
import torch

from gpu_util import coins, dev, host, lwe, master_seeds, params

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("per_sm", [0, 8.5])
@pytest.mark.parametrize("multi", [False, True])
def test_valid_items_after_a_call_that_rejected_all(per_sm, multi):
    torch.cuda.set_device(0)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    count = int(per_sm * sms) or 7
    p, _ = params("P640", n=64)
    ctx = lwe.Ctx(p, max_batch=count)
    pk, sk, ct = ctx.empty_pk(1), ctx.empty_sk(1), ctx.empty_ct(count)
    ctx.keygen(dev(master_seeds(1, seed=5)), pk, sk)
    K = torch.empty((count, 32), dtype=torch.uint8, device="cuda")
    ctx.encaps(pk, dev(coins(count, seed=5)), ct, K)
    bad = ct.clone()
    bad[:, 3] ^= 64
    sk_ptrs = torch.full((count,), sk.data_ptr(), dtype=torch.int64, device="cuda")

    def decaps(c):
        out = torch.empty((len(c), 32), dtype=torch.uint8, device="cuda")
        if multi:
            ctx.decaps_multi(sk_ptrs[:len(c)], c, out)
        else:
            ctx.decaps(sk, c, out)
        return host(out)

    K_h = host(K)
    for items in (count, count - 2):
        assert not (decaps(bad) == K_h).all(axis=1).any()
        assert np.array_equal(decaps(ct[:items]), K_h[:items])
    ctx.close()
