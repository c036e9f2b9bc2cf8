"""The tree hash with ten threads per Keccak state (k_tree_warp, and
k_tree_leaves_tri + k_tree_roots for long messages) against hashlib, through
KeyGen's H(pk): messages of one chunk, of chunk counts that do and do not
divide by the three states of a warp, of more than one CTA, and of more than
96 chunks; one item and several."""
import hashlib

import numpy as np
import pytest
import torch

from gpu_util import dev, host, lwe, master_seeds, params

pytestmark = pytest.mark.gpu


def _tree(msg: bytes) -> bytes:
    leaves = [hashlib.sha3_256(msg[i:i + 1024]).digest() for i in range(0, len(msg), 1024)]
    return hashlib.sha3_256(b"".join(leaves)).digest()


@pytest.mark.parametrize("n,count", [(16, 1), (16, 700), (64, 5), (128, 2), (640, 7), (1344, 4),
                                     (1600, 1), (4096, 3), (6208, 1), (6208, 5), (10240, 2)])
def test_key_hash_matches_hashlib(n, count):
    torch.cuda.set_device(0)
    p, _ = params("P640", n=n)
    ctx = lwe.Ctx(p, max_batch=count)
    pk, sk = ctx.empty_pk(count), ctx.empty_sk(count)
    ctx.keygen(dev(master_seeds(count, seed=n)), pk, sk)
    pk_h, sk_h = host(pk), host(sk)
    for i in range(0, count, max(1, count // 16)):
        got = sk_h[i, 8 * n + 32:8 * n + 64].tobytes()
        assert got == _tree(pk_h[i].tobytes()), i
    ctx.close()


@pytest.mark.parametrize("n,count", [(400, 10700), (1344, 2900), (1344, 2750), (976, 3990),
                                     (640, 1501)])
def test_batch_schedules_agree_with_it(n, count):
    """Encaps' keys from the batched tree schedules (two launches for more than
    32 messages or 13 leaf warps per SM; the balanced and the dense one with
    their roots three per warp) equal those of one message per CTA; ragged
    last CTAs."""
    torch.cuda.set_device(0)
    p, _ = params("P640", n=n, logq=16)
    ctx = lwe.Ctx(p, max_batch=count)
    pk, sk = ctx.empty_pk(1), ctx.empty_sk(1)
    ctx.keygen(dev(master_seeds(1, seed=n)), pk, sk)
    coins = dev(np.random.default_rng(n).integers(0, 256, (count, 32), dtype=np.uint8))
    ct = ctx.empty_ct(count)
    keys = []
    for warp_max in (-1, count):
        K = torch.empty((count, 32), dtype=torch.uint8, device="cuda")
        ctx.set_option(lwe.OPT_WARP_HASH_MAX, warp_max)
        ctx.encaps(pk, coins, ct, K)
        keys.append(host(K))
    assert np.array_equal(keys[0], keys[1])
    assert ctx.device_error() == 0
    ctx.close()


def test_one_wave_of_k_tree_agrees_with_it():
    """28 messages of 16 chunks per SM, more leaves than the packed schedules
    take (k_tree, its last CTA ragged): Encaps' keys and Decaps' equal those of
    one message per CTA."""
    torch.cuda.set_device(0)
    count = 28 * torch.cuda.get_device_properties(0).multi_processor_count - 5
    p, _ = params("P976")
    ctx = lwe.Ctx(p, max_batch=count)
    pk, sk = ctx.empty_pk(1), ctx.empty_sk(1)
    ctx.keygen(dev(master_seeds(1, seed=28)), pk, sk)
    coins = dev(np.random.default_rng(28).integers(0, 256, (count, 32), dtype=np.uint8))
    ct = ctx.empty_ct(count)
    keys = []
    for warp_max in (-1, count):
        K, K2 = (torch.empty((count, 32), dtype=torch.uint8, device="cuda") for _ in range(2))
        ctx.set_option(lwe.OPT_WARP_HASH_MAX, warp_max)
        ctx.encaps(pk, coins, ct, K)
        ctx.decaps(sk, ct, K2)
        keys += [host(K), host(K2)]
    for k in keys[1:]:
        assert np.array_equal(keys[0], k)
    assert ctx.device_error() == 0
    ctx.close()
