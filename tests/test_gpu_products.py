"""The products of one request (csrc/products.cuh) against the oracle, bit for
bit, at the sizes where their tiles can go wrong: n below one tile, row counts
that are odd multiples of 16 (the second half of a 32-row tile absent, an odd
number of 16-row steps), column counts that are no multiple of a 32-column
chunk group or a 64-column group, S of the full int8 range, and the schedule
for many regenerated items."""
import numpy as np
import pytest
import torch

from gpu_util import O, as_u16, dev, host, lwe, master_seeds, params
from test_gpu_dispatch import grids

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _device():
    assert torch.cuda.is_available()
    torch.cuda.set_device(0)


@pytest.mark.parametrize("n", [16, 48, 80, 640, 976, 1008, 2064, 4112])
@pytest.mark.parametrize("stored", [True, False])
@pytest.mark.parametrize("logq,k,amp", [(16, 8, 12), (15, 24, 127)])
def test_products_match_oracle(n, stored, logq, k, amp):
    r = np.random.default_rng(n + k)
    seed = r.integers(0, 256, 16, dtype=np.uint8)
    A_o = O.expand_A(bytes(seed), n, logq)
    St = r.integers(-amp - 1, amp + 1, size=(8, n)).astype(np.int8)
    E = r.integers(-amp - 1, amp + 1, size=(n, 8)).astype(np.int8)
    S = r.integers(-amp - 1, amp + 1, size=(k, n)).astype(np.int8)
    E2 = r.integers(-amp - 1, amp + 1, size=(k, n)).astype(np.int8)
    A = dev(A_o.view(np.int16)) if stored else None
    sd = None if stored else dev(seed)
    out = torch.empty((n, 8), dtype=torch.int16, device="cuda")
    lwe.matmul_modq(lwe.SIDE_AS, dev(St), out, n, logq, A=A, seedA=sd, E=dev(E))
    assert np.array_equal(as_u16(out), O.mul_AS(A_o, St, E, logq))
    out2 = torch.empty((k, n), dtype=torch.int16, device="cuda")
    lwe.matmul_modq(lwe.SIDE_SA, dev(S), out2, n, logq, A=A, seedA=sd, E=dev(E2))
    assert np.array_equal(as_u16(out2), O.mul_SA(S, A_o, E2, logq))


@pytest.mark.parametrize("n,count", [(304, 250), (16, 2500), (640, 130)])
def test_many_regenerated_items_match_oracle(n, count):
    """Enough row tiles that a warp takes whole tiles (k_mul_as_gen); at n =
    16 a CTA's range spans more items than it holds tables for."""
    p, po = params("P640", n=n)
    ctx = lwe.Ctx(p, max_batch=count)
    ms = master_seeds(count, seed=n)
    pk, sk = ctx.empty_pk(count), ctx.empty_sk(count)
    ctx.keygen(dev(ms), pk, sk)
    pk_h, sk_h = host(pk), host(sk)
    for i in list(range(0, count, max(1, count // 40))) + [count - 1]:
        pk_o, sk_o = O.keygen(po, bytes(ms[i]))
        assert np.array_equal(pk_h[i], pk_o), i
        assert np.array_equal(sk_h[i], sk_o), i
    ctx.close()


@pytest.mark.parametrize("n", [512, 528, 4112])
def test_products_exact_at_the_largest_sums(n):
    """Every byte of A 255 and S = -128: the accumulators reach their bound,
    512 terms of 255 x 128 below 2^24, and are emptied in time beyond it."""
    A = np.full((n, n), 0xFFFF, dtype=np.uint16)
    S = np.full((8, n), -128, dtype=np.int8)
    S[1::2] = 127
    A_d = dev(A.view(np.int16))
    out = torch.empty((n, 8), dtype=torch.int16, device="cuda")
    lwe.matmul_modq(lwe.SIDE_AS, dev(S), out, n, 16, A=A_d)
    assert np.array_equal(as_u16(out), O.mul_AS(A, S, None, 16))
    out2 = torch.empty((8, n), dtype=torch.int16, device="cuda")
    lwe.matmul_modq(lwe.SIDE_SA, dev(S), out2, n, 16, A=A_d)
    assert np.array_equal(as_u16(out2), O.mul_SA(S, A, None, 16))


@pytest.mark.parametrize("n", [7312, 8192])
def test_stored_AS_of_one_wave_matches_exact_sums(n):
    """The 4-warp instance of the stored A S (more than three 16-row tiles
    per SM), whose column stride of 128 chunks n = 7312 is no multiple of:
    against whole-number sums in 64-bit floating point."""
    g = torch.Generator(device="cuda")
    g.manual_seed(n)
    A = torch.randint(0, 65536, (n, n), generator=g, device="cuda", dtype=torch.int32).to(torch.int16)
    St = torch.randint(-128, 128, (8, n), generator=g, device="cuda", dtype=torch.int8)
    E = torch.randint(-128, 128, (n, 8), generator=g, device="cuda", dtype=torch.int8)
    out = torch.empty((n, 8), dtype=torch.int16, device="cuda")
    lwe.matmul_modq(lwe.SIDE_AS, St, out, n, 16, A=A, E=E)
    exact = (A.to(torch.int32) & 0xFFFF).to(torch.float64) @ St.to(torch.float64).T
    exact = (exact.to(torch.int64) + E.long()) & 0xFFFF
    assert np.array_equal(as_u16(out).astype(np.int64), host(exact))


@pytest.mark.parametrize("n", [16, 304])
def test_items_beyond_the_tables_a_cta_holds_match_oracle(n):
    """KeyGen of so many items that a warp takes whole row tiles (at least 32
    per SM).  n = 16, one tile each: a CTA's range spans 33 or 34 items, nine
    rounds of the four keys whose tables it holds; n = 304, 19 tiles: ranges
    begin inside an item.  The items at both sides of the CTAs' and of the
    rounds' boundaries."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    tiles = n // 16
    count = -(-33 * sms // tiles) + 7
    p, po = params("P640", n=n)
    ctx = lwe.Ctx(p, max_batch=count)
    ms = master_seeds(count, seed=n + 1)
    seeds, pk, sk = dev(ms), ctx.empty_pk(count), ctx.empty_sk(count)
    ctx.keygen(seeds, pk, sk)
    assert len(grids(lambda: ctx.keygen(seeds, pk, sk), "k_mul_as_gen")) == 1
    pk_h, sk_h = host(pk), host(sk)
    units, check = count * tiles, {0, count - 1}
    for b in (0, 1, 2, sms // 2, sms - 1):
        first, last = units * b // sms // tiles, (units * (b + 1) // sms - 1) // tiles
        check |= {i for i in range(first - 1, first + 10)} | {last - 1, last, last + 1}
    for i in sorted(i for i in check if 0 <= i < count):
        pk_o, sk_o = O.keygen(po, bytes(ms[i]))
        assert np.array_equal(pk_h[i], pk_o), i
        assert np.array_equal(sk_h[i], sk_o), i
    ctx.close()
