"""Which kernels a call launches, read from the CUDA graph that captures it:
the rules that choose between kernels on size, at both sides of their lines,
for the number of SMs of the device that runs the test."""
import ctypes as C
import re

import pytest
import torch

from gpu_util import PRESETS, coins, dev, lwe, master_seeds

pytestmark = pytest.mark.gpu


class _KernelParams(C.Structure):  # cudaKernelNodeParams
    _fields_ = [("func", C.c_void_p), ("grid", C.c_uint * 3), ("block", C.c_uint * 3),
                ("smem", C.c_uint), ("params", C.c_void_p), ("extra", C.c_void_p)]


class _Edge(C.Structure):  # cudaGraphEdgeData
    _fields_ = [("from_port", C.c_ubyte), ("to_port", C.c_ubyte), ("type", C.c_ubyte),
                ("reserved", C.c_ubyte * 5)]


def launches(call):
    """(mangled kernel name, grid, early) of every kernel of one call, by
    capture; early: it may start before a kernel that it depends on has ended
    (a programmatic edge)."""
    rt = C.CDLL("libcudart.so.13")
    call()  # lazy set-up happens outside the capture
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(g):
        call()
    graph, n = C.c_void_p(g.raw_cuda_graph()), C.c_size_t()
    assert rt.cudaGraphGetNodes(graph, None, C.byref(n)) == 0
    nodes = (C.c_void_p * n.value)()
    assert rt.cudaGraphGetNodes(graph, nodes, C.byref(n)) == 0
    m = C.c_size_t()
    assert rt.cudaGraphGetEdges(graph, None, None, None, C.byref(m)) == 0
    tails, heads, data = (C.c_void_p * m.value)(), (C.c_void_p * m.value)(), (_Edge * m.value)()
    if m.value:
        assert rt.cudaGraphGetEdges(graph, tails, heads, data, C.byref(m)) == 0
    early = {heads[i] for i in range(m.value) if data[i].type == 1}  # programmatic
    out = []
    for node in nodes:
        kind, p, name = C.c_int(), _KernelParams(), C.c_char_p()
        assert rt.cudaGraphNodeGetType(C.c_void_p(node), C.byref(kind)) == 0
        if kind.value == 0:  # cudaGraphNodeTypeKernel
            assert rt.cudaGraphKernelNodeGetParams(C.c_void_p(node), C.byref(p)) == 0
            assert rt.cudaFuncGetName(C.byref(name), C.c_void_p(p.func)) == 0
            out.append((name.value.decode(), tuple(p.grid), node in early))
    return out


def grids(call, kernel):
    """The grids of the call's launches of `kernel` (any template instance)."""
    # after the name: template arguments, a namespace's end or a parameter type
    name_in = re.compile(kernel + r"(?=I|E|\d+[A-Z][a-z])")
    return [grid for name, grid, _ in launches(call) if name_in.search(name)]


def sms():
    torch.cuda.set_device(0)
    return torch.cuda.get_device_properties(0).multi_processor_count


def matmul_call(n, items, pair):
    """S A on the tensor cores: 8 items rows."""
    ctx = lwe.Ctx(lwe.Params(n=n, logq=16, B=2, clip=10, sigma=2.3), max_batch=items)
    ctx.set_path(lwe.PATH_TENSOR)
    if pair is not None:
        ctx.set_option(lwe.OPT_GEMM_PAIR, pair)
    A = torch.zeros((n, n), dtype=torch.int16, device="cuda")
    S = torch.zeros((8 * items, n), dtype=torch.int8, device="cuda")
    out = torch.empty((8 * items, n), dtype=torch.int16, device="cuda")
    return lambda: lwe.matmul_modq(lwe.SIDE_SA, S, out, n, 16, A=A, ctx=ctx)


@pytest.mark.parametrize("pair", [1, 0, -1, None])
@pytest.mark.parametrize("more", [0, 1])
def test_gemm_pair_option_selects_the_kernel(pair, more):
    """1 and 0 hold for every size; -1, the default, takes CTA pairs from more
    than SMs / 4 tiles of 256 x 128 on (128 columns: one tile per 32 items)."""
    n, tiles = 128, sms() // 4 + more
    call = matmul_call(n, 32 * tiles, pair)
    pairs, singles = len(grids(call, "k_gemm_sa2")), len(grids(call, "k_gemm_sa"))
    assert pairs + singles == 1
    assert pairs == (more if pair in (-1, None) else pair)


def kem_calls(n, count, path=lwe.PATH_AUTO, stored=True):
    """Encaps and Decaps of `count` items against a bound key."""
    ctx = lwe.Ctx(lwe.Params(**dict(PRESETS["P640"], n=n)), max_batch=count)
    ctx.set_path(path)
    pk, sk, ct = ctx.empty_pk(1), ctx.empty_sk(1), ctx.empty_ct(count)
    A = torch.empty((n, n), dtype=torch.int16, device="cuda") if stored else None
    ctx.keygen(dev(master_seeds(1, seed=n)), pk, sk, A_out=A)
    ctx.bind_key(pk, sk, A)
    cs = dev(coins(count, seed=n))
    K = torch.empty((count, 32), dtype=torch.uint8, device="cuda")
    return lambda: ctx.encaps(pk, cs, ct, K, A=A), lambda: ctx.decaps(sk, ct, K, A=A)


@pytest.mark.parametrize("n,count,stored,first", [
    (640, 8, True, True), (640, 64, True, True), (8192, 1, True, True), (976, 5, False, True),
    (640, 1, True, False), (1344, 200, True, False), (640, 30, False, False)])
def test_decaps_lets_its_hash_start_before_the_noise(n, count, stored, first):
    """Where the noise would fill every SM and the hash of the ciphertexts, on
    the other stream, needs few, the main chain's first kernel does not start
    beside the call before (its followers, and so the noise, may)."""
    encaps, decaps = kem_calls(n, count, stored=stored)

    def both():
        encaps()
        decaps()

    (early,) = [e for name, _, e in launches(both) if "9k_decrypt" in name]
    assert early != first


def test_leaf_launch_waits_for_the_kernel_before_it():
    """The leaves of a batch hashed in two launches are spread evenly over the
    SMs: the launch does not start beside the GEMM's last CTAs.  The roots do
    start beside the leaves."""
    encaps, _ = kem_calls(208, 33 * sms(), path=lwe.PATH_TENSOR)
    early = {name: e for name, _, e in launches(encaps)}
    assert [e for name, e in early.items() if "13k_tree_leaves" in name] == [False]
    assert [e for name, e in early.items() if "12k_tree_roots" in name] == [True]


@pytest.mark.parametrize("n,per_sm", [(16, 16), (400, 5), (640, 4), (976, 2), (1344, 2),
                                      (1600, 1.5), (2000, 1)])
def test_latency_tree_hash_stays_within_one_wave(n, per_sm):
    """H(c) runs three Keccak states per warp while its CTAs (or clusters of
    two, from n = 1600 on) are all resident, and not with one message more (n =
    16, one leaf each: 16 per SM)."""
    count = int(per_sm * sms())
    for items, warp in ((count, 1), (count + 1, 0)):
        encaps, _ = kem_calls(n, items)
        assert len(grids(encaps, "k_tree_warp")) == warp, items


@pytest.mark.parametrize("per_sm,kernel", [(27, "k_tree_bal"), (28, "k_tree"), (29, "k_tree_leaves")])
def test_tree_schedule_beyond_thirteen_leaf_warps(per_sm, kernel):
    """At n = 976 (15 full chunks and a short one) 27 messages per SM are 13
    leaf warps; 28 are one wave of k_tree; 29 are not."""
    encaps, _ = kem_calls(976, per_sm * sms())
    assert len(grids(encaps, kernel)) == 1


@pytest.mark.parametrize("per_sm,warps", [(3, 8), (3.01, 4), (5, 4), (5.01, 8)])
def test_stored_AS_takes_four_warps_where_they_are_one_wave(per_sm, warps):
    """A S with A stored: 16-row tiles per SM on both sides of the lines."""
    n = 16 * (int(per_sm) * sms() + (per_sm > int(per_sm)))
    A = torch.zeros((n, n), dtype=torch.int16, device="cuda")
    St = torch.zeros((8, n), dtype=torch.int8, device="cuda")
    out = torch.empty((n, 8), dtype=torch.int16, device="cuda")
    names = [name for name, _, _ in launches(lambda: lwe.matmul_modq(lwe.SIDE_AS, St, out, n, 16, A=A))]
    assert len(names) == 1 and "8k_mul_asILi%dE" % warps in names[0]


@pytest.mark.parametrize("n", [1344, 1600, 6208, 7200])
def test_regenerated_AS_split_counts_the_barriers(n):
    """One item's A S with A regenerated: one CTA per 16-row tile where that
    fills the rounds of the SMs well, not clusters whose barriers cost more
    than the even split gains (on 152 SMs)."""
    if sms() != 152:
        pytest.skip("sizes chosen for 152 SMs")
    seed = torch.zeros(16, dtype=torch.uint8, device="cuda")
    St = torch.zeros((8, n), dtype=torch.int8, device="cuda")
    out = torch.empty((n, 8), dtype=torch.int16, device="cuda")
    (grid,) = grids(lambda: lwe.matmul_modq(lwe.SIDE_AS, St, out, n, 16, seedA=seed),
                    "k_mul_as_gen_split")
    assert grid == (1, min(n // 16, sms()), 1)


@pytest.mark.parametrize("n,items", [(640, 20), (976, 5), (976, 10), (1344, 10), (2048, 5), (16384, 2)])
def test_stored_SA_split_fits_the_clusters_that_run_at_once(n, items):
    """S' A with A stored, a few items: the split does not count on CTAs that
    its clusters leave no room for (a seventh of the SMs for clusters of 7)."""
    if sms() != 152:
        pytest.skip("clusters counted on 152 SMs")
    A = torch.zeros((n, n), dtype=torch.int16, device="cuda")
    S = torch.zeros((8 * items, n), dtype=torch.int8, device="cuda")
    out = torch.empty((8 * items, n), dtype=torch.int16, device="cuda")
    (grid,) = grids(lambda: lwe.matmul_modq(lwe.SIDE_SA, S, out, n, 16, A=A), "k_sa")
    room = {2: 304, 3: 291, 4: 296, 5: 290, 6: 276, 7: 266, 8: 288}
    assert grid[1] == 1 or grid[0] * grid[1] * grid[2] <= room[grid[1]]
