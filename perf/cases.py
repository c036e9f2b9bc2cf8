"""The calls whose time counts, as data: what a user of this library has it do,
through the Python binding, from one request to a batch that fills the GPU.

A case is a dict of plain values.  Its "kind" says which entry points a pass
goes through:

  request   one request: (KeyGen,) Encaps and Decaps with count = 1, A
            regenerated from its seed or stored, the key bound or not
  keygen    a batch of key pairs in one call, A regenerated
  multi     Encaps and Decaps of a batch of requests for different keys
            (per-item key pointers), as the server issues them
  batch     Encaps of a batch against one key, then the Decaps of it
  graph     the same through BatchedKem: key bound, replayed CUDA graph
  expand    A from its 16-byte seed into device memory
  product   A S + E and S' A + E' on their own, A stored or regenerated
  pp        the paper's own parameter profile: KeyGen, Encaps, Decaps

Outputs are the bytes and words that the calls write: public and secret keys,
ciphertexts, session keys, A, products.
"""
import numpy as np
import torch

from paper_2606_01211_gb300 import batch, lwe
from paper_2606_01211_gb300.inputs import PRESETS

DEV = "cuda"


def preset(name, **more):
    return dict(PRESETS[name], **more)


def listed():
    return [
        # one client asking for everything once, nothing known beforehand:
        # the smallest calls, all latency
        dict(name="request_n640", kind="request", keygen=True, stored=False, bound=False,
             **preset("P640")),
        # one request at a time against a long-lived key (bound, A resident)
        dict(name="request_n1344_bound", kind="request", keygen=False, stored=True, bound=True,
             **preset("P1344")),
        # a dimension no CPU serves, with A too large to keep for one key
        dict(name="request_n32768_seed", kind="request", keygen=False, stored=False, bound=False,
             **preset("P32768")),
        # provisioning: key pairs made in a batch of no round size
        dict(name="keygen_n976_x250", kind="keygen", count=250, **preset("P976")),
        # a server's dispatch: requests for many keys, most of them distinct
        dict(name="multi_n976_x61", kind="multi", count=61, keys=48, stored=True,
             **preset("P976")),
        # a hot key's queue, emptied as it stands: ragged, key not bound
        dict(name="batch_n640_x777", kind="batch", count=777, stored=True, bound=False,
             **preset("P640")),
        # the headline workload: 4096 Encaps and their Decaps, graph replayed
        dict(name="graph_n976_x4096", kind="graph", preset="P976", count=4096),
        # large n in a batch: the product dominates
        dict(name="batch_n16384_x1024", kind="batch", count=1024, stored=True, bound=False,
             **preset("P16384")),
        # filling a cache of expanded A
        dict(name="expand_n4096", kind="expand", n=4096, logq=16),
        # the hot kernels on their own, A streamed from memory
        dict(name="product_n8192_stored", kind="product", n=8192, logq=16, rows=8, clip=12,
             stored=True),
        # and with A made on the fly
        dict(name="product_n4096_seed", kind="product", n=4096, logq=16, rows=8, clip=12,
             stored=False),
        # the scheme as the paper states it: odd q, 256 message bits
        dict(name="pp_n4096", kind="pp", preset="PP4096", bound=False),
    ]


def spread(rng, lo, hi, step=1):
    """A whole number of lo .. hi, even over the logarithm, a multiple of step."""
    v = lo * (hi / lo) ** rng.random()
    return int(min(hi, max(lo, round(v / step) * step)))


def draw(rng):
    kind = rng.choice(["request", "request", "keygen", "multi", "multi", "batch", "batch", "graph",
                       "expand", "product", "product", "pp"])
    like = dict(PRESETS[rng.choice(["P640", "P976", "P1344", "P4096"])])
    if kind == "request":
        n = spread(rng, 640, 8192, 16)
        return dict(like, kind=kind, n=n, keygen=rng.random() < 0.5, stored=rng.random() < 0.5,
                    bound=rng.random() < 0.5)
    if kind == "keygen":
        return dict(like, kind=kind, n=spread(rng, 640, 2048, 16), count=spread(rng, 2, 512))
    if kind == "multi":
        count = spread(rng, 2, 256)
        return dict(like, kind=kind, n=spread(rng, 640, 4096, 16), count=count,
                    keys=min(count, spread(rng, 1, 64)), stored=rng.random() < 0.6)
    if kind == "batch":
        n = spread(rng, 640, 4096, 16)
        return dict(like, kind=kind, n=n, count=spread(rng, 24, 4096 if n <= 1344 else 1024),
                    stored=rng.random() < 0.7, bound=rng.random() < 0.5)
    if kind == "graph":  # BatchedKem takes the named parameter sets
        name = rng.choice(["P640", "P976", "P1344", "P4096"])
        return dict(kind=kind, preset=name,
                    count=spread(rng, 64, 1024 if name == "P4096" else 4096))
    if kind == "expand":
        return dict(kind=kind, n=spread(rng, 640, 16384, 16), logq=rng.choice([15, 16]))
    if kind == "product":
        stored = rng.random() < 0.5
        return dict(kind=kind, n=spread(rng, 640, 16384 if stored else 8192, 16),
                    logq=rng.choice([15, 16]), rows=8 * rng.choice([1, 1, 2, 5]),
                    clip=rng.choice([6, 10, 12]), stored=stored)
    return dict(kind="pp", preset=rng.choice(["PP512", "PP1024", "PP2048", "PP4096", "PP8192"]),
                bound=rng.random() < 0.5)


# ---- inputs -----------------------------------------------------------------
def _random(seed):
    return np.random.Generator(np.random.PCG64(seed))


def _bytes(g, *shape):
    return torch.from_numpy(g.integers(0, 256, size=shape, dtype=np.uint8)).to(DEV)


def _params(case):
    return lwe.Params(n=case["n"], logq=case["logq"], B=case["B"], clip=case["clip"],
                      sigma=case["sigma"])


def _small(g, clip, *shape):
    """Entries of a rounded Gaussian's shape, |x| <= clip, as int8."""
    x = np.clip(np.rint(g.standard_normal(shape, dtype=np.float32) * (clip / 4.3)), -clip, clip)
    return torch.from_numpy(x.astype(np.int8)).to(DEV)


def _uniform_A(g, n, logq):
    t = torch.Generator(device=DEV)
    t.manual_seed(int(g.integers(0, 2**62)))
    return torch.randint(0, 1 << logq, (n, n), generator=t, device=DEV,
                         dtype=torch.int32).to(torch.int16)


def prepare(case, seed):
    g = _random(seed)
    kind, s = case["kind"], {"case": case}
    if kind in ("request", "keygen", "multi", "batch"):
        p = _params(case)
        count = case.get("count", 1)
        ctx = lwe.Ctx(p, max_batch=count)
        s.update(ctx=ctx, seeds=_bytes(g, count, 32), coins=_bytes(g, count, 32),
                 ct=ctx.empty_ct(count), K=torch.empty((count, 32), dtype=torch.uint8, device=DEV),
                 K2=torch.empty((count, 32), dtype=torch.uint8, device=DEV))
    if kind == "keygen" or (kind == "request" and case["keygen"]):
        s.update(pk=ctx.empty_pk(count), sk=ctx.empty_sk(count), A=None)
        if kind == "request" and case["stored"]:
            s["A"] = torch.empty((p.n, p.n), dtype=torch.int16, device=DEV)
    elif kind in ("request", "batch"):
        s.update(pk=ctx.empty_pk(1), sk=ctx.empty_sk(1), A=None)
        if case["stored"]:
            s["A"] = torch.empty((p.n, p.n), dtype=torch.int16, device=DEV)
        ctx.keygen(s["seeds"][:1], s["pk"], s["sk"], A_out=s["A"])
    if kind in ("request", "batch") and case["bound"] and not case.get("keygen"):
        ctx.bind_key(s["pk"], s["sk"], s["A"])
    elif kind == "multi":
        keys = case["keys"]
        kctx = lwe.Ctx(p, max_batch=keys)
        s.update(pk=kctx.empty_pk(keys), sk=kctx.empty_sk(keys), A=None)
        if case["stored"]:
            s["A"] = torch.empty((keys, p.n, p.n), dtype=torch.int16, device=DEV)
        kctx.keygen(_bytes(g, keys, 32), s["pk"], s["sk"], A_out=s["A"])
        torch.cuda.synchronize()
        kctx.close()
        who = g.integers(0, keys, size=count)
        at = lambda base, step, off=0: torch.from_numpy(base + off + step * who).to(DEV)  # noqa: E731
        s.update(pk_ptrs=at(s["pk"].data_ptr(), p.pk_bytes),
                 sk_ptrs=at(s["sk"].data_ptr(), p.sk_bytes),
                 pkh_ptrs=at(s["sk"].data_ptr(), p.sk_bytes, 8 * p.n + 32),
                 A_ptrs=at(s["A"].data_ptr(), 2 * p.n * p.n) if case["stored"] else None)
    elif kind == "graph":
        kem = batch.BatchedKem(case["preset"], case["count"], seed=int(g.integers(0, 2**31)))
        kem.capture()
        s.update(kem=kem, coins=_bytes(g, case["count"], 32))
    elif kind == "expand":
        n = case["n"]
        s.update(seed=_bytes(g, 16), A=torch.empty((n, n), dtype=torch.int16, device=DEV))
    elif kind == "product":
        n, k = case["n"], case["rows"]
        s.update(St=_small(g, case["clip"], 8, n), E=_small(g, case["clip"], n, 8),
                 S=_small(g, case["clip"], k, n), E2=_small(g, case["clip"], k, n),
                 out=torch.empty((n, 8), dtype=torch.int16, device=DEV),
                 out2=torch.empty((k, n), dtype=torch.int16, device=DEV), A=None, seedA=None)
        if case["stored"]:
            s["A"] = _uniform_A(g, n, case["logq"])
        else:
            s["seedA"] = _bytes(g, 16)
    elif kind == "pp":
        p = lwe.PpParams(case["preset"])
        ctx = lwe.PpCtx(p)
        s.update(ctx=ctx, seed=_bytes(g, 32), coins=_bytes(g, 32), pk=ctx.empty_pk(),
                 sk=ctx.empty_sk(), A=ctx.empty_A(), ct=ctx.empty_ct(),
                 K=torch.empty(32, dtype=torch.uint8, device=DEV),
                 K2=torch.empty(32, dtype=torch.uint8, device=DEV))
        if case["bound"]:
            ctx.keygen(s["seed"], s["pk"], s["sk"], s["A"])
            ctx.bind_key(s["pk"], s["A"])
    return s


# ---- one pass ---------------------------------------------------------------
def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind in ("request", "batch"):
        ctx, made = s["ctx"], {}
        if case.get("keygen"):
            ctx.keygen(s["seeds"], s["pk"], s["sk"], A_out=s["A"])
            made = {"pk": s["pk"], "sk": s["sk"]}
        ctx.encaps(s["pk"], s["coins"], s["ct"], s["K"], A=s["A"])
        ctx.decaps(s["sk"], s["ct"], s["K2"], A=s["A"])
        return dict(made, ct=s["ct"], K=s["K"], K2=s["K2"])
    if kind == "keygen":
        s["ctx"].keygen(s["seeds"], s["pk"], s["sk"])
        return {"pk": s["pk"], "sk": s["sk"]}
    if kind == "multi":
        s["ctx"].encaps_multi(s["pk_ptrs"], s["coins"], s["ct"], s["K"], pkh_ptrs=s["pkh_ptrs"],
                              A_ptrs=s["A_ptrs"])
        s["ctx"].decaps_multi(s["sk_ptrs"], s["ct"], s["K2"], A_ptrs=s["A_ptrs"])
        return {"ct": s["ct"], "K": s["K"], "K2": s["K2"]}
    if kind == "graph":
        kem = s["kem"]
        kem.replay(s["coins"])
        return {"ct": kem.ct, "K": kem.K, "K2": kem.K2}
    if kind == "expand":
        lwe.expand_A(s["seed"], case["n"], case["logq"], s["A"])
        return {"A": s["A"]}
    if kind == "product":
        n, logq = case["n"], case["logq"]
        lwe.matmul_modq(lwe.SIDE_AS, s["St"], s["out"], n, logq, A=s["A"], seedA=s["seedA"],
                        E=s["E"])
        lwe.matmul_modq(lwe.SIDE_SA, s["S"], s["out2"], n, logq, A=s["A"], seedA=s["seedA"],
                        E=s["E2"])
        return {"AS": s["out"], "SA": s["out2"]}
    ctx, made = s["ctx"], {}
    if not case["bound"]:
        ctx.keygen(s["seed"], s["pk"], s["sk"], s["A"])
        made = {"pk": s["pk"], "sk": s["sk"], "A": s["A"]}
    ctx.encaps(s["pk"], s["A"], s["coins"], s["ct"], s["K"])
    ctx.decaps(s["sk"], s["A"], s["ct"], s["K2"])
    return dict(made, ct=s["ct"], K=s["K"], K2=s["K2"])


# ---- what a pass cannot do without ------------------------------------------
def work(case):
    """Bytes of inputs and outputs, each once, and the operations (multiply
    and add) of the products mod q; hashing and AES are neither."""
    kind = case["kind"]
    if kind == "expand":
        return {"bytes": 16 + 2 * case["n"] ** 2, "flops": 0}
    if kind == "product":
        n, k = case["n"], case["rows"]
        a = 2 * n * n if case["stored"] else 16
        return {"bytes": a + 8 * n * (1 + 1 + 2) + k * n * (1 + 1 + 2),
                "flops": 2 * n * n * (8 + k)}
    if kind == "pp":
        n = lwe.PpParams(case["preset"]).n
        ct, keys = 1024 * n + 1024, 9 * n + 96  # pk and sk together
        return {"bytes": (4 if case["bound"] else 8) * n * n + 2 * ct
                + keys * (1 if case["bound"] else 2),
                "flops": 4 * 256 * n * (n + 2) + (0 if case["bound"] else 2 * n * n)}
    n, count = PRESETS[case["preset"]]["n"] if kind == "graph" else case["n"], case.get("count", 1)
    pk, sk, ct = 16 * n + 16, 24 * n + 80, 16 * n + 128
    made = {"bytes": count * (32 + pk + sk), "flops": count * 16 * n * n}
    if kind == "keygen":
        return made
    keys = case.get("keys", 1)
    stored = kind == "graph" or case["stored"]
    w = {"bytes": keys * (pk + sk + (2 * n * n if stored else 0)) + count * (2 * ct + 32 + 64),
         "flops": count * 2 * (2 * 8 * n * (n + 8)) + count * 128 * n}
    if case.get("keygen"):
        w = {k: w[k] + made[k] for k in w}
    return w


# ---- the same by other means ------------------------------------------------
def _sbox():
    """S(x) of FIPS-197: the affine map of the inverse in GF(2^8)."""
    log, alog, x = [0] * 256, [0] * 255, 1
    for i in range(255):
        alog[i], log[x] = x, i
        x ^= (x << 1) ^ (0x11B if x & 0x80 else 0)
        x &= 0xFF
    box = []
    for v in range(256):
        b = alog[(255 - log[v]) % 255] if v else 0
        y = b
        for r in range(1, 5):
            y ^= ((b << r) | (b >> (8 - r))) & 0xFF
        box.append(y ^ 0x63)
    return np.array(box, dtype=np.uint8)


def _aes_ctr_A(seed16, n, logq):
    """A: entry words of the AES-128 counter stream of domain 0, block
    (i n + j) / 8, masked to logq bits; plain byte-wise AES."""
    box = _sbox()
    key = [list(seed16[4 * i:4 * i + 4]) for i in range(4)]
    rcon = 1
    for i in range(4, 44):
        t = list(key[i - 1])
        if i % 4 == 0:
            t = [int(box[b]) for b in t[1:] + t[:1]]
            t[0] ^= rcon
            rcon = ((rcon << 1) ^ (0x11B if rcon & 0x80 else 0)) & 0xFF
        key.append([a ^ b for a, b in zip(key[i - 4], t)])
    rk = torch.tensor(key, dtype=torch.uint8, device=DEV).reshape(11, 16)
    S = torch.from_numpy(box).to(DEV)
    shift = torch.tensor([(r + 4 * ((c + r) % 4)) for c in range(4) for r in range(4)], device=DEV)
    nblk, parts = n * n // 8, []
    for b0 in range(0, nblk, 1 << 20):
        idx = torch.arange(b0, min(nblk, b0 + (1 << 20)), device=DEV, dtype=torch.int64)
        st = torch.zeros((len(idx), 16), dtype=torch.uint8, device=DEV)
        for i in range(8):
            st[:, 15 - i] = ((idx >> (8 * i)) & 0xFF).to(torch.uint8)
        st ^= rk[0]
        for r in range(1, 11):
            st = S[st.long()][:, shift]
            if r < 10:
                m = st.reshape(-1, 4, 4)
                twice = (m << 1) ^ ((m >> 7) * 0x1B)
                rot = lambda v, k: torch.roll(v, -k, dims=2)  # noqa: E731
                st = (twice ^ rot(twice, 1) ^ rot(m, 1) ^ rot(m, 2) ^ rot(m, 3)).reshape(-1, 16)
            st = st ^ rk[r]
        parts.append(st)
    words = torch.cat(parts).reshape(n, n, 2).to(torch.int32)
    return (words[..., 0] | (words[..., 1] << 8)) & ((1 << logq) - 1)


def exact(case, seed):
    """The products and A in 64 bits (every sum is a whole number below 2^53);
    None for the key exchanges, whose results are bytes of hashes."""
    if case["kind"] not in ("expand", "product"):
        return None
    s = prepare(case, seed)
    n, logq = case["n"], case["logq"]
    if case["kind"] == "expand":
        return {"A": _aes_ctr_A(s["seed"].cpu().tolist(), n, logq).to(torch.int16)}
    if case["stored"]:
        A = s["A"].to(torch.int32) & 0xFFFF
    else:
        A = _aes_ctr_A(s["seedA"].cpu().tolist(), n, logq)
    A = A.to(torch.float64)
    mask = (1 << logq) - 1
    AS = (A @ s["St"].to(torch.float64).T).to(torch.int64) + s["E"].long()
    SA = (s["S"].to(torch.float64) @ A).to(torch.int64) + s["E2"].long()
    return {"AS": (AS & mask).to(torch.int16), "SA": (SA & mask).to(torch.int16)}
