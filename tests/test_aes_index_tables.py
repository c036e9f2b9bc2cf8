"""The per-byte tables of the product kernels' AES counter blocks (aes_f_entry
and aes_f_start in csrc/aes.cuh) restated in Python: for indices below 2^32
the state after round 2 is the XOR of four table entries, one per index byte.
Checked against the oracle's AES-CTR block for random keys and for indices
whose bytes are 0 or 255 or cross 2^16 and 2^24."""
import random

from oracle import oracle as O
from test_aes_window import T, bswap, key_expand, rounds_from


def entry(rk, domain, j, x):
    """F_j[x]: index byte j (0 the lowest) in column j of round 1, its four
    terms of round 2 (with round key 2 in F_3)."""
    s = [bswap(domain >> 32) ^ rk[0], bswap(domain & 0xFFFFFFFF) ^ rk[1], rk[2],
         rk[3] ^ (x << (8 * (3 - j)))]
    t = (T(0, 0, s[j]) ^ T(1, 1, s[(j + 1) % 4]) ^ T(2, 2, s[(j + 2) % 4])
         ^ T(3, 3, s[(j + 3) % 4]) ^ rk[4 + j])
    # column j feeds output column c = j - k through T_k
    out = [T((j - c) % 4, (j - c) % 4, t) for c in range(4)]
    return [v ^ (rk[8 + c] if j == 3 else 0) for c, v in enumerate(out)]


def test_index_byte_tables_equal_the_oracle():
    rng = random.Random(9)
    for trial in range(12):
        key = bytes(rng.randrange(256) for _ in range(16))
        domain = rng.choice([0, 0, 3, rng.randrange(1 << 64)])
        rk = key_expand(key)
        for index in [0, 255, 256, 0xFFFF, 0x10000, 0xFFFFFF, 0x1000000, (1 << 29) - 1,
                      0xFFFFFFFF] + [rng.randrange(1 << 32) for _ in range(3)]:
            s = [0, 0, 0, 0]
            for j in range(4):
                s = [a ^ b for a, b in zip(s, entry(rk, domain, j, (index >> (8 * j)) & 0xFF))]
            ref = O.ctr_stream(key, domain, index, 1).tobytes()
            assert rounds_from(rk, tuple(s), 3) == ref, (trial, index)
