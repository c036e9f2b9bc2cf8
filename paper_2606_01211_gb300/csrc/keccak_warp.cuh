// keccak_warp.cuh -- Keccak-f[1600] and SHA3-256 (FIPS 202) with three states
// per warp, ten threads each, for hashes whose latency counts: launches of
// few messages, the roots of long ones, the derivations of one request.
//
// Thread r < 10 of a group holds half h = r % 2 of five lanes, bit-interleaved
// (h = 0: the even bits of each 64-bit lane, h = 1: the odd ones), so that a
// 64-bit rotation is one 32-bit rotation and, for odd offsets, a swap of the
// halves, which the shuffle that moves the lane anyway absorbs.  In theta the
// five lanes are a column (x = r / 2), so its parity is local and only C[x - 1]
// and C[x + 1] are fetched; rho and pi then move five lanes into a row (y = r /
// 2), chi and iota are local there, and five shuffles bring the columns back:
// 12 32-bit shuffles in three dependent stages and about 30 ALU instructions
// a round for three states.  Bound by the shuffle latency (about 28 clocks
// each, and 4 for every further one of a stage).  With one lane of one state
// per thread (18 shuffles in four stages) a round took 227 clocks alone and
// 345 with 16 warps on the SM; this takes 167 and 284 for three states.  One
// state per thread (keccak.cuh) needs 384 for 32 states, so it keeps the
// batches that fill it.
//
// A shuffle publishes one register index for all its source threads, but the
// lane that rho/pi or the way back wants sits at an index that depends on the
// thread.  The lanes are therefore numbered diagonally, column form: register
// i = lane (x, b x + i), row form: register j = lane (a y + j, y), indices mod
// 5.  pi (x = X + 3 Y, y = X) then reads register (1 - b) j for every thread
// if (1 - b) a = 3 b, and the way back register -a i if a b' = 1 for the next
// round's b'.  That gives b = 3, 2, 4 with a = 3, 4, 1 in turn; the third way
// back would need b' = 1, which has no a, so there the row is first rotated
// by y (15 selects) to return to b = 3.
#pragma once
#include "keccak.cuh"

// iota's constants, bit-interleaved: entry 2 r + h (the bits h, h + 2, ... of
// round r's constant)
struct KeccakRcHalves {
  uint32_t v[48];
};
constexpr KeccakRcHalves keccak_rc_halves() {
  constexpr uint64_t rc[24] = {KECCAK_RC};
  KeccakRcHalves t{};
  for (int r = 0; r < 24; r++)
    for (int h = 0; h < 2; h++) {
      uint32_t w = 0;
      for (int b = 0; b < 32; b++) w |= (uint32_t)((rc[r] >> (2 * b + h)) & 1) << b;
      t.v[2 * r + h] = w;
    }
  return t;
}
__constant__ KeccakRcHalves kKeccakRcHalves = keccak_rc_halves();

struct KeccakTri {
  uint32_t grp;            // this thread's state (0..2)
  uint32_t r, x, h;        // thread of the group; column (row) and half
  uint32_t rot[3][5];      // rho of register i, by form b
  uint32_t src[3][5];      // pi: source thread of row register j
  uint32_t back[3][5];     // the way back: source thread of column register i
  uint32_t cm, cp, cp_rot; // C[x - 1]; C[x + 1] rotated by 1
  uint32_t row0;           // all-ones on row 0 (iota)
};

// rho offset of lane i = x + 5y: (t + 1)(t + 2) / 2 mod 64 where (x, y) is
// reached at step t of the walk (1, 0) -> (y, 2x + 3y); lane 0 has none.
constexpr uint32_t keccak_rho_offset(uint32_t i) {
  uint32_t x = 1, y = 0;
  for (uint32_t t = 0; t < 24; t++) {
    if (x + 5 * y == i) return ((t + 1) * (t + 2) / 2) % 64;
    const uint32_t nx = y, ny = (2 * x + 3 * y) % 5;
    x = nx;
    y = ny;
  }
  return 0;
}
// The offsets of column x, 6 bits per lane, and the odd ones of all 25 lanes:
// immediates, as tables in memory indexed per thread cost microseconds of
// set-up in each launch.
constexpr uint32_t keccak_rho_column(uint32_t x) {
  uint32_t v = 0;
  for (uint32_t y = 0; y < 5; y++) v |= keccak_rho_offset(x + 5 * y) << (6 * y);
  return v;
}
constexpr uint32_t keccak_rho_odd() {
  uint32_t v = 0;
  for (uint32_t i = 0; i < 25; i++) v |= (keccak_rho_offset(i) & 1u) << i;
  return v;
}

constexpr uint32_t kRhoCol0 = keccak_rho_column(0), kRhoCol1 = keccak_rho_column(1),
                   kRhoCol2 = keccak_rho_column(2), kRhoCol3 = keccak_rho_column(3),
                   kRhoCol4 = keccak_rho_column(4), kRhoOdd = keccak_rho_odd();

// The thread constants; lanes 30 and 31 mirror lanes 20 and 21.
LWE_DEV KeccakTri keccak_tri(uint32_t lane) {
  constexpr uint32_t B[3] = {3, 2, 4}, A[3] = {3, 4, 1}, NB[3] = {2, 4, 3};
  const uint32_t l = lane < 30 ? lane : lane - 10;
  KeccakTri m;
  m.grp = l / 10;
  m.r = l % 10;
  m.x = m.r >> 1;
  m.h = m.r & 1;
  const uint32_t base = 10 * m.grp, x = m.x, h = m.h;
  const uint32_t col =
      x == 0 ? kRhoCol0 : (x == 1 ? kRhoCol1 : (x == 2 ? kRhoCol2 : (x == 3 ? kRhoCol3 : kRhoCol4)));
#pragma unroll
  for (uint32_t k = 0; k < 3; k++) {
#pragma unroll
    for (uint32_t i = 0; i < 5; i++) {
      const uint32_t y = (B[k] * x + i) % 5;
      m.rot[k][i] = (((col >> (6 * y)) & 63u) + h) >> 1;
      const uint32_t X = (A[k] * x + i) % 5, sx = (X + 3 * x) % 5;  // row x, lane (X, x)
      m.src[k][i] = base + 2 * sx + (h ^ ((kRhoOdd >> (sx + 5 * X)) & 1u));
      m.back[k][i] = base + 2 * ((NB[k] * x + i) % 5) + h;
    }
  }
  m.cm = base + 2 * ((x + 4) % 5) + h;
  m.cp = base + 2 * ((x + 1) % 5) + (h ^ 1u);
  m.cp_rot = h ^ 1u;
  m.row0 = x == 0 ? ~0u : 0u;
  return m;
}

LWE_DEV uint32_t tri_shfl(uint32_t v, uint32_t src) {
  return __shfl_sync(0xffffffffu, v, (int)src);
}

// index x + 5 y of the lane in column register i (b = 3, before the first
// round and after the last)
LWE_DEV uint32_t tri_lane(const KeccakTri &m, uint32_t i) { return m.x + 5 * ((3 * m.x + i) % 5); }

// 24 rounds on the warp's three states (every thread of the warp calls it).
LWE_DEV void keccak_f1600_tri(const KeccakTri &m, uint32_t s[5]) {
#pragma unroll 1
  for (int it = 0; it < 24; it += 3) {
#pragma unroll
    for (int k = 0; k < 3; k++) {
      constexpr int PI[3] = {3, 4, 2}, BK[3] = {2, 1, 3};  // (1 - b), -a (third: after the rotation)
      // theta, and rho of the lanes that leave
      const uint32_t c = s[0] ^ s[1] ^ s[2] ^ s[3] ^ s[4];
      const uint32_t cm = tri_shfl(c, m.cm), cq = tri_shfl(c, m.cp);
      const uint32_t cp = __funnelshift_l(cq, cq, m.cp_rot);
      uint32_t t[5], u[5];
#pragma unroll
      for (int i = 0; i < 5; i++) {
        const uint32_t v = s[i] ^ cm ^ cp;
        t[i] = __funnelshift_l(v, v, m.rot[k][i]);
      }
      // pi
#pragma unroll
      for (int j = 0; j < 5; j++) u[j] = tri_shfl(t[(PI[k] * j) % 5], m.src[k][j]);
      // chi and iota: X + 1, X + 2 are registers j + 1, j + 2; X = 0 of row 0 is j = 0
      const int rc = 2 * (it + k);
#pragma unroll
      for (int j = 0; j < 5; j++) t[j] = u[j] ^ (~u[(j + 1) % 5] & u[(j + 2) % 5]);
      t[0] ^= (m.h ? kKeccakRcHalves.v[rc + 1] : kKeccakRcHalves.v[rc]) & m.row0;
      if (k == 2) {
#pragma unroll
        for (int b = 0; b < 3; b++) {
          const bool on = (m.x >> b) & 1u;
#pragma unroll
          for (int i = 0; i < 5; i++) u[i] = on ? t[(i + (1 << b)) % 5] : t[i];
#pragma unroll
          for (int i = 0; i < 5; i++) t[i] = u[i];
        }
      }
#pragma unroll
      for (int i = 0; i < 5; i++) s[i] = tri_shfl(t[(BK[k] * i) % 5], m.back[k][i]);
    }
  }
}

// half h of a 64-bit word: its bits h, h + 2, ...  (Each 32-bit half is
// compressed upward, t | t << k as a multiplication, which leaves the 16 bits
// at 7..14 and 23..30.)
LWE_DEV uint32_t tri_half(uint64_t w, uint32_t h) {
  uint32_t a = ((uint32_t)w >> h) & 0x55555555u, b = ((uint32_t)(w >> 32) >> h) & 0x55555555u;
  a = (a * 3u) & 0x66666666u;
  b = (b * 3u) & 0x66666666u;
  a = (a * 5u) & 0x78787878u;
  b = (b * 5u) & 0x78787878u;
  a = (a * 17u) & 0x7f807f80u;
  b = (b * 17u) & 0x7f807f80u;
  return __byte_perm(a >> 7, b >> 7, 0x6420);
}

// 32-bit word r of the state's first four lanes (the digest) on thread r < 8
// of each group (every thread of the warp calls it)
LWE_DEV uint32_t tri_digest_word(const KeccakTri &m, const uint32_t s[5]) {
  // lane (x, 0) is register -3 x = 2 x
  const uint32_t i = (2 * m.x) % 5;
  uint32_t v = s[0];
#pragma unroll
  for (uint32_t k = 1; k < 5; k++) v = i == k ? s[k] : v;
  const uint32_t o = __shfl_xor_sync(0xffffffffu, v, 1);  // groups start at even lanes
  // thread h = 0 the low 16 bits of both halves, h = 1 the high ones
  uint32_t e = m.h ? o >> 16 : v & 0xffffu, d = m.h ? v >> 16 : o & 0xffffu;
  auto spread = [](uint32_t t) {
    t = (t | (t << 8)) & 0x00ff00ffu;
    t = (t | (t << 4)) & 0x0f0f0f0fu;
    t = (t | (t << 2)) & 0x33333333u;
    return (t | (t << 1)) & 0x55555555u;
  };
  return spread(e) | (spread(d) << 1);
}

// One padded block whose 64-bit word w < 17 is word(w), into an empty state.
template <typename F>
LWE_DEV void tri_one_block(const KeccakTri &m, uint32_t s[5], F word) {
#pragma unroll
  for (uint32_t i = 0; i < 5; i++) {
    const uint32_t w = tri_lane(m, i);
    s[i] = w < SHA3_RATE / 8 ? tri_half(word(w), m.h) : 0u;
  }
  keccak_f1600_tri(m, s);
}

// 64-bit word w of block blk of a `len`-byte message at an 8-byte aligned
// address, with the SHA-3 domain bits and pad10*1 of the last block; words
// beyond it and the capacity's are zero.  GLB: global memory (read-only path).
template <bool GLB>
LWE_DEV uint64_t tri_msg_word(const uint8_t *msg, uint32_t len, uint32_t blk, uint32_t w) {
  if (w >= SHA3_RATE / 8 || blk > len / SHA3_RATE) return 0;
  const uint32_t base = blk * SHA3_RATE + 8 * w;
  uint64_t v = 0;
  if (base + 8 <= len) {
    const uint64_t *p = reinterpret_cast<const uint64_t *>(msg + base);
    v = GLB ? __ldg(p) : *p;
  } else if (base < len) {
    for (uint32_t b = 0; b < len - base; b++) v |= (uint64_t)msg[base + b] << (8 * b);
  }
  if (base <= len && len < base + 8) v ^= (uint64_t)0x06 << (8 * (len - base));
  if (w == SHA3_RATE / 8 - 1 && blk == len / SHA3_RATE) v ^= 0x8000000000000000ull;
  return v;
}

// Absorbs blocks k0 .. of each group's message, to its end (msg, len are the
// group's, k0 the warp's; a group without a message passes len 0 and ignores
// its digest).  The warp runs as many permutations as its longest message
// needs; a group that is done keeps its state.  The next block's words are
// fetched before a permutation.
template <bool GLB>
LWE_DEV void sha3_absorb_tri(const KeccakTri &m, const uint8_t *msg, uint32_t len, uint32_t k0,
                             uint32_t s[5]) {
  const uint32_t full = len / SHA3_RATE, nblk = full + 1;
  const uint32_t most = __reduce_max_sync(0xffffffffu, nblk);
  uint32_t lane[5];
  uint64_t w[5];
  auto fetch = [&](uint32_t k) {
    if (k < full) {  // whole blocks: no padding
      const uint64_t *p = reinterpret_cast<const uint64_t *>(msg) + (SHA3_RATE / 8) * k;
#pragma unroll
      for (uint32_t i = 0; i < 5; i++)
        w[i] = lane[i] < SHA3_RATE / 8 ? (GLB ? __ldg(p + lane[i]) : p[lane[i]]) : 0ull;
    } else {
#pragma unroll
      for (uint32_t i = 0; i < 5; i++) w[i] = tri_msg_word<GLB>(msg, len, k, lane[i]);
    }
  };
#pragma unroll
  for (uint32_t i = 0; i < 5; i++) {
    lane[i] = tri_lane(m, i);
  }
  fetch(k0);
  for (uint32_t k = k0; k < most; k++) {
    uint32_t v[5];
#pragma unroll
    for (uint32_t i = 0; i < 5; i++) v[i] = s[i] ^ tri_half(w[i], m.h);
    if (k + 1 < most) fetch(k + 1);
    keccak_f1600_tri(m, v);
#pragma unroll
    for (uint32_t i = 0; i < 5; i++) s[i] = k < nblk ? v[i] : s[i];
  }
}

// SHA3-256 of each group's message.
template <bool GLB>
LWE_DEV void sha3_256_tri(const KeccakTri &m, const uint8_t *msg, uint32_t len, uint32_t s[5]) {
#pragma unroll
  for (uint32_t i = 0; i < 5; i++) s[i] = 0;
  sha3_absorb_tri<GLB>(m, msg, len, 0, s);
}
