// kem_kernels.cu -- kernels of the plain-LWE KEM hot path (sm_103a) but for
// the batched GEMM (gemm_tc.cu).
//
//   k_expand_A      sample(seedA) of Alg. 1: AES-128-CTR expansion of A,
//                   16-byte coalesced stores.
//   k_noise         the error/secret distributions of Alg. 1-2 (Tab. 1:
//                   rounded Gaussian) by CDF-table inverse sampling of AES
//                   counter streams.
//   products.cuh    k_mul_as, k_mul_as_gen, k_mul_as_gen_split: B = A S + E
//                   of Alg. 1 (A stored, or regenerated from its seed);
//                   k_sa, k_sa_gen: B' = S' A + E' and C = S' B + E'' +
//                   Enc(mu) of Alg. 2, with a compare epilogue for Alg. 5.
//   k_decrypt       M = C - B' S and mu' = Dec(M) of Alg. 3.
//   k_keygen_seeds, k_derive, k_tree, k_final_key: the hashing of
//                   Alg. 4-5 (SHA3-256) and the Fujisaki-Okamoto selection.
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include <algorithm>
#include <vector>

#include "aes.cuh"
#include "common.cuh"
#include "gemm_tc.h"
#include "kem_kernels.h"
#include "pp_types.h"
#include "keccak_warp.cuh"

// The round table T0 (see aes.cuh) and the replicated shared-memory image of
// all four tables; both written by lwe_upload_aes_table.
__device__ uint32_t g_aes_T0[256];
__device__ uint4 g_aes_img[AES_TABLE_WORDS / 4];

// ---------------------------------------------------------------------------
// A expansion: a warp per run of 128 counter blocks (16-byte blocks of A),
// grid-stride over the runs; one key per grid.y.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(512, 1) k_expand_A(const uint8_t *__restrict__ seeds,
                                                  uint32_t seed_stride, uint32_t n,
                                                  uint32_t logq, uint16_t *__restrict__ A,
                                                  uint64_t a_stride) {
  extern __shared__ uint32_t sT[];
  pdl_trigger();
  aes_fill_smem(sT, g_aes_img);
  __syncthreads();
  pdl_wait();
  const AesTab tab = aes_tab(sT);
  const uint32_t e = blockIdx.y;
  uint32_t key[4], rk[44];
  aes_load_key(seeds + (size_t)e * seed_stride, key);
  aes_key_expand(tab, key, rk);
  const uint32_t m = (1u << logq) - 1u;
  const uint32_t mm = m | (m << 16);
  const uint64_t nblk = (uint64_t)n * n / 8;
  uint4 *out = reinterpret_cast<uint4 *>(A + (size_t)e * a_stride);
  // a warp takes runs of 128 consecutive blocks (4 per lane, two at a time);
  // a run lies inside one 256-aligned counter window (aes_ctr_run), whose
  // constants are worked out for 32 runs at a time, one per lane, and
  // passed to the warp by shuffles as in noise_runs
  const uint32_t lane = threadIdx.x & 31;
  const uint64_t nruns = (nblk + 127) / 128, nw = (uint64_t)gridDim.x * (blockDim.x >> 5);
  // (warp-major: the runs of the last, partial round go to all SMs alike)
  const uint64_t gw = (uint64_t)(threadIdx.x >> 5) * gridDim.x + blockIdx.x;
  for (uint64_t g = 0; gw + nw * g < nruns; g += 32) {
    AesCtrRun mine{};
    if (gw + nw * (g + lane) < nruns) mine = aes_ctr_run(tab, rk, 0, (gw + nw * (g + lane)) * 128);
    for (uint32_t jr = 0; jr < 32; jr++) {
      const uint64_t run = gw + nw * (g + jr);
      if (run >= nruns) break;  // the same for every lane
      const uint64_t first = run * 128;
      const AesCtrRun win = aes_ctr_run_shfl(mine, jr);
      const uint32_t x0 = (uint32_t)(first & 255u) + lane;
      if (first + 128 <= nblk) {
#pragma unroll
        for (uint32_t j = 0; j < 4; j += 2) {
          uint4 va = aes_ctr_run_block(tab, rk, win, x0 + 32 * j);
          uint4 vb = aes_ctr_run_block(tab, rk, win, x0 + 32 * j + 32);
          out[first + lane + 32 * j] = make_uint4(va.x & mm, va.y & mm, va.z & mm, va.w & mm);
          out[first + lane + 32 * j + 32] = make_uint4(vb.x & mm, vb.y & mm, vb.z & mm, vb.w & mm);
        }
      } else {
#pragma unroll 1
        for (uint32_t x = x0; first + (x - x0) + lane < nblk; x += 32) {
          const uint4 v = aes_ctr_run_block(tab, rk, win, x);
          out[first + (x - x0) + lane] = make_uint4(v.x & mm, v.y & mm, v.z & mm, v.w & mm);
        }
      }
    }
  }
}

// ---------------------------------------------------------------------------
// Noise: a warp generates one run of counter blocks of one stream of one item
// (4 blocks per lane, two at a time, in batches; one in small calls; contiguous
// stores).  Sampling (Tab. 1, rounded Gaussian by CDF inversion): a 16-bit word
// w gives t = w >> 1, |e| = #{i : t > T[i]}, e < 0 iff w & 1.  A table of e for
// all 65536 words (64 KB of int8) sits in shared memory, so a sample costs one
// byte load; it is made from T with the same comparison rule when the context
// is created and copied in by each CTA, or made by the CTA where there is no
// context.
// ---------------------------------------------------------------------------
#define NOISE_TAB_OFF AES_SMEM_BYTES
#define NOISE_SMEM_BYTES (AES_SMEM_BYTES + 65536)

LWE_DEV int cdf_mag(uint32_t t, const NoiseArgs &a) {
  int mag = 0;
#pragma unroll
  for (int i = 0; i < 15; i++) mag += (t > a.T[i]) ? 1 : 0;
  return mag;
}

LWE_DEV void noise_fill_table(uint32_t *tab, const NoiseArgs &a) {
  // word j holds the samples of w = 4j .. 4j+3 (t = 2j, 2j, 2j+1, 2j+1)
  for (uint32_t j = threadIdx.x; j < 16384; j += blockDim.x) {
    const int m0 = cdf_mag(2 * j, a), m1 = cdf_mag(2 * j + 1, a);
    tab[j] = (uint32_t)(m0 & 0xff) | ((uint32_t)(-m0 & 0xff) << 8) | ((uint32_t)(m1 & 0xff) << 16) |
             ((uint32_t)(-m1 & 0xff) << 24);
  }
}

LWE_DEV int tab_sample(const char *smem, uint32_t w16) {
  return *reinterpret_cast<const int8_t *>(smem + NOISE_TAB_OFF + w16);
}

LWE_DEV void noise_store_i8(const int smp[8], uint8_t *base, uint32_t b, uint32_t nsamples) {
  if (8 * b + 8 <= nsamples) {
    const uint32_t lo = __byte_perm(__byte_perm(smp[0], smp[1], 0x0040),
                                    __byte_perm(smp[2], smp[3], 0x0040), 0x5410);
    const uint32_t hi = __byte_perm(__byte_perm(smp[4], smp[5], 0x0040),
                                    __byte_perm(smp[6], smp[7], 0x0040), 0x5410);
    *reinterpret_cast<uint2 *>(base + 8 * (size_t)b) = make_uint2(lo, hi);
  } else {
    for (int t = 0; t < 8; t++)
      if (8 * b + t < nsamples) base[8 * (size_t)b + t] = (uint8_t)(int8_t)smp[t];
  }
}

// small integers are exact in bf16
LWE_DEV void noise_store_bf16(const int smp[8], uint8_t *base, uint32_t b, uint32_t nsamples) {
  __nv_bfloat16 *bp = reinterpret_cast<__nv_bfloat16 *>(base);
  if (8 * b + 8 <= nsamples) {
    uint32_t pk[4];
#pragma unroll
    for (int t = 0; t < 4; t++) {
      __nv_bfloat162 h2 = __floats2bfloat162_rn((float)smp[2 * t], (float)smp[2 * t + 1]);
      pk[t] = *reinterpret_cast<uint32_t *>(&h2);
    }
    *reinterpret_cast<uint4 *>(bp + 8 * (size_t)b) = make_uint4(pk[0], pk[1], pk[2], pk[3]);
  } else {
    for (int t = 0; t < 8; t++)
      if (8 * b + t < nsamples) bp[8 * (size_t)b + t] = __float2bfloat16_rn((float)smp[t]);
  }
}

// PP: the paper profile's launches, with its two further formats
template <bool PP>
LWE_DEV void noise_store(const char *smem, const NoiseArgs &a, const NoiseOut &o, uint8_t *base,
                         uint32_t b, uint4 v) {
  const uint32_t w[4] = {v.x, v.y, v.z, v.w};
  if (PP && o.fmt == NOISE_UNIFORM) {
    int32_t *dst = reinterpret_cast<int32_t *>(base);
    for (uint32_t t = 0; t < 8; t++) {
      const uint32_t h = (w[t >> 1] >> (16 * (t & 1))) & 0xffffu;
      if (8 * b + t < o.nsamples)
        dst[8 * (size_t)b + t] = (int)(((2u * a.kunif + 1u) * h) >> 16) - (int)a.kunif;
    }
    return;
  }
  int smp[8];
#pragma unroll
  for (int t = 0; t < 4; t++) {
    smp[2 * t] = tab_sample(smem, w[t] & 0xffffu);
    smp[2 * t + 1] = tab_sample(smem, w[t] >> 16);
  }
  if (o.fmt != NOISE_BF16) noise_store_i8(smp, base, b, o.nsamples);
  if (o.fmt == NOISE_BF16 || (PP && o.fmt == NOISE_BOTH))
    noise_store_bf16(smp, PP && o.fmt == NOISE_BOTH ? reinterpret_cast<uint8_t *>(o.base2) : base, b,
                     o.nsamples);
}

// The runs of one warp: warp `gwarp` of `nwarps` takes runs gwarp,
// gwarp + nwarps, ...  A run's window constants (aes_ctr_run: 27 lookups)
// are the same for all 32 lanes, so they are worked out for 32 runs at a
// time, lane l for the warp's (g + l)-th run with that run's item key, and
// passed to the whole warp by shuffles when the run comes up: 27 lookup
// instructions per 32 runs instead of per run.
struct NoiseRun {
  uint32_t e, r, s;  // item, run within the item's streams, stream
};

LWE_DEV NoiseRun noise_run_of(const NoiseArgs &a, uint64_t run) {
  NoiseRun x;
  if (run >> 32) {
    x.e = (uint32_t)(run / a.runs_per_item);
  } else {  // a 32-bit division where it does (the other takes ~100 instructions)
    x.e = (uint32_t)run / a.runs_per_item;
  }
  x.r = (uint32_t)(run - (uint64_t)x.e * a.runs_per_item);
  x.s = 0;
  while (x.s + 1 < a.nout && x.r >= a.out[x.s].runs) {
    x.r -= a.out[x.s].runs;
    x.s++;
  }
  return x;
}

LWE_DEV void noise_load_rk(const NoiseArgs &a, uint32_t e, uint32_t rk[44]) {
  const uint4 *rkp = reinterpret_cast<const uint4 *>(a.rk + 44 * (size_t)e);
#pragma unroll
  for (int i = 0; i < 11; i++) {
    const uint4 v = __ldg(rkp + i);
    rk[4 * i] = v.x;
    rk[4 * i + 1] = v.y;
    rk[4 * i + 2] = v.z;
    rk[4 * i + 3] = v.w;
  }
}

template <bool PP>
LWE_DEV void noise_runs(const NoiseArgs &a, const AesTab &tab, const char *smem, uint64_t gwarp,
                        uint64_t nwarps) {
  const uint32_t lane = threadIdx.x & 31;
  const uint64_t nruns = (uint64_t)a.count * a.runs_per_item;
  for (uint64_t g = 0; gwarp + nwarps * g < nruns; g += 32) {
    // window constants of this warp's runs g .. g + 31, one per lane
    AesCtrRun mine{};
    {
      const uint64_t run = gwarp + nwarps * (g + lane);
      if (run < nruns) {
        const NoiseRun x = noise_run_of(a, run);
        if (LWE_BOUNDS(x.e < a.count, 108)) {
          uint32_t rk[44];
          noise_load_rk(a, x.e, rk);
          mine = aes_ctr_run(tab, rk, a.out[x.s].domain, x.r * a.run);
        }
      }
    }
    for (uint32_t j = 0; j < 32; j++) {
      const uint64_t run = gwarp + nwarps * (g + j);
      if (run >= nruns) break;  // the same for every lane
      const AesCtrRun win = aes_ctr_run_shfl(mine, j);
      const NoiseRun x = noise_run_of(a, run);
      if (!LWE_BOUNDS(x.e < a.count, 108)) continue;
      const NoiseOut o = a.out[x.s];
      uint32_t rk[44];
      noise_load_rk(a, x.e, rk);
      const uint32_t nblk = (o.nsamples + 7) / 8;
      uint8_t *base = reinterpret_cast<uint8_t *>(o.base) + (size_t)x.e * o.item_stride;
      // a run lies inside one 256-aligned window of counter indices, whose
      // first two AES rounds are in `win`
      const uint32_t first = x.r * a.run, b0 = first + lane, x0 = (first & 255u) + lane;
      if (a.run == NOISE_RUN && first + NOISE_RUN <= nblk) {
        // full run: two independent blocks in flight per lane
#pragma unroll
        for (uint32_t jj = 0; jj < NOISE_RUN / 32; jj += 2) {
          const uint4 va = aes_ctr_run_block(tab, rk, win, x0 + 32 * jj);
          const uint4 vb = aes_ctr_run_block(tab, rk, win, x0 + 32 * jj + 32);
          noise_store<PP>(smem, a, o, base, b0 + 32 * jj, va);
          noise_store<PP>(smem, a, o, base, b0 + 32 * jj + 32, vb);
        }
      } else {
#pragma unroll 1
        for (uint32_t b = b0; b < min(nblk, first + a.run); b += 32)
          noise_store<PP>(smem, a, o, base, b, aes_ctr_run_block(tab, rk, win, x0 + (b - b0)));
      }
    }
  }
}

template <bool PP>
__global__ void __launch_bounds__(512, 1) k_noise(NoiseArgs a) {
  extern __shared__ uint32_t sT[];
  pdl_trigger();
  aes_fill_smem(sT, g_aes_img);
  if (a.tab_img) {
    // the context's prebuilt sampler table (k_noise_table's output)
    uint4 *d = reinterpret_cast<uint4 *>(sT + NOISE_TAB_OFF / 4);
#pragma unroll 4
    for (uint32_t i = threadIdx.x; i < 65536 / 16; i += blockDim.x) d[i] = a.tab_img[i];
  } else {
    noise_fill_table(sT + NOISE_TAB_OFF / 4, a);
  }
  __syncthreads();
  pdl_wait();
  const AesTab tab = aes_tab(sT);
  // large calls: a CTA's warps take consecutive runs (mostly one item's);
  // small ones: consecutive runs go to different SMs
  const uint64_t nw = blockDim.x >> 5, w = threadIdx.x >> 5;
  noise_runs<PP>(a, tab, reinterpret_cast<const char *>(sT),
             a.run == NOISE_RUN ? blockIdx.x * nw + w : w * gridDim.x + blockIdx.x, gridDim.x * nw);
}

LWE_BOUNDS_READER(lwe_bounds_read_kem)

// The sampler table exactly as k_noise builds and reads it, for all 65536
// words: out[w] = the sample of word w (a check of the table against the
// definition of the sampler; one CTA).
__global__ void __launch_bounds__(512, 1) k_noise_table(NoiseArgs a, int8_t *out) {
  extern __shared__ uint32_t sT[];
  noise_fill_table(sT + NOISE_TAB_OFF / 4, a);
  __syncthreads();
  const char *smem = reinterpret_cast<const char *>(sT);
  for (uint32_t w = threadIdx.x; w < 65536; w += blockDim.x) out[w] = (int8_t)tab_sample(smem, w);
}

#include "products.cuh"

// ---------------------------------------------------------------------------
// Rows times S^T: out[r][l] = sum_j X[r][j] * St[l][j] for l < 8.
// A warp owns a row; a lane takes 8-element chunks (16 bytes of X, one AES
// block when X = A is regenerated) and uses dp2a: two 16-bit entries of X
// (as signed halves, the same residues mod 2^16) times two int8 of S^T.
// ---------------------------------------------------------------------------
LWE_DEV void dot8_chunk(const uint4 x, const int8_t *__restrict__ St, uint32_t n,
                        uint32_t j, int acc[8]) {
#pragma unroll
  for (int l = 0; l < 8; l++) {
    const uint2 s = ld_nc_u2(St + (size_t)l * n + j);
    acc[l] = __dp2a_lo((int)x.x, (int)s.x, acc[l]);
    acc[l] = __dp2a_hi((int)x.y, (int)s.x, acc[l]);
    acc[l] = __dp2a_lo((int)x.z, (int)s.y, acc[l]);
    acc[l] = __dp2a_hi((int)x.w, (int)s.y, acc[l]);
  }
}

LWE_DEV void warp_allreduce8(int acc[8]) {
#pragma unroll
  for (int l = 0; l < 8; l++) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc[l] += __shfl_xor_sync(0xffffffffu, acc[l], o);
  }
}

// Decrypt (Alg. 3): warp r of CTA e computes row r of M = C - B' S and the
// B message bits of its eight coefficients.
__global__ void __launch_bounds__(256) k_decrypt(DecryptArgs a) {
  pdl_trigger();
  pdl_wait();
  const uint32_t e = blockIdx.x;
  const uint32_t r = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t n = a.n;
  const uint8_t *ct = a.ct + (size_t)e * a.ct_bytes;
  const uint16_t *Brow = reinterpret_cast<const uint16_t *>(ct) + (size_t)r * n;
  const int8_t *St = a.sk_ptrs ? reinterpret_cast<const int8_t *>(a.sk_ptrs[e]) : a.St;
  int acc[8] = {0, 0, 0, 0, 0, 0, 0, 0};
  // up to four 16-byte chunks of the row per lane are requested together,
  // so a warp waits for one memory latency per 2048 bytes, not per chunk
  const uint32_t nch = n / 8;
  for (uint32_t base = 0; base < nch; base += 128) {
    uint4 x[4];
#pragma unroll
    for (int k = 0; k < 4; k++) {
      const uint32_t jc = base + lane + 32 * k;
      x[k] = jc < nch ? ld_nc_u4(Brow + 8 * (size_t)jc) : make_uint4(0, 0, 0, 0);
    }
#pragma unroll
    for (int k = 0; k < 4; k++) {
      const uint32_t jc = base + lane + 32 * k;
      if (jc < nch) dot8_chunk(x[k], St, n, 8 * jc, acc);
    }
  }
  warp_allreduce8(acc);
  if (lane == 0) {
    const uint32_t D = a.logq, Bb = a.B, m = (1u << D) - 1u;
    const uint16_t *C = reinterpret_cast<const uint16_t *>(ct + 16 * (size_t)n) + 8 * r;
    uint32_t bits = 0;
#pragma unroll
    for (int l = 0; l < 8; l++) {
      const uint32_t M = ((uint32_t)C[l] - (uint32_t)acc[l]) & m;
      const uint32_t sym = ((M + (1u << (D - Bb - 1))) >> (D - Bb)) & ((1u << Bb) - 1u);
      bits |= sym << (l * Bb);
    }
    uint8_t *mu = a.mu + (size_t)e * 32 + r * Bb;
    for (uint32_t t = 0; t < Bb; t++) mu[t] = (uint8_t)(bits >> (8 * t));
  }
}

// ---------------------------------------------------------------------------
// Hashing: seeds (Alg. 1), derivation of K' and seedSE' (Alg. 4-5), tree
// hash of pk / c, and the final keys.
// ---------------------------------------------------------------------------
// 32 bytes at any alignment as four little-endian words
LWE_DEV void load32_le(const uint8_t *p, uint64_t w[4]) {
  if ((reinterpret_cast<uintptr_t>(p) & 7) == 0) {
    const uint64_t *q = reinterpret_cast<const uint64_t *>(p);
#pragma unroll
    for (int i = 0; i < 4; i++) w[i] = q[i];
  } else {
#pragma unroll
    for (int i = 0; i < 4; i++) {
      uint64_t v = 0;
#pragma unroll
      for (int b = 0; b < 8; b++) v |= (uint64_t)p[8 * i + b] << (8 * b);
      w[i] = v;
    }
  }
}

// SHA3-256 of prefix || 32 bytes, built lane by lane (the 33-byte message
// is the 32 bytes shifted up one byte; padding opens byte 1 of lane 4)
LWE_DEV void sha3_prefixed32(uint8_t prefix, const uint8_t *msg32, uint64_t s[25]) {
  uint64_t w[4];
  load32_le(msg32, w);
  s[0] = (uint64_t)prefix | (w[0] << 8);
#pragma unroll
  for (int j = 1; j < 4; j++) s[j] = (w[j - 1] >> 56) | (w[j] << 8);
  s[4] = (w[3] >> 56) | ((uint64_t)0x06 << 8);
#pragma unroll
  for (int j = 5; j < 25; j++) s[j] = 0;
  s[SHA3_RATE / 8 - 1] ^= 0x8000000000000000ull;
  keccak_f1600(s);
}

__global__ void k_keygen_seeds(KeygenSeedArgs a) {
  pdl_trigger();
  pdl_wait();
  const uint32_t e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= a.count) return;
  const uint8_t *ms = a.ms + 32 * (size_t)e;
  uint64_t s[25];
  uint8_t *pk = a.pk + (size_t)e * a.pk_bytes;
  uint8_t *sk = a.sk + (size_t)e * a.sk_bytes;
  uint8_t *ws = a.ws_seeds + 32 * (size_t)e;
  sha3_prefixed32(0x41, ms, s);  // seedA
  sha3_digest16(s, pk);
  sha3_digest16(s, sk + a.sk_pk_off);
  sha3_digest16(s, ws);
  sha3_prefixed32(0x53, ms, s);  // seedSE
  sha3_digest16(s, ws + 16);
  {
    const uint32_t key[4] = {(uint32_t)s[0], (uint32_t)(s[0] >> 32), (uint32_t)s[1],
                             (uint32_t)(s[1] >> 32)};
    uint32_t rk[44];
    aes_key_expand_global(g_aes_T0, key, rk);
    uint4 *dst = reinterpret_cast<uint4 *>(a.ws_rk + 44 * (size_t)e);
#pragma unroll
    for (int i = 0; i < 11; i++) dst[i] = make_uint4(rk[4 * i], rk[4 * i + 1], rk[4 * i + 2], rk[4 * i + 3]);
  }
  sha3_prefixed32(0x5A, ms, s);  // z
  sha3_digest(s, sk + a.sk_z_off);
}

// Alg. 4 / 5 seeds of the (re-)encryption.  mu is 8 B bytes (B <= 4), i.e.
// whole 64-bit lanes, so both messages are built lane by lane with
// compile-time state indices (nothing leaves the registers):
//   Encaps: mu = H(0x4D || coins)[0 : 8 B]
//   K' = H(pkh || mu),  seedSE' = H(0x01 || pkh || mu)[0 : 16]
// K' and seedSE' do not depend on each other: a CTA of two warps takes 32
// items, warp 0 computing K' and warp 1 seedSE' and its key schedule (both
// warps hash mu themselves), so each item waits for two permutations in
// Encaps and one in Decaps instead of three and two.
__global__ void __launch_bounds__(64) k_derive(DeriveArgs a) {
  __shared__ uint32_t sT0[256];  // the key expansion's S-box lookups stay on chip
  pdl_trigger();
  for (uint32_t i = threadIdx.x; i < 256; i += blockDim.x) sT0[i] = g_aes_T0[i];
  __syncthreads();
  pdl_wait();
  const uint32_t w = threadIdx.x >> 5;
  const uint32_t e = blockIdx.x * 32 + (threadIdx.x & 31);
  if (e >= a.count) return;
  uint64_t s[25];
  uint64_t *mu64 = reinterpret_cast<uint64_t *>(a.mu + 32 * (size_t)e);
  if (a.flags && w == 0) a.flags[e] = 0;
  const uint32_t nb = a.mu_bytes / 8;  // lanes of mu, 1..4
  uint64_t x[8];                       // pkh (4 lanes) || mu (nb lanes) || zeros
  if (a.coins) {
    sha3_prefixed32(0x4D, a.coins + 32 * (size_t)e, s);
#pragma unroll
    for (int i = 0; i < 4; i++) {
      x[4 + i] = (uint32_t)i < nb ? s[i] : 0;
      if (w == 0) mu64[i] = x[4 + i];
    }
  } else {
#pragma unroll
    for (int i = 0; i < 4; i++) x[4 + i] = (uint32_t)i < nb ? mu64[i] : 0;
  }
  const uint8_t *pkh = a.pkh_ptrs ? a.pkh_ptrs[e] + a.pkh_off : a.pkh + (size_t)e * a.pkh_stride;
  load32_le(pkh, x);
  // (every lane is written unconditionally with a selected value: a
  // conditional store to lane 4 + nb would become a dynamically indexed
  // state, i.e. local memory)
  if (w == 0) {
    // K' = H(pkh || mu): 32 + 8 nb bytes, padding opens lane 4 + nb
#pragma unroll
    for (int i = 0; i < 25; i++) s[i] = i < 8 ? x[i] : 0;
#pragma unroll
    for (int i = 5; i < 9; i++) s[i] ^= (uint32_t)i == 4 + nb ? 0x06ull : 0ull;
    s[SHA3_RATE / 8 - 1] ^= 0x8000000000000000ull;
    keccak_f1600(s);
    sha3_digest(s, a.kprime + 32 * (size_t)e);
    return;
  }
  // seedSE' = H(0x01 || pkh || mu): the same lanes one byte later; the
  // padding byte lands in byte 1 of lane 4 + nb
  s[0] = 0x01 | (x[0] << 8);
#pragma unroll
  for (int j = 1; j < 9; j++) s[j] = (x[j - 1] >> 56) | (j < 8 ? x[j] << 8 : 0);
#pragma unroll
  for (int j = 9; j < 25; j++) s[j] = 0;
#pragma unroll
  for (int i = 5; i < 9; i++) s[i] ^= (uint32_t)i == 4 + nb ? 0x0600ull : 0ull;
  s[SHA3_RATE / 8 - 1] ^= 0x8000000000000000ull;
  keccak_f1600(s);
  sha3_digest16(s, a.seeds + 32 * (size_t)e);
  const uint32_t key[4] = {(uint32_t)s[0], (uint32_t)(s[0] >> 32), (uint32_t)s[1],
                           (uint32_t)(s[1] >> 32)};
  uint32_t rk[44];
  aes_key_expand_global(sT0, key, rk);
  uint4 *dst = reinterpret_cast<uint4 *>(a.rk + 44 * (size_t)e);
#pragma unroll
  for (int i = 0; i < 11; i++) dst[i] = make_uint4(rk[4 * i], rk[4 * i + 1], rk[4 * i + 2], rk[4 * i + 3]);
}

// ---------------------------------------------------------------------------
// The same hashes with ten threads per Keccak state (keccak_warp.cuh), for
// launches of few items: one permutation then takes ~2 us instead of one
// thread's ~5.6 us, and the independent hashes of an item run side by side in
// one warp.
// ---------------------------------------------------------------------------
LWE_DEV uint64_t ld_le64(const uint8_t *p) {
  if ((reinterpret_cast<uintptr_t>(p) & 7) == 0) return *reinterpret_cast<const uint64_t *>(p);
  uint64_t v = 0;
#pragma unroll
  for (int b = 0; b < 8; b++) v |= (uint64_t)p[b] << (8 * b);
  return v;
}

LWE_DEV void st_le32(uint8_t *p, uint32_t v) {
  if ((reinterpret_cast<uintptr_t>(p) & 3) == 0) {
    *reinterpret_cast<uint32_t *>(p) = v;
  } else {
#pragma unroll
    for (int b = 0; b < 4; b++) p[b] = (uint8_t)(v >> (8 * b));
  }
}

// word w of a padded single-block message of 8 nw bytes
LWE_DEV uint64_t sha3_pad_word(uint32_t w, uint32_t nw) {
  return (w == nw ? 0x06ull : 0ull) ^ (w == SHA3_RATE / 8 - 1 ? 0x8000000000000000ull : 0ull);
}

// word w of prefix || 32 bytes, padded: the 32 bytes shifted up one byte,
// the padding opening byte 1 of word 4
LWE_DEV uint64_t prefixed32_word(uint8_t prefix, const uint8_t *msg32, uint32_t w) {
  uint64_t v = sha3_pad_word(w, 4) & ~0xffull;
  if (w < 4) v |= ld_le64(msg32 + 8 * w) << 8;
  if (w >= 1 && w <= 4) v |= ld_le64(msg32 + 8 * (w - 1)) >> 56;
  if (w == 0) v |= prefix;
  if (w == 4) v |= 0x0600ull;
  return v;
}

// The key schedule of the 16-byte seed held as digest words 0..3 by the
// threads first .. first + 3, written to rk; the whole warp calls it.
LWE_DEV void warp_store_schedule(const uint32_t *sT0, uint32_t v, uint32_t first, uint32_t lane,
                                 uint32_t *out) {
  uint32_t key[4], rk[44];
#pragma unroll
  for (uint32_t i = 0; i < 4; i++) key[i] = tri_shfl(v, first + i);
  if (lane != first) return;
  aes_key_expand_global(sT0, key, rk);
  uint4 *dst = reinterpret_cast<uint4 *>(out);
#pragma unroll
  for (int i = 0; i < 11; i++)
    dst[i] = make_uint4(rk[4 * i], rk[4 * i + 1], rk[4 * i + 2], rk[4 * i + 3]);
}

// KeyGen seeds (Alg. 1): group j of the item's warp hashes prefix j || ms;
// four items per CTA
__global__ void __launch_bounds__(128) k_keygen_seeds_warp(KeygenSeedArgs a) {
  __shared__ uint32_t sT0[256];
  pdl_trigger();
  const uint32_t e = blockIdx.x * 4 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  for (uint32_t i = threadIdx.x; i < 256; i += 128) sT0[i] = g_aes_T0[i];
  const KeccakTri km = keccak_tri(lane);
  __syncthreads();
  pdl_wait();
  if (e >= a.count) return;  // the whole warp
  const uint8_t prefix = km.grp == 0 ? 0x41 : (km.grp == 1 ? 0x53 : 0x5A);
  const uint8_t *ms = a.ms + 32 * (size_t)e;
  uint32_t s[5];
  tri_one_block(km, s, [&](uint32_t w) { return prefixed32_word(prefix, ms, w); });
  const uint32_t v = tri_digest_word(km, s), r = km.r;
  uint8_t *pk = a.pk + (size_t)e * a.pk_bytes;
  uint8_t *sk = a.sk + (size_t)e * a.sk_bytes;
  uint8_t *ws = a.ws_seeds + 32 * (size_t)e;
  if (lane < 30) {
    if (km.grp == 0 && r < 4) {  // seedA
      st_le32(pk + 4 * r, v);
      st_le32(sk + a.sk_pk_off + 4 * r, v);
      st_le32(ws + 4 * r, v);
    } else if (km.grp == 1 && r < 4) {  // seedSE
      st_le32(ws + 16 + 4 * r, v);
    } else if (km.grp == 2 && r < 8) {  // z
      st_le32(sk + a.sk_z_off + 4 * r, v);
    }
  }
  warp_store_schedule(sT0, v, 10, lane, a.ws_rk + 44 * (size_t)e);
}

// Encaps / Decaps derivation (Alg. 4, 5): every group hashes mu (Encaps),
// then group 0 K' = H(pkh || mu) and group 1 seedSE' = H(0x01 || pkh || mu)
// with its key schedule
__global__ void __launch_bounds__(128) k_derive_warp(DeriveArgs a) {
  __shared__ uint32_t sT0[256];
  __shared__ uint64_t sxs[4][9];  // per warp: pkh (4 words) || mu (4 words) || 0
  pdl_trigger();
  const uint32_t e = blockIdx.x * 4 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  uint64_t *sx = sxs[threadIdx.x >> 5];
  for (uint32_t i = threadIdx.x; i < 256; i += 128) sT0[i] = g_aes_T0[i];
  const KeccakTri km = keccak_tri(lane);
  if (lane == 8) sx[8] = 0;
  __syncthreads();
  pdl_wait();
  if (e >= a.count) return;  // the whole warp
  if (a.flags && lane == 0) a.flags[e] = 0;
  const uint32_t nb = a.mu_bytes / 8;  // words of mu, 1..4
  uint32_t *mu = reinterpret_cast<uint32_t *>(a.mu + 32 * (size_t)e);
  const uint8_t *pkh = a.pkh_ptrs ? a.pkh_ptrs[e] + a.pkh_off : a.pkh + (size_t)e * a.pkh_stride;
  if (lane >= 16 && lane < 20) sx[lane - 16] = ld_le64(pkh + 8 * (lane - 16));
  uint32_t s[5];
  uint32_t m = 0;  // thread r < 8: 32-bit word r of mu (zero beyond nb words)
  if (a.coins) {
    const uint8_t *coins = a.coins + 32 * (size_t)e;
    tri_one_block(km, s, [&](uint32_t w) { return prefixed32_word(0x4D, coins, w); });
    m = tri_digest_word(km, s);
    if (lane < 8) {
      if (lane >= 2 * nb) m = 0;
      mu[lane] = m;
    }
  } else if (lane < 2 * nb) {
    m = mu[lane];
  }
  if (lane < 8) reinterpret_cast<uint32_t *>(sx + 4)[lane] = m;
  __syncwarp();
  // the two messages: x || padding, and the same one byte later after 0x01
  const bool enc = km.grp == 1;
  tri_one_block(km, s, [&](uint32_t w) -> uint64_t {
    const uint64_t x = sx[min(w, 8u)], pad = sha3_pad_word(w, 4 + nb);
    if (!enc) return x ^ pad;
    const uint64_t xp = w == 0 ? 0ull : sx[min(w - 1, 8u)];
    return (w == 0 ? 0x01ull : xp >> 56) ^ (x << 8) ^ (pad & ~0xffull) ^
           (w == 4 + nb ? 0x0600ull : 0ull);
  });
  const uint32_t v = tri_digest_word(km, s), r = km.r;
  if (lane < 30) {
    if (km.grp == 0 && r < 8) st_le32(a.kprime + 32 * (size_t)e + 4 * r, v);
    if (km.grp == 1 && r < 4) st_le32(a.seeds + 32 * (size_t)e + 4 * r, v);
  }
  warp_store_schedule(sT0, v, 10, lane, a.rk + 44 * (size_t)e);
}

// Decaps key (Alg. 5): K = H(K' || H(c)) when the re-encryption matched,
// else H(z || H(c)); one warp per item
__global__ void __launch_bounds__(128) k_final_key_warp(FinalKeyArgs a) {
  pdl_trigger();
  const uint32_t e = blockIdx.x * 4 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  const KeccakTri km = keccak_tri(lane);
  pdl_wait();
  if (e >= a.count) return;  // the whole warp
  const uint32_t f = a.flags[e];
  const uint64_t keep = (uint64_t)0 - (uint64_t)(((f | (0u - f)) >> 31) ^ 1u);
  const uint64_t *kp = reinterpret_cast<const uint64_t *>(a.kprime + 32 * (size_t)e);
  const uint64_t *z = reinterpret_cast<const uint64_t *>(a.z_ptrs ? a.z_ptrs[e] + a.z_off : a.z);
  const uint64_t *hc = reinterpret_cast<const uint64_t *>(a.hc + 32 * (size_t)e);
  uint32_t s[5];
  tri_one_block(km, s, [&](uint32_t w) -> uint64_t {
    uint64_t v = sha3_pad_word(w, 8);
    if (w < 4) v ^= (kp[w] & keep) | (z[w] & ~keep);
    else if (w < 8) v ^= hc[w - 4];
    return v;
  });
  const uint32_t v = tri_digest_word(km, s);
  if (lane < 8) st_le32(a.K + 32 * (size_t)e + 4 * lane, v);
}

// Tree hash: tpi threads per message compute its 1024-byte-chunk digests
// into shared memory; threads 0..ipc-1 (one per message, so the root phase
// fills whole warps) then hash the digests -- the root -- and, for Encaps,
// derive the key.  A message's digests sit at a stride of 4 m + 1 words so
// the root threads' 64-bit reads fall in different banks.
__global__ void __launch_bounds__(TREE_MAX_THREADS) k_tree(TreeArgs a) {
  extern __shared__ uint64_t sleaf[];  // [ipc][4 m + 1]
  pdl_trigger();
  pdl_wait();
  const uint32_t words = 4 * a.m + 1;
  const uint32_t e0 = blockIdx.x * a.ipc;
  {
    const uint32_t li = threadIdx.x / a.tpi, lt = threadIdx.x % a.tpi;
    const uint32_t e = e0 + li;
    if (li < a.ipc && e < a.count) {
      const uint8_t *msg = a.msg_ptrs ? a.msg_ptrs[e] : a.msgs + (size_t)e * a.stride;
      uint64_t *mine = sleaf + (size_t)li * words;
      uint64_t s[25];
      for (uint32_t c = lt; c < a.m; c += a.tpi) {
        const uint32_t off = c * LWE_TREE_CHUNK;
        if (!LWE_BOUNDS(off < a.len, 106)) continue;
        sha3_256_global(msg + off, min((uint32_t)LWE_TREE_CHUNK, a.len - off), s);
        mine[4 * c] = s[0];
        mine[4 * c + 1] = s[1];
        mine[4 * c + 2] = s[2];
        mine[4 * c + 3] = s[3];
      }
    }
  }
  __syncthreads();
  const uint32_t e = e0 + threadIdx.x;
  if (threadIdx.x >= a.ipc || e >= a.count) return;
  uint64_t s[25];
  sha3_256_mem(reinterpret_cast<const uint8_t *>(sleaf + (size_t)threadIdx.x * words), 32 * a.m, s);
  if (a.mode == TREE_DIGEST) {
    sha3_digest(s, a.out + (size_t)e * a.out_stride);
    if (a.out2) sha3_digest(s, a.out2 + (size_t)e * a.out2_stride);
    return;
  }
  // Encaps (Alg. 4): K = H(K' || H(c))
  uint64_t lanes[SHA3_RATE / 8];
  lanes_zero(lanes);
  const uint64_t *kp = reinterpret_cast<const uint64_t *>(a.kprime + 32 * (size_t)e);
  for (int i = 0; i < 4; i++) lanes[i] = kp[i];
  for (int i = 0; i < 4; i++) lanes[4 + i] = s[i];
  sha3_256_lanes(lanes, 64, s);
  sha3_digest(s, a.out + 32 * (size_t)e);
}

LWE_DEV void bar_arrive(uint32_t id, uint32_t n) {
  asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(n) : "memory");
}
LWE_DEV void bar_sync(uint32_t id, uint32_t n) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(n) : "memory");
}

// The end of a tree hash (s: the final state of each group's root, message e
// of the group if `in`): digest mode stores H into out (and out2); Encaps mode
// derives K = H(K' || H(c)) (Alg. 4), one 64-byte block.
LWE_DEV void tree_tri_out(const TreeArgs &a, uint32_t e, bool in, const KeccakTri &km,
                          uint32_t lane, uint32_t s[5]) {
  uint32_t v = tri_digest_word(km, s);
  const bool st = in && lane < 30 && km.r < 8;
  if (a.mode == TREE_DIGEST) {
    if (st) st_le32(a.out + (size_t)e * a.out_stride + 4 * km.r, v);
    if (st && a.out2) st_le32(a.out2 + (size_t)e * a.out2_stride + 4 * km.r, v);
    return;
  }
  uint64_t hc[4];
#pragma unroll
  for (uint32_t i = 0; i < 4; i++)
    hc[i] = (uint64_t)tri_shfl(v, 10 * km.grp + 2 * i) |
            ((uint64_t)tri_shfl(v, 10 * km.grp + 2 * i + 1) << 32);
  const uint64_t *kp = reinterpret_cast<const uint64_t *>(a.kprime + 32 * (size_t)(in ? e : 0));
  tri_one_block(km, s, [&](uint32_t w) -> uint64_t {
    uint64_t x = sha3_pad_word(w, 8);
    if (w < 4) x ^= kp[w];
#pragma unroll
    for (uint32_t i = 0; i < 4; i++) x ^= w == 4 + i ? hc[i] : 0ull;
    return x;
  });
  v = tri_digest_word(km, s);
  if (st) st_le32(a.out + 32 * (size_t)e + 4 * km.r, v);
}

// Tree hash of batches whose full-length leaves need 13 warps per CTA (one
// CTA per SM; e.g. 4096 ciphertexts of n = 976: 27 per CTA, 405 leaves of
// 8 permutations).  With one leaf per thread, 13 leaf warps put 4 warps on
// one SM sub-partition (SMSP) and 3 on the others: the loaded one needs 32
// warp-permutations where the others need 24, and the roots then run alone.
// Here, 16 warps with fixed roles:
//   - warps 0, 4, 8, 12 (SMSP 0) take the 128 leaves with the highest chunk
//     indices and run only TB_SPLIT of their 8 permutations; their sponge
//     states go to shared memory ([25][128] words);
//   - the nine other leaf warps (3 per SMSP 1-3) take the remaining leaves
//     whole;
//   - helper warps 14 and 15 (SMSPs 2, 3) finish the leaves of SMSP 0, two
//     warps' worth each, once those have stopped;
//   - warp 13 (SMSP 1) hashes the short last chunk of every message, then
//     starts the roots: their first blocks absorb digests of low chunk
//     indices, which all come from SMSPs 1-3, so they run while the helpers
//     work; it leaves the sponge states in shared memory ([ipc][25] words);
//   - the rest of the roots (and the Encaps keys) follows the helpers, three
//     per warp (keccak_warp.cuh) on warps whose leaves are done: two or three
//     permutations of ~2.4 us, where warp 13 alone took 4.7 each.
// Named barriers (fixed thread counts, every warp meets each of its
// barriers exactly once): 1 leaf warps of SMSPs 1-3 -> warp 13 (320);
// 2 warps 0, 4 -> helper 14 (96); 4 warps 8, 12 -> helper 15 (96);
// 3 helpers and warp 13 -> the eleven root warps (448).  At most 96 registers
// per thread (20 bytes of spill stores, 44 of loads; k_tree_dense 16 and 12): a
// CTA then leaves room in the SM's register file for the CTAs of Decaps' small
// kernels, which run beside its H(c) on the other stream.
#define TB_SPLIT 6
#define TB_SLOTS 128

__global__ void __maxnreg__(96) k_tree_bal(TreeArgs a) {
  extern __shared__ uint64_t sm[];
  pdl_trigger();
  pdl_wait();
  const uint32_t words = 4 * a.m + 1;
  uint64_t *sdig = sm;                              // [ipc][4 m + 1]
  uint64_t *shand = sm + (size_t)a.ipc * words;     // [25][TB_SLOTS]
  uint64_t *sroot = shand + 25 * TB_SLOTS;          // [ipc][25]
  const uint32_t e0 = blockIdx.x * a.ipc;
  const uint32_t nmsg = min(a.ipc, a.count - e0);
  const uint32_t warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t ML = a.ml;                         // full-length chunks per message
  const uint32_t NL = nmsg * ML;
  const uint32_t fullp = LWE_TREE_CHUNK / SHA3_RATE + 1;  // permutations per full chunk
  // root blocks whose digests all come from chunks below the lowest chunk
  // index held by SMSP 0 are absorbed before the helpers finish
  const uint32_t held = min((uint32_t)TB_SLOTS, NL);
  const uint32_t cmin = held ? ML - 1 - (held - 1) / nmsg : a.m;
  const uint32_t rlen = 32 * a.m, nb = rlen / SHA3_RATE + 1;
  uint32_t early = 0;
  while (early < nb && min(rlen - 1, SHA3_RATE * early + SHA3_RATE - 1) / 32 < cmin) early++;
  uint64_t s[25];
  auto msg_of = [&](uint32_t li) -> const uint8_t * {
    const uint32_t e = e0 + li;
    return a.msg_ptrs ? a.msg_ptrs[e] : a.msgs + (size_t)e * a.stride;
  };
  // leaf k (k < NL): chunk ML - 1 - k / nmsg of message k % nmsg, so the
  // first TB_SLOTS leaves are the highest chunk indices
  auto put_digest = [&](uint32_t li, uint32_t c, const uint64_t *st) {
    if (!LWE_BOUNDS(li < nmsg && c < a.m, 102)) return;
    uint64_t *d = sdig + (size_t)li * words + 4 * c;
    d[0] = st[0];
    d[1] = st[1];
    d[2] = st[2];
    d[3] = st[3];
  };
  if (warp < 13 && (warp & 3) == 0) {
    // SMSP 0: the first TB_SPLIT permutations of leaves 0 .. TB_SLOTS-1
    const uint32_t k = 32 * (warp >> 2) + lane;
    if (k < NL && LWE_BOUNDS(k < TB_SLOTS, 101)) {
      const uint32_t li = k % nmsg, c = ML - 1 - k / nmsg;
      sha3_init(s);
      if (LWE_BOUNDS((c + 1) * LWE_TREE_CHUNK <= a.len, 103))
        sha3_absorb_global(msg_of(li) + (size_t)c * LWE_TREE_CHUNK, LWE_TREE_CHUNK, 0, TB_SPLIT, s);
#pragma unroll
      for (int i = 0; i < 25; i++) shand[i * TB_SLOTS + k] = s[i];
    }
    __syncwarp();
    bar_arrive(warp < 8 ? 2 : 4, 96);
    if (warp >= 8) return;
  } else if (warp < 13) {
    // SMSPs 1-3: whole leaves TB_SLOTS ..
    const uint32_t idx = warp - 1 - (warp >> 2);  // 0 .. 8
    const uint32_t k = TB_SLOTS + 32 * idx + lane;
    if (k < NL) {
      const uint32_t li = k % nmsg, c = ML - 1 - k / nmsg;
      sha3_init(s);
      if (LWE_BOUNDS((c + 1) * LWE_TREE_CHUNK <= a.len, 103))
        sha3_absorb_global(msg_of(li) + (size_t)c * LWE_TREE_CHUNK, LWE_TREE_CHUNK, 0, fullp, s);
      put_digest(li, c, s);
    }
    __syncwarp();
    bar_arrive(1, 320);
  } else if (warp >= 14) {
    // helpers: the last permutations of two SMSP-0 warps' leaves each
    bar_sync(warp == 14 ? 2 : 4, 96);
    for (uint32_t g = 0; g < 2; g++) {
      const uint32_t k = 32 * (2 * (warp - 14) + g) + lane;
      if (k < NL && LWE_BOUNDS(k < TB_SLOTS, 104)) {
        const uint32_t li = k % nmsg, c = ML - 1 - k / nmsg;
#pragma unroll
        for (int i = 0; i < 25; i++) s[i] = shand[i * TB_SLOTS + k];
        sha3_absorb_global(msg_of(li) + (size_t)c * LWE_TREE_CHUNK, LWE_TREE_CHUNK, TB_SPLIT,
                           fullp, s);
        put_digest(li, c, s);
      }
    }
    __syncwarp();
    bar_arrive(3, 448);
    return;
  } else {
    // warp 13: the short last chunks, then the first blocks of the roots
    const uint32_t li = lane;
    const bool mine = li < nmsg;
    if (mine && ML < a.m) {
      const uint32_t c = a.m - 1, off = c * LWE_TREE_CHUNK, len = a.len - off;
      sha3_init(s);
      if (LWE_BOUNDS(off < a.len && len <= LWE_TREE_CHUNK, 105))
        sha3_absorb_global(msg_of(li) + off, len, 0, len / SHA3_RATE + 1, s);
      put_digest(li, c, s);
    }
    __syncwarp();
    bar_sync(1, 320);
    if (mine) {
      sha3_init(s);
      sha3_absorb_mem(reinterpret_cast<const uint8_t *>(sdig + (size_t)li * words), rlen, 0, early, s);
#pragma unroll
      for (int i = 0; i < 25; i++) sroot[li * 25 + i] = s[i];
    }
    __syncwarp();
    bar_arrive(3, 448);
    return;
  }
  // the roots' last blocks: warps 1-3, 5-7, 9-11, then 0 and 4, three each
  bar_sync(3, 448);
  const uint32_t ti = (warp & 3) ? warp - 1 - (warp >> 2) : 9 + (warp >> 2);
  if (3 * ti >= nmsg) return;
  const KeccakTri km = keccak_tri(lane);
  const uint32_t li = 3 * ti + km.grp;
  const bool in = li < nmsg;
  uint32_t st[5];
#pragma unroll
  for (uint32_t i = 0; i < 5; i++)
    st[i] = tri_half(sroot[(in ? li : 0) * 25 + tri_lane(km, i)], km.h);
  sha3_absorb_tri<false>(km, reinterpret_cast<const uint8_t *>(sdig + (size_t)(in ? li : 0) * words),
                         in ? rlen : 0u, early, st);
  tree_tri_out(a, e0 + li, in, km, lane, st);
}

// Tree hash of batches whose full-length leaves fill at most 12 warps per
// CTA (e.g. 4096 ciphertexts of n = 640: 27 per SM, 270 leaves): the leaves
// are packed densely, leaf k on warp k / 32 of warps 0-11, so consecutive
// warps fall on consecutive SM sub-partitions and every SMSP holds
// floor or ceil of WL / 4 leaf warps (k_tree instead gives each message a
// power-of-two group of threads, which leaves lanes idle).  The short last
// chunks run on one warp of the SMSP with the fewest leaf warps, `rw`; then,
// behind one named barrier (the twelve leaf warps, whether or not they hold
// leaves, and rw: 416 threads), the roots.
__global__ void __maxnreg__(96) k_tree_dense(TreeArgs a) {
  extern __shared__ uint64_t sm[];
  pdl_trigger();
  pdl_wait();
  const uint32_t words = 4 * a.m + 1;
  uint64_t *sdig = sm;  // [ipc][4 m + 1]
  const uint32_t e0 = blockIdx.x * a.ipc;
  const uint32_t nmsg = min(a.ipc, a.count - e0);
  const uint32_t warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t ML = a.ml, NL = nmsg * ML;
  const uint32_t fullp = LWE_TREE_CHUNK / SHA3_RATE + 1;
  uint64_t s[25];
  auto msg_of = [&](uint32_t li) -> const uint8_t * {
    const uint32_t e = e0 + li;
    return a.msg_ptrs ? a.msg_ptrs[e] : a.msgs + (size_t)e * a.stride;
  };
  auto put_digest = [&](uint32_t li, uint32_t c, const uint64_t *st) {
    if (!LWE_BOUNDS(li < nmsg && c < a.m, 111)) return;
    uint64_t *d = sdig + (size_t)li * words + 4 * c;
    d[0] = st[0];
    d[1] = st[1];
    d[2] = st[2];
    d[3] = st[3];
  };
  if (warp < 12) {
    const uint32_t k = 32 * warp + lane;  // leaf k: chunk k % ML of message k / ML
    if (k < NL) {
      const uint32_t li = k / ML, c = k % ML;
      sha3_init(s);
      if (LWE_BOUNDS((c + 1) * LWE_TREE_CHUNK <= a.len, 112))
        sha3_absorb_global(msg_of(li) + (size_t)c * LWE_TREE_CHUNK, LWE_TREE_CHUNK, 0, fullp, s);
      put_digest(li, c, s);
    }
  } else if (warp != a.rw) {
    return;
  } else {
    const uint32_t li = lane;
    if (li < nmsg && ML < a.m) {
      const uint32_t c = a.m - 1, off = c * LWE_TREE_CHUNK, len = a.len - off;
      sha3_init(s);
      if (LWE_BOUNDS(off < a.len && len <= LWE_TREE_CHUNK, 113))
        sha3_absorb_global(msg_of(li) + off, len, 0, len / SHA3_RATE + 1, s);
      put_digest(li, c, s);
    }
  }
  __syncwarp();
  bar_sync(1, 416);
  // the roots (and Encaps' keys), three per warp: chains of 4-5 permutations
  // at ~2.3 us each where one warp of one root per thread took 4.7
  if (3 * warp >= nmsg) return;
  const KeccakTri km = keccak_tri(lane);
  const uint32_t li = 3 * warp + km.grp;
  const bool in = li < nmsg;
  uint32_t st[5];
  sha3_256_tri<false>(km, reinterpret_cast<const uint8_t *>(sdig + (size_t)(in ? li : 0) * words),
                      in ? 32 * a.m : 0u, st);
  tree_tri_out(a, e0 + li, in, km, lane, st);
}

// Tree hash with three Keccak states per warp (keccak_warp.cuh), for launches
// whose leaves leave the SMs so empty that a permutation's latency counts.  A
// thread-block cluster of Q CTAs (W warps each) takes one message: warp w of
// CTA q hashes chunks 3 (qW + w) .. + 2, then those 3 QW further on, and
// stores each digest in the shared memory of the cluster's first CTA, whose
// warp 0 then hashes the digests (the root) and, for Encaps, derives the key.
LWE_DEV void st_cluster_u32(uint32_t addr, uint32_t v) {
  asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}

__global__ void __maxnreg__(112) k_tree_warp(TreeArgs a) {
  extern __shared__ uint64_t sdig[];  // [m][4], used in the cluster's first CTA
  pdl_trigger();
  uint32_t q, nq;
  asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(q));
  asm("mov.u32 %0, %%cluster_nctarank;" : "=r"(nq));
  const uint32_t e = blockIdx.x / nq, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint32_t nw = blockDim.x >> 5;
  const KeccakTri km = keccak_tri(lane);
  // every CTA of the cluster has started before any stores into the first
  if (nq > 1) cluster_barrier();
  pdl_wait();
  const uint8_t *msg = a.msg_ptrs ? a.msg_ptrs[e] : a.msgs + (size_t)e * a.stride;
  const uint32_t dig0 = cluster_map(sdig, 0);
  const uint32_t len = a.tail_len && e == a.count - 1 ? a.tail_len : a.len;
  const uint32_t mc = (len + LWE_TREE_CHUNK - 1) / LWE_TREE_CHUNK;
  uint32_t s[5];
  for (uint32_t c0 = 3 * (q * nw + warp); c0 < mc; c0 += 3 * nq * nw) {
    const uint32_t c = c0 + km.grp, off = c * LWE_TREE_CHUNK;
    const bool in = c < mc && LWE_BOUNDS(off < len, 106);
    sha3_256_tri<true>(km, msg + (in ? off : 0),
                       in ? min((uint32_t)LWE_TREE_CHUNK, len - off) : 0u, s);
    const uint32_t v = tri_digest_word(km, s);
    if (in && lane < 30 && km.r < 8) st_cluster_u32(dig0 + 4 * (8 * c + km.r), v);
  }
  if (nq > 1) cluster_barrier();  // every digest is in the first CTA's shared memory
  else __syncthreads();
  if (q != 0 || warp != 0) return;
  sha3_256_tri<false>(km, reinterpret_cast<const uint8_t *>(sdig), km.grp ? 0u : 32 * mc, s);
  tree_tri_out(a, e, km.grp == 0, km, lane, s);
}

// Tree hash in two launches: long messages, and batches beyond what one CTA per
// SM packs.  k_tree_leaves hashes every 1024-byte chunk of the batch on its own
// thread (message e's chunk c on thread e m + c, all SMs busy whatever the
// batch size) and writes the digests to a.dig ([count][m][4] words);
// k_tree_roots then runs the roots, sequential sponges over 32 m bytes, three
// per warp with ten threads each (keccak_warp.cuh), which takes 2.3 us a
// permutation against one thread's 4.7-5.6, and for Encaps derives the keys.
// k_tree gives each message a group of up to 256 threads and runs the root on
// one thread while the group waits.
__global__ void __launch_bounds__(256) k_tree_leaves(TreeArgs a) {
  pdl_trigger();
  pdl_wait();
  const uint64_t L = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (L >= (uint64_t)a.count * a.m) return;
  const uint32_t e = (uint32_t)(L / a.m), c = (uint32_t)(L % a.m);
  const uint8_t *msg = a.msg_ptrs ? a.msg_ptrs[e] : a.msgs + (size_t)e * a.stride;
  const uint32_t off = c * LWE_TREE_CHUNK;
  if (!LWE_BOUNDS(off < a.len && 4 * (L + 1) <= a.dig_words, 114)) return;
  uint64_t s[25];
  sha3_256_global(msg + off, min((uint32_t)LWE_TREE_CHUNK, a.len - off), s);
  uint4 *d = reinterpret_cast<uint4 *>(a.dig + 4 * L);
  d[0] = make_uint4((uint32_t)s[0], (uint32_t)(s[0] >> 32), (uint32_t)s[1], (uint32_t)(s[1] >> 32));
  d[1] = make_uint4((uint32_t)s[2], (uint32_t)(s[2] >> 32), (uint32_t)s[3], (uint32_t)(s[3] >> 32));
}

// The leaves with three states per warp, where one thread per leaf would leave
// the SMs behind a few warps' 5.6 us permutations.
__global__ void __launch_bounds__(64) k_tree_leaves_tri(TreeArgs a) {
  pdl_trigger();
  const uint32_t lane = threadIdx.x & 31;
  const KeccakTri km = keccak_tri(lane);
  const uint64_t L = 3ull * (blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5)) + km.grp;
  pdl_wait();
  const uint32_t e = (uint32_t)(L / a.m), off = (uint32_t)(L % a.m) * LWE_TREE_CHUNK;
  const bool in = L < (uint64_t)a.count * a.m &&
                  LWE_BOUNDS(off < a.len && 4 * (L + 1) <= a.dig_words, 114);
  const uint8_t *msg = !in ? nullptr : a.msg_ptrs ? a.msg_ptrs[e] : a.msgs + (size_t)e * a.stride;
  uint32_t s[5];
  sha3_256_tri<true>(km, msg + (in ? off : 0), in ? min((uint32_t)LWE_TREE_CHUNK, a.len - off) : 0u,
                     s);
  const uint32_t v = tri_digest_word(km, s);
  if (in && lane < 30 && km.r < 8) reinterpret_cast<uint32_t *>(a.dig + 4 * L)[km.r] = v;
}

__global__ void __launch_bounds__(64) k_tree_roots(TreeArgs a) {
  pdl_trigger();
  const uint32_t lane = threadIdx.x & 31;
  const KeccakTri km = keccak_tri(lane);
  const uint32_t e = 3 * (blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5)) + km.grp;
  pdl_wait();
  const bool in = e < a.count && LWE_BOUNDS(4ull * (e + 1) * a.m <= a.dig_words, 115);
  uint32_t s[5];
  sha3_256_tri<false>(km, reinterpret_cast<const uint8_t *>(a.dig + (in ? 4ull * e * a.m : 0)),
                      in ? 32 * a.m : 0u, s);
  tree_tri_out(a, e, in, km, lane, s);
}

__global__ void __launch_bounds__(128) k_final_key(FinalKeyArgs a) {
  pdl_trigger();
  pdl_wait();
  const uint32_t e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= a.count) return;
  // all-ones when the re-encryption matched (flag == 0), else zero
  const uint32_t f = a.flags[e];
  const uint64_t keep = (uint64_t)0 - (uint64_t)(((f | (0u - f)) >> 31) ^ 1u);
  const uint64_t *kp = reinterpret_cast<const uint64_t *>(a.kprime + 32 * (size_t)e);
  const uint64_t *z = reinterpret_cast<const uint64_t *>(a.z_ptrs ? a.z_ptrs[e] + a.z_off : a.z);
  const uint64_t *hc = reinterpret_cast<const uint64_t *>(a.hc + 32 * (size_t)e);
  uint64_t lanes[SHA3_RATE / 8];
  lanes_zero(lanes);
  for (int i = 0; i < 4; i++) lanes[i] = (kp[i] & keep) | (z[i] & ~keep);
  for (int i = 0; i < 4; i++) lanes[4 + i] = hc[i];
  uint64_t s[25];
  sha3_256_lanes(lanes, 64, s);
  sha3_digest(s, a.K + 32 * (size_t)e);
}

// ---------------------------------------------------------------------------
// Operand preparation of the tensor path: the columns of [A | B] split into
// signed 8-bit limbs, x = lo + 256 hi (mod 2^16), written K-major as bf16
// (limbs[l][c][i]); a 64 x 64 tile is transposed through shared memory.
// ---------------------------------------------------------------------------
// The 64 x 64 tile sits in shared memory with its 16-byte chunks swizzled:
// chunk q of row r at position q ^ ((r >> 3) & 7).  The transposed read
// (each lane a column, lanes over rows 8 apart) then meets 8 different
// chunks, all 32 banks, where an unswizzled (even a padded) row layout put
// those rows on one or two banks.
LWE_DEV uint32_t limb_tile_at(uint32_t r, uint32_t c) {
  return r * 64 + 8 * ((c >> 3) ^ ((r >> 3) & 7)) + (c & 7);
}

// One instance per source of A: the stored one carries no AES state, so it
// needs few registers and more CTAs per SM keep more loads in flight.  The
// regenerating one walks 64 x TC tiles with one CTA per SM, which fills the AES
// tables once, TC / 64 blocks side by side per thread; a CTA per 64 x 64 tile,
// as for the stored one, filled 128 KB for every 8 KB that it made.  TC = 64
// where tiles of 128 would not fill the SMs, and NT = 256 threads where there
// is one 64 x 64 tile per CTA, which leaves the other stream's kernels registers.
// (Encaps and Decaps with the key not bound: 200 requests at n = 4096 832 ->
// 678 us, 300 at 1344 269 -> 257.)
template <bool FUSED, uint32_t TC, uint32_t NT>
__global__ void __launch_bounds__(NT, !FUSED ? 6 : NT == 256 ? 3 : 1) k_limbs(GemmLimbArgs a) {
  extern __shared__ uint32_t sT[];
  constexpr uint32_t NH = 8 * TC / NT;  // 16-byte chunks per thread, FUSED
  __shared__ __align__(16) uint16_t tile[64 * TC];
  const uint32_t n = a.n, nch = n / 8, ncols = n + (a.B ? 8u : 0u), tid = threadIdx.x;
  const uint32_t mq = (1u << a.logq) - 1u, mm = mq | (mq << 16);
  const uint32_t tiles_c = (ncols + TC - 1) / TC, tiles = tiles_c * ((n + 63) / 64);
  auto at = [](uint32_t r, uint32_t c) { return (c >> 6) * 4096 + limb_tile_at(r, c & 63); };
  // one or two tiles per CTA (TC = 64) do not pay for the index tables
  constexpr bool USE_F = FUSED && TC == 128;
  AesTab tab;
  AesF F;
  uint32_t rk[44];  // USE_F: round keys 3 .. 10 in the first 32
  pdl_trigger();
  if (FUSED) {
    aes_fill_smem(sT, g_aes_img);
    __syncthreads();
  }
  pdl_wait();
  if (FUSED && !USE_F) {
    tab = aes_tab(sT);
    uint32_t key[4];
    aes_load_key(a.seedA, key);
    aes_key_expand(tab, key, rk);
  }
  if (USE_F) {
    uint4 *sF = reinterpret_cast<uint4 *>(reinterpret_cast<uint8_t *>(sT) + PRD_F_OFF);
    uint32_t *srk = reinterpret_cast<uint32_t *>(reinterpret_cast<uint8_t *>(sT) + PRD_RK_OFF(1));
    tab = aes_tab(sT);
    if (prd_warp() == 0) prd_expand_key(tab, a.seedA, srk);
    __syncthreads();
    aes_f_fill(sF, tab, srk, 0, tid, NT);
    __syncthreads();
    prd_load_rk(srk, rk);
    F = aes_f_open(sF, srk);
  }
  for (uint32_t tl = blockIdx.x; tl < tiles; tl += gridDim.x) {
    const uint32_t c0 = (tl % tiles_c) * TC, i0 = tl / tiles_c * 64;
    if (FUSED) {
      constexpr uint32_t RP = 64 / NH;  // rows per pass of the threads
      const uint32_t cq = tid % (TC / 8), r = tid / (TC / 8), c = c0 + 8 * cq;
      uint4 v[NH];
      if (c < n) {  // rows beyond n are counters whose blocks nothing reads
        uint32_t s[NH][4];
        if (USE_F) {
#pragma unroll
          for (uint32_t h = 0; h < NH; h++)
            aes_f_start(F, tab, 0, (i0 + r + RP * h) * nch + c / 8, s[h]);
          aes_rounds_3_9<NH>(tab, rk, s);
        }
#pragma unroll
        for (uint32_t h = 0; h < NH; h++) {
          v[h] = USE_F ? aes_last(tab, rk + 28, s[h])
                       : aes_ctr_block(tab, rk, 0, (uint64_t)(i0 + r + RP * h) * nch + c / 8);
          v[h] = make_uint4(v[h].x & mm, v[h].y & mm, v[h].z & mm, v[h].w & mm);
        }
      } else {
#pragma unroll
        for (uint32_t h = 0; h < NH; h++)
          v[h] = a.B && c == n && i0 + r + RP * h < n ? ld_nc_u4(a.B + 16 * (size_t)(i0 + r + RP * h))
                                                      : make_uint4(0, 0, 0, 0);
      }
#pragma unroll
      for (uint32_t h = 0; h < NH; h++)
        *reinterpret_cast<uint4 *>(&tile[at(r + RP * h, 8 * cq)]) = v[h];
    } else {
      for (uint32_t idx = tid; idx < 512; idx += NT) {
        const uint32_t r = idx >> 3, cq = idx & 7;
        const uint32_t i = i0 + r, c = c0 + 8 * cq;
        uint4 v = make_uint4(0, 0, 0, 0);
        if (i < n) {
          if (c + 8 <= n)
            v = ld_nc_u4(a.A + (size_t)i * n + c);
          else if (a.B && c == n)
            v = ld_nc_u4(a.B + 16 * (size_t)i);
        }
        *reinterpret_cast<uint4 *>(&tile[at(r, 8 * cq)]) = v;
      }
    }
    __syncthreads();
    for (uint32_t idx = tid; idx < 8 * TC; idx += NT) {
      const uint32_t cl = idx >> 3, ic = idx & 7;
      const uint32_t c = c0 + cl, i = i0 + 8 * ic;
      if (c >= ncols || i >= n) continue;
      uint32_t lo[4], hi[4];
#pragma unroll
      for (int t = 0; t < 8; t += 2) {
        float fl[2], fh[2];
#pragma unroll
        for (int u = 0; u < 2; u++) {
          const int x = tile[at(8 * ic + t + u, cl)];
          const int l = (int)(int8_t)(uint8_t)(x & 0xff);
          const int h = (int)(int8_t)(uint8_t)(((x - l) >> 8) & 0xff);
          fl[u] = (float)l;
          fh[u] = (float)h;
        }
        __nv_bfloat162 bl = __floats2bfloat162_rn(fl[0], fl[1]);
        __nv_bfloat162 bh = __floats2bfloat162_rn(fh[0], fh[1]);
        lo[t / 2] = *reinterpret_cast<uint32_t *>(&bl);
        hi[t / 2] = *reinterpret_cast<uint32_t *>(&bh);
      }
      uint16_t *L = a.limbs;
      *reinterpret_cast<uint4 *>(L + (size_t)c * n + i) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
      *reinterpret_cast<uint4 *>(L + ((size_t)ncols + c) * n + i) =
          make_uint4(hi[0], hi[1], hi[2], hi[3]);
    }
    if (FUSED) __syncthreads();  // the tile is read before the next one is written
  }
}

__global__ void k_s_to_bf16(const int8_t *__restrict__ S, uint64_t count, uint16_t *out) {
  pdl_trigger();
  pdl_wait();
  for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < count;
       i += (uint64_t)gridDim.x * blockDim.x) {
    __nv_bfloat16 b = __float2bfloat16_rn((float)S[i]);
    out[i] = *reinterpret_cast<uint16_t *>(&b);
  }
}

#include "pp_kernels.cuh"

// ---------------------------------------------------------------------------
// Host-side launch wrappers (called from lwe_api.cu)
// ---------------------------------------------------------------------------
// ---------------------------------------------------------------------------
// Measurement probes: the instruction sequences of the two integer-bound
// kernels without memory traffic, for their practical peak on this GPU.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) k_probe_keccak(uint32_t iters, uint32_t *sink) {
  const uint32_t gid = blockIdx.x * blockDim.x + threadIdx.x;
  uint64_t s[25];
#pragma unroll
  for (int i = 0; i < 25; i++) s[i] = ((uint64_t)gid << 32) ^ (uint64_t)(i * 0x9E3779B9u);
  for (uint32_t it = 0; it < iters; it++) keccak_f1600(s);
  sink[gid] = (uint32_t)(s[0] ^ s[7] ^ s[24]);
}

__global__ void __launch_bounds__(512, 1) k_probe_aes(uint32_t iters, uint32_t *sink) {
  extern __shared__ uint32_t sT[];
  aes_fill_smem(sT, g_aes_img);
  __syncthreads();
  const AesTab tab = aes_tab(sT);
  const uint32_t gid = blockIdx.x * blockDim.x + threadIdx.x;
  uint32_t key[4] = {gid, gid * 0x9E3779B9u, ~gid, gid ^ 0x5A5A5A5Au}, rk[44];
  aes_key_expand(tab, key, rk);
  uint32_t acc = 0;
  const uint64_t base = (uint64_t)gid * iters;
  for (uint32_t b = 0; b < iters; b += 2) {  // two blocks in flight, the plain sequence
    const uint4 v = aes_ctr_block(tab, rk, 3, base + b);
    const uint4 w = aes_ctr_block(tab, rk, 3, base + b + 1);
    acc ^= v.x ^ v.y ^ v.z ^ v.w ^ w.x ^ w.y ^ w.z ^ w.w;
  }
  sink[gid] = acc;
}

// The windowed sequence of k_noise: per lane, NOISE_RUN / 32 blocks of one
// run, two at a time; the window constants of 32 runs worked out at once
// (one per lane) and passed by shuffles.
__global__ void __launch_bounds__(512, 1) k_probe_aes_run(uint32_t iters, uint32_t *sink) {
  extern __shared__ uint32_t sT[];
  aes_fill_smem(sT, g_aes_img);
  __syncthreads();
  const AesTab tab = aes_tab(sT);
  const uint32_t gid = blockIdx.x * blockDim.x + threadIdx.x, lane = threadIdx.x & 31;
  // one key per warp, as for a run of the noise (the shared window
  // constants depend on it)
  const uint32_t wid = gid >> 5;
  uint32_t key[4] = {wid, wid * 0x9E3779B9u, ~wid, wid ^ 0x5A5A5A5Au}, rk[44];
  aes_key_expand(tab, key, rk);
  uint32_t acc = 0;
  const uint64_t base = (uint64_t)wid * iters * 32;
  constexpr uint32_t PER = NOISE_RUN / 32;  // blocks per lane and run
  for (uint32_t g = 0; g < iters; g += 32 * PER) {
    const AesCtrRun mine = aes_ctr_run(tab, rk, 3, base + 32 * (uint64_t)(g + PER * lane));
    for (uint32_t jr = 0; jr < 32 && g + PER * jr < iters; jr++) {
      const uint64_t first = base + 32 * (uint64_t)(g + PER * jr);
      const AesCtrRun win = aes_ctr_run_shfl(mine, jr);
      const uint32_t x0 = (uint32_t)(first & 255u) + lane;
#pragma unroll
      for (uint32_t j = 0; j < PER; j += 2) {
        const uint4 v = aes_ctr_run_block(tab, rk, win, x0 + 32 * j);
        const uint4 w = aes_ctr_run_block(tab, rk, win, x0 + 32 * j + 32);
        acc ^= v.x ^ v.y ^ v.z ^ v.w ^ w.x ^ w.y ^ w.z ^ w.w;
      }
    }
  }
  sink[gid] = acc;
}

__global__ void __launch_bounds__(32) k_probe_keccak_warp(uint32_t iters, uint32_t *sink) {
  __shared__ uint32_t sh[2][25];
  const uint32_t lane = threadIdx.x, t = lane % 25;
  const KeccakTri km = keccak_tri(lane);
  uint32_t s[5];
#pragma unroll
  for (uint32_t i = 0; i < 5; i++)
    s[i] = tri_half(((uint64_t)blockIdx.x << 32) ^ (uint64_t)(tri_lane(km, i) * 0x9E3779B9u), km.h);
  for (uint32_t it = 0; it < iters; it++) keccak_f1600_tri(km, s);
  if (lane < 10)
#pragma unroll
    for (uint32_t i = 0; i < 5; i++) sh[km.h][tri_lane(km, i)] = s[i];
  __syncwarp();
  uint64_t v = 0;
  for (uint32_t b = 0; b < 32; b++)
    v |= ((uint64_t)((sh[0][t] >> b) & 1u) << (2 * b)) | ((uint64_t)((sh[1][t] >> b) & 1u) << (2 * b + 1));
  sink[32 * blockIdx.x + lane] = (uint32_t)(v ^ (v >> 32));
}

int launch_probe(int kind, uint32_t ctas, uint32_t iters, uint32_t *sink, cudaStream_t st) {
  if (kind == 0) {
    k_probe_keccak<<<ctas, 256, 0, st>>>(iters, sink);
    return 0;
  }
  if (kind == 1) {
    k_probe_aes<<<ctas, 512, AES_SMEM_BYTES, st>>>(iters, sink);
    return 0;
  }
  if (kind == 2) {
    k_probe_keccak_warp<<<ctas, 32, 0, st>>>(iters, sink);
    return 0;
  }
  if (kind == 3) {
    k_probe_aes_run<<<ctas, 512, AES_SMEM_BYTES, st>>>(iters, sink);
    return 0;
  }
  return -1;
}

static int grid_for(uint64_t work, int per_cta, int max_ctas) {
  uint64_t g = (work + per_cta - 1) / per_cta;
  if (g > (uint64_t)max_ctas) g = max_ctas;
  if (g < 1) g = 1;
  return (int)g;
}

cudaError_t lwe_upload_aes_table(const uint32_t T0[256]) {
  cudaError_t e = cudaMemcpyToSymbol(g_aes_T0, T0, 256 * sizeof(uint32_t));
  if (e != cudaSuccess) return e;
  std::vector<uint32_t> img(AES_TABLE_WORDS);
  for (uint32_t i = 0; i < AES_TABLE_WORDS; i++) img[i] = aes_table_word(T0, i);
  return cudaMemcpyToSymbol(g_aes_img, img.data(), AES_TABLE_WORDS * sizeof(uint32_t));
}

// CTAs that run at once in clusters of R, per device: of the AES product
// kernels (one per SM) and of k_sa (two).  Clusters do not straddle GPCs, so on
// a 152-SM GB300 not every R uses every SM: 152, 152, 138, 144, 140, 138, 105,
// 120 for R = 1 .. 8, and 304, 304, 291, 296, 290, 276, 266, 288 of k_sa.
// Filled by lwe_kernel_smem_setup.
static uint32_t g_cluster_slots[128][9], g_sa_slots[128][9];

// the current device's row of a table
static const uint32_t *device_slots(const uint32_t (*table)[9]) {
  int dev = 0;
  return cudaGetDevice(&dev) == cudaSuccess && dev >= 0 && dev < 128 ? table[dev] : nullptr;
}
static uint32_t cluster_slots(const uint32_t *row, uint32_t R, uint32_t per_sm, uint32_t sms) {
  return std::max(R, row && row[R] ? row[R] : per_sm * sms / R * R);
}

static cudaError_t query_cluster_slots() {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess || dev < 0 || dev >= 128) return e;
  for (uint32_t R = 1; R <= 8; R++) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(1, R, 1);
    cfg.blockDim = dim3(512, 1, 1);
    cfg.dynamicSmemBytes = PRD_SMEM;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = 1;
    at[0].val.clusterDim.y = R;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    int n = 0;
    e = cudaOccupancyMaxActiveClusters(&n, k_sa_gen<false>, &cfg);
    if (e != cudaSuccess) return e;
    g_cluster_slots[dev][R] = (uint32_t)n * R;
    cfg.blockDim = dim3(256, 1, 1);
    cfg.dynamicSmemBytes = 0;
    e = cudaOccupancyMaxActiveClusters(&n, k_sa<false>, &cfg);
    if (e != cudaSuccess) return e;
    g_sa_slots[dev][R] = (uint32_t)n * R;
  }
  return cudaSuccess;
}

// How many ways (1 .. 8, one cluster) to split each of `tiles` equal pieces
// of `work` units so that the last wave wastes least; every CTA has a fixed
// cost of `fixed` units.
static uint32_t best_split(uint64_t tiles, uint32_t work, uint32_t fixed, uint32_t sms) {
  const uint32_t *row = device_slots(g_cluster_slots);
  uint32_t best = 1;
  uint64_t best_cost = ~0ull;
  for (uint32_t R = 1; R <= 8 && R <= work; R++) {
    const uint32_t slots = cluster_slots(row, R, 1, sms);
    const uint64_t waves = (tiles * R + slots - 1) / slots;
    const uint64_t cost = waves * ((work + R - 1) / R + fixed);
    if (cost < best_cost) {
      best_cost = cost;
      best = R;
    }
  }
  return best;
}

cudaError_t lwe_kernel_smem_setup() {
  cudaError_t e;
  e = cudaFuncSetAttribute(k_expand_A, cudaFuncAttributeMaxDynamicSharedMemorySize, AES_SMEM_BYTES);
  if (e != cudaSuccess) return e;
  for (auto k : {k_noise<false>, k_noise<true>}) {
    e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, NOISE_SMEM_BYTES);
    if (e != cudaSuccess) return e;
  }
  e = cudaFuncSetAttribute(k_noise_table, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           NOISE_SMEM_BYTES);
  if (e != cudaSuccess) return e;
  e = cudaFuncSetAttribute(k_mul_as_gen, cudaFuncAttributeMaxDynamicSharedMemorySize, AS_GEN_SMEM);
  if (e != cudaSuccess) return e;
  e = cudaFuncSetAttribute(k_mul_as_gen_split, cudaFuncAttributeMaxDynamicSharedMemorySize, PRD_SMEM);
  if (e != cudaSuccess) return e;
  e = cudaFuncSetAttribute(k_sa_gen<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, PRD_SMEM);
  if (e != cudaSuccess) return e;
  e = cudaFuncSetAttribute(k_sa_gen<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, PRD_SMEM);
  if (e != cudaSuccess) return e;
  e = query_cluster_slots();
  if (e != cudaSuccess) return e;
  e = cudaFuncSetAttribute(k_probe_aes, cudaFuncAttributeMaxDynamicSharedMemorySize, AES_SMEM_BYTES);
  if (e != cudaSuccess) return e;
  e = cudaFuncSetAttribute(k_probe_aes_run, cudaFuncAttributeMaxDynamicSharedMemorySize, AES_SMEM_BYTES);
  if (e != cudaSuccess) return e;
  e = cudaFuncSetAttribute(k_pp_expand_A, cudaFuncAttributeMaxDynamicSharedMemorySize, AES_SMEM_BYTES);
  if (e != cudaSuccess) return e;
  e = cudaFuncSetAttribute(k_pp_noise, cudaFuncAttributeMaxDynamicSharedMemorySize, AES_SMEM_BYTES);
  if (e != cudaSuccess) return e;
  for (auto k : {k_limbs<true, 64, 256>, k_limbs<true, 64, 512>, k_limbs<true, 128, 512>}) {
    e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, PRD_SMEM);
    if (e != cudaSuccess) return e;
  }
  return e;
}

void launch_expand_A(const uint8_t *seeds, uint32_t seed_stride, uint32_t count, uint32_t n,
                     uint32_t logq, uint16_t *A, uint64_t a_stride, int num_sms, cudaStream_t st) {
  const uint64_t nblk = (uint64_t)n * n / 8;
  const int gx = grid_for(nblk, 512 * 4, num_sms);
  launch_k(k_expand_A, dim3(gx, count), 512, AES_SMEM_BYTES, st, seeds, seed_stride, n, logq, A,
           a_stride);
}

void launch_noise_table(const NoiseArgs &a, int8_t *out, cudaStream_t st) {
  launch_k(k_noise_table, 1, 512, NOISE_SMEM_BYTES, st, a, out);
}

void launch_noise(const NoiseArgs &a, int num_sms, cudaStream_t st, bool pp) {
  const int g = grid_for((uint64_t)a.count * a.runs_per_item, a.run == NOISE_RUN ? 16 : 1, num_sms);
  if (pp)
    launch_k(k_noise<true>, g, 512, NOISE_SMEM_BYTES, st, a);
  else
    launch_k(k_noise<false>, g, 512, NOISE_SMEM_BYTES, st, a);
}

void launch_mul_as(const MulAsArgs &a, uint32_t count, bool fused, int num_sms, cudaStream_t st) {
  const uint32_t rows = a.rows ? a.rows : a.n, sms = (uint32_t)std::max(num_sms, 1);
  if (!fused) {
    // 8 warps per 16-row tile (78 registers: three CTAs per SM), but 4 (94:
    // five) where those take in one wave what 8 leave a short second wave of.
    // Back to back, with 8 and with 4: n = 7008 (2.9 tiles per SM) 16.7 and
    // 18.5 us, 7312 (3.01) 22.7 and 20.6, 8192 27.2 and 23.0, 12160 (5) 51.3
    // and 45.6, 12176 (5.01) 51.3 and 61.4, 14592 (6) 71.2 and 84.1, 16384 94.2
    // and 101.7
    const uint64_t tiles = (uint64_t)(rows / 16) * count;
    if (tiles > 3ull * sms && tiles <= 5ull * sms)
      launch_k(k_mul_as<4>, dim3(rows / 16, count), 128, 0, st, a);
    else
      launch_k(k_mul_as<8>, dim3(rows / 16, count), 256, 0, st, a);
    return;
  }
  const uint64_t units = (uint64_t)count * (rows / 16);
  if (units >= 32ull * sms) {
    launch_k(k_mul_as_gen, sms, 512, AS_GEN_SMEM, st, a, count);
    return;
  }
  // Clusters of R CTAs walk the 16-row tiles of each item.  A tile's time goes
  // by its groups of 4 chunks, 16 per CTA and step; a cluster's barriers cost
  // about as much as one more step, the last tile's less.  With 1, 2 and 4 CTAs:
  // n = 1344 12.5, 18.5, 20.6 us; 3600 43.1, 41.1, 59.4; 5008 79.9, 77.9, 98.4;
  // 6208 97.1, 111, 123; 8192 156, 152, 187; 16384 524, 553, 626.  One round:
  // KeyGen, Encaps and Decaps at n = 640 with 1, 2 and 3 178.9, 176.1, 174.1,
  // at n = 976 193.9, 187.5, 194.6 (two rounds with 3).
  const uint32_t tiles = rows / 16, groups = (a.n / 8 + 3) / 4;
  const uint32_t *row = device_slots(g_cluster_slots);
  uint32_t best_R = 1, best_G = 1;
  uint64_t best_cost = ~0ull;
  for (uint32_t R = 1; R <= 8; R++) {
    const uint32_t slots = cluster_slots(row, R, 1, sms);
    const uint32_t G = std::min(tiles, std::max<uint32_t>(1u, slots / (R * count)));
    const uint64_t ctas = (uint64_t)R * G * count;
    const uint64_t rounds = ((ctas + slots - 1) / slots) * ((tiles + G - 1) / G);
    const uint64_t cost = rounds * groups * 840 / R + (R > 1 ? (15 * rounds - 6) * 840 : 0);
    if (cost < best_cost) {
      best_cost = cost;
      best_R = R;
      best_G = G;
    }
  }
  launch_k_cluster(k_mul_as_gen_split, dim3(best_R, best_G, count), 512, PRD_SMEM, st, best_R, a);
}

void launch_decrypt(const DecryptArgs &a, uint32_t count, cudaStream_t st) {
  launch_k(k_decrypt, count, 256, 0, st, a);
}

void launch_mul_sa(const MulSaArgs &a, uint32_t items, bool fused, bool cmp, int num_sms,
                   cudaStream_t st) {
  const uint32_t sms = (uint32_t)std::max(num_sms, 1);
  const uint32_t steps = ((a.row1 ? a.row1 : a.n) - a.row0) / 16;  // 16-row steps
  uint32_t R, cgs = 1, cbs = (a.n + 63) / 64;
  if (fused) {
    R = best_split((uint64_t)cbs * items, steps, 14, sms);
  } else {
    // column groups per CTA and row split: few waves of the CTAs that run at
    // once (two per SM at 88 registers, less what clusters leave), counting 64
    // steps for a CTA's start and end, and two row steps per warp at least; of
    // equals the narrowest, whose clusters are small.  A from memory, n = 8192:
    // 256 CTAs as 1 x 2, 2 x 4 or 4 x 8 take 28.6, 30.8 and 30.8 us, 384 as 1 x
    // 3 38.8; n = 16384, two items: 2 x 1 171, 4 x 7 227.
    // Small calls: n = 976, 10 items, 160 CTAs as 1 x 1 9.9 us, 280 as 4 x 7,
    // more than the 266 that run at once, 16.5; 640, 20 items, 1 x 1 9.1, 300 as
    // 2 x 3 13.9
    const uint32_t *row = device_slots(g_sa_slots);
    uint64_t best_cost = ~0ull;
    R = 1;
    for (uint32_t g = 1; g <= 4; g *= 2)
      for (uint32_t r = 1; r <= 8 && (r == 1 || steps * g >= 16 * r); r++) {
        const uint64_t slots = cluster_slots(row, r, 2, sms);
        const uint64_t ctas = (uint64_t)((a.n + 64 * g - 1) / (64 * g)) * items * r;
        const uint64_t cost = (ctas + slots - 1) / slots * ((uint64_t)steps * g / r + 64);
        if (cost < best_cost) {
          best_cost = cost;
          cgs = g;
          R = r;
        }
      }
    cbs = (a.n + 64 * cgs - 1) / (64 * cgs);
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(cbs + (a.vcols ? 1 : 0), R, items);
  cfg.dynamicSmemBytes = fused ? PRD_SMEM : 0;
  cfg.blockDim = dim3(fused ? 512 : 256, 1, 1);
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = g_launch_pdl ? 1 : 0;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = 1;
  attr[1].val.clusterDim.y = R;
  attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = R > 1 ? 2 : 1;
  if (fused) {
    if (cmp)
      cudaLaunchKernelEx(&cfg, k_sa_gen<true>, a);
    else
      cudaLaunchKernelEx(&cfg, k_sa_gen<false>, a);
  } else {
    if (cmp)
      cudaLaunchKernelEx(&cfg, k_sa<true>, a, cgs);
    else
      cudaLaunchKernelEx(&cfg, k_sa<false>, a, cgs);
  }
}

void launch_keygen_seeds(const KeygenSeedArgs &a, uint32_t warp_max, cudaStream_t st) {
  if (a.count <= warp_max) {
    launch_k(k_keygen_seeds_warp, (a.count + 3) / 4, 128, 0, st, a);
    return;
  }
  launch_k(k_keygen_seeds, (a.count + 63) / 64, 64, 0, st, a);
}

void launch_derive(const DeriveArgs &a, uint32_t warp_max, cudaStream_t st) {
  if (a.count <= warp_max) {
    launch_k(k_derive_warp, (a.count + 3) / 4, 128, 0, st, a);
    return;
  }
  launch_k(k_derive, (a.count + 31) / 32, 64, 0, st, a);
}

// Few messages: three Keccak states per warp.  Else one state per thread, one
// CTA per SM where the batch allows (the leaf work is one wave: CTAs of equal
// size spread it evenly): k_tree_bal and k_tree_dense, then k_tree for one wave
// of short messages or without a digest buffer (at most TREE_MAX_THREADS
// threads and 48 KB of digests per CTA); two launches for the rest.
void launch_tree(TreeArgs &a, int num_sms, uint32_t warp_max, cudaStream_t st) {
  a.m = (a.len + LWE_TREE_CHUNK - 1) / LWE_TREE_CHUNK;
  const uint32_t sms = num_sms > 0 ? (uint32_t)num_sms : 1u;
  const bool dig_fits = a.dig && (uint64_t)a.count * a.m * 4 <= a.dig_words;
  if (a.count <= warp_max) {
    if (a.m > 96 && dig_fits) {
      // more leaves than a cluster of 8 CTAs runs at full speed
      const uint64_t warps = ((uint64_t)a.count * a.m + 2) / 3;
      launch_k(k_tree_leaves_tri, (uint32_t)((warps + 1) / 2), 64, 0, st, a);
      launch_k(k_tree_roots, (a.count + 5) / 6, 64, 0, st, a);
      return;
    }
    const TreeWarpShape s = tree_warp_shape(a.m);
    launch_k_cluster(k_tree_warp, a.count * s.ctas, 32 * s.warps, (size_t)a.m * 32, st, s.ctas, a);
    return;
  }
  auto two_launches = [&] {
    // small leaf CTAs when the batch fills the SMs only a few warps deep
    const uint64_t leaves = (uint64_t)a.count * a.m;
    const uint32_t lt = leaves >= (uint64_t)sms * 1024 ? 256u : 64u;
    // plainly: started beside the last CTAs of the launch before it (the
    // GEMM's, in Encaps), the leaves crowd on the SMs that come free first,
    // and the warps of one SM set the time (Encaps of 6000 requests at n =
    // 208: 365 us, 197 so; 2900 at 1344: 577 and 443)
    const bool pdl = g_launch_pdl;
    g_launch_pdl = false;
    launch_k(k_tree_leaves, (uint32_t)((leaves + lt - 1) / lt), lt, 0, st, a);
    g_launch_pdl = pdl;
    launch_k(k_tree_roots, (a.count + 5) / 6, 64, 0, st, a);
  };
  if (a.m > 128 && dig_fits) {  // few messages per CTA: no packing to gain
    two_launches();
    return;
  }
  {
    // the balanced schedule of k_tree_bal: leaves of full length filling
    // more than 12 and at most 13 warps per CTA, every message's short
    // chunk and root on one warp
    const uint32_t last = a.len - (a.m - 1) * LWE_TREE_CHUNK;
    const uint32_t ml = a.m - (last < LWE_TREE_CHUNK ? 1u : 0u);
    const uint32_t ipc = (a.count + sms - 1) / sms;
    const uint32_t nl = ipc * ml;
    const size_t smem = ((size_t)ipc * (4 * a.m + 1 + 25) + 25 * TB_SLOTS) * 8;
    if (a.m >= 2 && nl > 12 * 32 && nl <= 13 * 32 && ipc <= 32 && smem <= 48 * 1024 &&
        (a.count + ipc - 1) / ipc <= sms) {
      a.ipc = ipc;
      a.ml = ml;
      launch_k(k_tree_bal, (a.count + ipc - 1) / ipc, 512, smem, st, a);
      return;
    }
    // leaves of at most 12 warps: dense packing, roots on the least loaded
    // SMSP (warp 12 + s of SMSP s)
    const size_t smem_d = (size_t)ipc * (4 * a.m + 1) * 8;
    if (a.m >= 2 && ml >= 1 && nl <= 12 * 32 && ipc <= 32 && smem_d <= 48 * 1024 &&
        (a.count + ipc - 1) / ipc <= sms) {
      const uint32_t wl = (nl + 31) / 32;
      uint32_t best = 3, load_best = 99;
      for (int sp = 3; sp >= 0; sp--) {
        const uint32_t load = wl > (uint32_t)sp ? (wl - 1 - sp) / 4 + 1 : 0;  // leaf warps on SMSP sp
        if (load < load_best) {
          load_best = load;
          best = (uint32_t)sp;
        }
      }
      a.ipc = ipc;
      a.ml = ml;
      a.rw = 12 + best;
      launch_k(k_tree_dense, (a.count + ipc - 1) / ipc, 512, smem_d, st, a);
      return;
    }
  }
  uint32_t t = 1;
  while (t < a.m && t < 256) t <<= 1;
  a.tpi = t;
  const uint32_t words = 4 * a.m + 1;
  uint32_t cap = TREE_MAX_THREADS / t;
  cap = std::min<uint32_t>(cap, (48u * 1024u) / (8u * words));
  cap = std::max<uint32_t>(cap, 1u);
  const uint32_t per_sm = (a.count + sms - 1) / sms;
  if (a.m >= 2 && dig_fits && !(a.m <= 16 && per_sm <= 32 && per_sm <= cap)) {
    // more leaves than 13 warps per SM (or than 32 messages): two launches
    // (Encaps of 4096 requests at n = 1344, 22 leaves each, 826 us with
    // k_tree), but k_tree where it is one wave of up to 14 warps and its roots,
    // one thread each, are short (at n = 976, 16 leaves, 28 messages per SM:
    // 442 + 451 us with k_tree, 452 + 490 with two launches; at 29, where
    // k_tree takes two waves, 626 + 618 against 459 + 499)
    two_launches();
    return;
  }
  a.ipc = std::min<uint32_t>(cap, per_sm);
  if (a.ipc == 0) a.ipc = 1;
  const uint32_t threads = (a.ipc * t + 31) / 32 * 32;
  const size_t smem = (size_t)a.ipc * words * 8;
  launch_k(k_tree, (a.count + a.ipc - 1) / a.ipc, threads, smem, st, a);
}

void launch_final_key(const FinalKeyArgs &a, uint32_t warp_max, cudaStream_t st) {
  if (a.count <= warp_max) {
    launch_k(k_final_key_warp, (a.count + 3) / 4, 128, 0, st, a);
    return;
  }
  launch_k(k_final_key, (a.count + 127) / 128, 128, 0, st, a);
}

void launch_gemm_limbs(const GemmLimbArgs &a, int num_sms, cudaStream_t st) {
  const uint32_t ncols = a.n + (a.B ? 8u : 0u), rows = (a.n + 63) / 64;
  const uint32_t sms = (uint32_t)std::max(num_sms, 1), t64 = (ncols + 63) / 64 * rows;
  const uint32_t t128 = (ncols + 127) / 128 * rows;
  if (a.A)
    launch_k(k_limbs<false, 64, 256>, t64, 256, 0, st, a);
  else if (t64 <= sms)
    launch_k(k_limbs<true, 64, 256>, t64, 256, AES_SMEM_BYTES, st, a);
  else if (t128 < sms)
    launch_k(k_limbs<true, 64, 512>, sms, 512, AES_SMEM_BYTES, st, a);
  else
    launch_k(k_limbs<true, 128, 512>, std::min(t128, sms), 512, PRD_SMEM, st, a);
}

void launch_s_to_bf16(const int8_t *S, uint64_t count, uint16_t *out, int num_sms, cudaStream_t st) {
  const int g = grid_for(count, 256 * 8, num_sms * 8);
  launch_k(k_s_to_bf16, g, 256, 0, st, S, count, out);
}

// ---- the paper's own parameter profile ------------------------------------
void launch_pp_expand_A(const uint8_t *seedA, uint32_t n, ModQ M, uint32_t *A, int num_sms,
                        cudaStream_t st) {
  const int g = grid_for((uint64_t)n * n / 4, 512 * 4, num_sms);
  launch_k(k_pp_expand_A, g, 512, AES_SMEM_BYTES, st, seedA, n, M, A);
}

void launch_pp_noise(const PpNoiseArgs &a, int num_sms, cudaStream_t st) {
  uint64_t blocks = 0;
  for (uint32_t s = 0; s < a.nout; s++)
    blocks += a.o[s].kind == PP_BINOMIAL ? (a.o[s].count + 15) / 16 : (a.o[s].count + 7) / 8;
  launch_k(k_pp_noise, grid_for(blocks, 512 * 4, num_sms), 512, AES_SMEM_BYTES, st, a);
}

void launch_pp_as(const PpAsArgs &a, cudaStream_t st) {
  launch_k(k_pp_as, (a.n + 7) / 8, 256, 0, st, a);
}

void launch_pp_encrypt(const PpEncArgs &a, bool cmp, cudaStream_t st) {
  const dim3 grid(a.n / PPE_BN, PP_MBITS / PPE_BM);
  if (cmp)
    launch_k(k_pp_encrypt<true>, grid, 256, 0, st, a);
  else
    launch_k(k_pp_encrypt<false>, grid, 256, 0, st, a);
}

void launch_pp_v(const PpVArgs &a, bool cmp, cudaStream_t st) {
  if (cmp)
    launch_k(k_pp_v<true>, PP_MBITS, 256, 0, st, a);
  else
    launch_k(k_pp_v<false>, PP_MBITS, 256, 0, st, a);
}

void launch_pp_decrypt(const PpDecArgs &a, cudaStream_t st) {
  launch_k(k_pp_decrypt, PP_MBITS, 256, 0, st, a);
}

void launch_pp_limbs(const uint32_t *A, uint32_t n, uint32_t q, uint16_t *limbs, cudaStream_t st) {
  launch_k(k_pp_limbs, dim3(n / 64, n / 64), 256, 0, st, A, n, q, limbs);
}
