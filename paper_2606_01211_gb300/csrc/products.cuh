// products.cuh -- A S + E (Alg. 1) and S' A + E' (Alg. 2) for one request or
// for items of different keys, A streamed from memory or regenerated from its
// seed.  Included once, by kem_kernels.cu (it uses that file's AES image).
//
// Eight columns of S (or rows of S') against n^2 entries of A leave these
// kernels bound by the bytes of A or by its AES blocks, not by arithmetic --
// unless the multiplies crowd the pipes that move the data: with two-row dot
// products (dp2a) an entry of A cost 4 instructions.  Here the multiplies run
// on the tensor cores (mma.sync m16n8k16, f16 operands, f32 accumulators): N
// is the 8 columns of S, M rows or columns of A.  An entry of A enters as its
// two bytes, A = lo + 256 hi, each taken as the f16 with those bits: a
// subnormal of value byte 2^-24, so splitting is one mask and needs no
// conversion, and 2^24 times an accumulator is a whole number, exact while
// below 2^24 (|S| <= 128: PRD_EXACT_K terms; then it is added to integers).
// No masking to log2 q bits is needed before the final one.  Rates measured
// on GB300 (clocks per SM and instruction): f16 / bf16 m16n8k16 2.05; s8
// m16n8k32, which would take the bytes as they are, 16.3, i.e. no faster
// than the copy of A from memory.  tcgen05 has no integer kind on sm_103a
// and its smallest M is 64, which would need the tile in shared memory first.
#pragma once

#define PRD_F_OFF AES_SMEM_BYTES               // F tables (aes.cuh)
#define PRD_RK_OFF(slots) (PRD_F_OFF + (slots) * AES_F_BYTES)
#define PRD_SMEM (PRD_RK_OFF(1) + 176)
#define AS_GEN_SMEM (PRD_RK_OFF(AS_SLOTS) + AS_SLOTS * 176)
#define AS_SLOTS 4                             // keys whose tables a CTA holds at once

#define PRD_EXACT_K 512  // terms of |byte x S| <= 255 x 128 that stay below 2^24

LWE_DEV void mma_f16_k16(float c[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3,
                         uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
      "{%0,%1,%2,%3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// bytes 0 and 2, or 1 and 3, of a word as two f16 subnormals
LWE_DEV uint32_t f16_lo(uint32_t w) { return w & 0x00ff00ffu; }
LWE_DEV uint32_t f16_hi(uint32_t w) { return __byte_perm(w, 0, 0x4341); }

// four int8 as two pairs of f16 whole numbers: 1024 + (x + 128) has x + 128
// in its low byte
LWE_DEV void f16_of_s8(uint32_t w, uint32_t &p01, uint32_t &p23) {
  const __half2 bias = __floats2half2_rn(1152.f, 1152.f);
  w ^= 0x80808080u;
  uint32_t u = __byte_perm(w, 0x64646464u, 0x4140), v = __byte_perm(w, 0x64646464u, 0x4342);
  const __half2 a = __hsub2(*reinterpret_cast<__half2 *>(&u), bias);
  const __half2 b = __hsub2(*reinterpret_cast<__half2 *>(&v), bias);
  p01 = *reinterpret_cast<const uint32_t *>(&a);
  p23 = *reinterpret_cast<const uint32_t *>(&b);
}

// lo + 256 hi (mod 2^32) of two accumulators
LWE_DEV int limb_sum(float lo, float hi) {
  return (int)((uint32_t)__float2int_rn(lo * 16777216.f) +
               ((uint32_t)__float2int_rn(hi * 16777216.f) << 8));
}

LWE_DEV uint32_t cluster_map(const void *p, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;"
               : "=r"(r)
               : "r"((uint32_t)__cvta_generic_to_shared(p)), "r"(rank));
  return r;
}
LWE_DEV int ld_cluster_s32(uint32_t addr) {
  int v;
  asm volatile("ld.shared::cluster.s32 %0, [%1];" : "=r"(v) : "r"(addr) : "memory");
  return v;
}
LWE_DEV void cluster_barrier() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::
                   : "memory");
}

LWE_DEV uint4 ld_stream_u4(const void *p) {
  uint4 v;
  asm("ld.global.nc.L1::no_allocate.v4.u32 {%0, %1, %2, %3}, [%4];"
      : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
      : "l"(p));
  return v;
}

LWE_DEV uint32_t ld_nc_u1(const void *p) { return __ldg(reinterpret_cast<const uint32_t *>(p)); }

// The warp's index, known to be the same for all its lanes: with threadIdx.x /
// 32 the loops over a warp's work look divergent, the table base cannot stay
// in a uniform register, and every AES lookup takes an instruction more to
// add it (537 -> 405 instructions a block in k_sa_gen).
LWE_DEV uint32_t prd_warp() { return __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0); }

// Round keys of the key at `key` to shared memory rks[44], by one warp.
LWE_DEV void prd_expand_key(const AesTab &tab, const uint8_t *key, uint32_t *rks) {
  uint32_t k[4], rk[44];
  aes_load_key(key, k);
  aes_key_expand(tab, k, rk);
  if ((threadIdx.x & 31) == 0) {
#pragma unroll
    for (int i = 0; i < 44; i++) rks[i] = rk[i];
  }
}

// ---------------------------------------------------------------------------
// A S + E.  M = rows of A, K = columns.  In m16n8k16 lane (g, t) = (lane / 4,
// lane % 4) supplies rows g and g + 8 at four values of K; taken as the first
// (or last) four columns of 8-column chunk t, two products per limb consume
// exactly ITS chunk t of those rows: one 16-byte load or one AES block each.
// S^T enters as the 8 bytes of row g at chunk t.  No shuffles and no
// reduction over lanes.
// ---------------------------------------------------------------------------
// the tile's sums: rows i0 + g and i0 + g + 8, columns 2 t and 2 t + 1
LWE_DEV void as_store(const MulAsArgs &a, uint32_t e, uint32_t i0, uint32_t g, uint32_t t,
                      const int v[4]) {
  const uint32_t mq = (1u << a.logq) - 1u;
#pragma unroll
  for (int h = 0; h < 2; h++) {
    const uint32_t i = i0 + g + 8 * h;
    int v0 = v[2 * h], v1 = v[2 * h + 1];
    if (a.E) {
      const uint32_t ev = *reinterpret_cast<const uint16_t *>(a.E + (size_t)e * a.e_stride +
                                                              (size_t)i * 8 + 2 * t);
      v0 += sext8(ev, 0);
      v1 += sext8(ev, 1);
    }
    const uint32_t w = ((uint32_t)v0 & mq) | (((uint32_t)v1 & mq) << 16);
    *reinterpret_cast<uint32_t *>(a.out + (size_t)e * a.out_stride + 16 * (size_t)i + 4 * t) = w;
    if (a.out2)
      *reinterpret_cast<uint32_t *>(a.out2 + (size_t)e * a.out2_stride + 16 * (size_t)i + 4 * t) = w;
  }
}

// 16 rows x 4 chunks: words x of rows g (p) and g + 8 (q), S^T words b of the
// chunk's four column pairs
LWE_DEV void as_mma_chunk(float lo[4], float hi[4], const uint32_t p[4], const uint32_t q[4],
                          const uint32_t b[4]) {
  mma_f16_k16(lo, f16_lo(p[0]), f16_lo(q[0]), f16_lo(p[1]), f16_lo(q[1]), b[0], b[1]);
  mma_f16_k16(hi, f16_hi(p[0]), f16_hi(q[0]), f16_hi(p[1]), f16_hi(q[1]), b[0], b[1]);
  mma_f16_k16(lo, f16_lo(p[2]), f16_lo(q[2]), f16_lo(p[3]), f16_lo(q[3]), b[2], b[3]);
  mma_f16_k16(hi, f16_hi(p[2]), f16_hi(q[2]), f16_hi(p[3]), f16_hi(q[3]), b[2], b[3]);
}

// the accumulators into integers, and cleared
LWE_DEV void as_flush(int sum[4], float lo[4], float hi[4]) {
#pragma unroll
  for (int j = 0; j < 4; j++) {
    sum[j] = (int)((uint32_t)sum[j] + (uint32_t)limb_sum(lo[j], hi[j]));
    lo[j] = hi[j] = 0.f;
  }
}

// Stored A: a CTA takes a tile of 16 rows, its NW warps split the columns
// (chunk groups of 4 in turn) with eight 16-byte loads in flight per lane,
// and their sums meet in shared memory.  Bound by the reads of A: n = 8192
// 23.0 us back to back, when a part of A is still in L2, 27.0 with L2 flushed
// (5.0 TB/s); 16384 94.2 us (5.7 TB/s).  Twelve loads in flight time the same.
template <int NW>
__global__ void __launch_bounds__(32 * NW) k_mul_as(MulAsArgs a) {
  __shared__ int red[128];
  constexpr int U = 4;  // chunk groups in flight
  pdl_trigger();
  if (threadIdx.x < 128) red[threadIdx.x] = 0;
  __syncthreads();
  pdl_wait();
  const uint32_t e = blockIdx.y, i0 = blockIdx.x * 16;
  const uint32_t warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  const uint32_t n = a.n, nch = n / 8;
  const int8_t *St = a.St + (size_t)e * a.st_stride + (size_t)g * n;
  const uint16_t *A0 = a.A + (size_t)e * a.a_stride + (size_t)(i0 + g) * n;
  float lo[4] = {}, hi[4] = {};
  int sum[4] = {};
  uint32_t terms = 0;
  for (uint32_t c0 = 4 * warp + t; c0 - t < nch; c0 += 4 * NW * U) {
    uint4 x[U][2];
    uint2 s[U];
#pragma unroll
    for (int u = 0; u < U; u++) {
      const uint32_t c = c0 + 4 * NW * u;
      const bool in = c < nch && LWE_BOUNDS(i0 + 16 <= (a.rows ? a.rows : n), 109);
#pragma unroll
      for (int h = 0; h < 2; h++)
        x[u][h] = in ? ld_stream_u4(A0 + (size_t)(8 * h) * n + 8 * (size_t)c) : make_uint4(0, 0, 0, 0);
      s[u] = in ? ld_nc_u2(St + 8 * (size_t)c) : make_uint2(0, 0);
    }
    if ((terms += 32 * U) > PRD_EXACT_K) {
      as_flush(sum, lo, hi);
      terms = 32 * U;
    }
#pragma unroll
    for (int u = 0; u < U; u++) {
      uint32_t b[4];
      f16_of_s8(s[u].x, b[0], b[1]);
      f16_of_s8(s[u].y, b[2], b[3]);
      const uint32_t p[4] = {x[u][0].x, x[u][0].y, x[u][0].z, x[u][0].w};
      const uint32_t q[4] = {x[u][1].x, x[u][1].y, x[u][1].z, x[u][1].w};
      as_mma_chunk(lo, hi, p, q, b);
    }
  }
  as_flush(sum, lo, hi);
#pragma unroll
  for (int j = 0; j < 4; j++) atomicAdd(&red[(g + 8 * (j >> 1)) * 8 + 2 * t + (j & 1)], sum[j]);
  __syncthreads();
  if (warp != 0) return;
  int v[4];
#pragma unroll
  for (int j = 0; j < 4; j++) v[j] = red[(g + 8 * (j >> 1)) * 8 + 2 * t + (j & 1)];
  as_store(a, e, i0, g, t, v);
}

// The chunk groups c0, c0 + cinc, ... of a row tile with A regenerated: the
// lane's blocks are rows g and g + 8, chunk c of the tile whose first row's
// first block has index b0.  The last round delivers the byte pairs as f16
// words.
LWE_DEV void as_gen_tile(const AesTab &tab, AesF &F, const uint32_t rk[32], const int8_t *St,
                         uint32_t nch, uint32_t b0, uint32_t c0, uint32_t cinc, uint32_t g,
                         uint32_t t, int sum[4]) {
  float lo[4] = {}, hi[4] = {};
  uint32_t terms = 0;
  for (uint32_t cg = c0; cg < nch; cg += cinc) {
    const uint32_t c = cg + t;
    const uint2 sw = c < nch ? ld_nc_u2(St + 8 * (size_t)c) : make_uint2(0, 0);
    uint32_t s[2][4];
#pragma unroll
    for (int h = 0; h < 2; h++) aes_f_start(F, tab, 0, b0 + (g + 8 * h) * nch + c, s[h]);
    aes_rounds_3_9<2>(tab, rk, s);
    if ((terms += 32) > PRD_EXACT_K) {
      as_flush(sum, lo, hi);
      terms = 32;
    }
    uint32_t b[4];
    f16_of_s8(sw.x, b[0], b[1]);
    f16_of_s8(sw.y, b[2], b[3]);
    const uint32_t *p = s[0], *q = s[1];
#pragma unroll
    for (int w = 0; w < 4; w += 2) {
      // word w: bytes 0, 2 are S of state words w, w + 2; bytes 1, 3 of w + 1, w + 3
      const uint32_t k = rk[28 + w], l = rk[29 + w];
      mma_f16_k16(lo, aes_last2<0, 2>(tab, p[w], p[w ^ 2], f16_lo(k)),
                  aes_last2<0, 2>(tab, q[w], q[w ^ 2], f16_lo(k)),
                  aes_last2<0, 2>(tab, p[w + 1], p[(w + 1) ^ 2], f16_lo(l)),
                  aes_last2<0, 2>(tab, q[w + 1], q[(w + 1) ^ 2], f16_lo(l)), b[w], b[w + 1]);
      mma_f16_k16(hi, aes_last2<1, 3>(tab, p[w + 1], p[(w + 3) & 3], f16_hi(k)),
                  aes_last2<1, 3>(tab, q[w + 1], q[(w + 3) & 3], f16_hi(k)),
                  aes_last2<1, 3>(tab, p[(w + 2) & 3], p[w], f16_hi(l)),
                  aes_last2<1, 3>(tab, q[(w + 2) & 3], q[w], f16_hi(l)), b[w], b[w + 1]);
    }
  }
  as_flush(sum, lo, hi);
}

LWE_DEV void prd_load_rk(const uint32_t *rks, uint32_t rk[32]) {
#pragma unroll
  for (int i = 0; i < 32; i++) rk[i] = rks[12 + i];
}

// Regenerated A, many row tiles: a warp takes whole 16-row tiles, so no sums
// are shared.  CTA b of the grid takes an equal, contiguous range of the
// count x tiles units; it holds the tables of up to AS_SLOTS keys of its
// range at a time, so its warps need not meet where the range passes from
// one item to the next.  250 keys of n = 976 (476 MB of keystream): 699 us
// with a CTA per item (1.6 waves) and dp2a, about 460 us now.
__global__ void __launch_bounds__(512, 1) k_mul_as_gen(MulAsArgs a, uint32_t count) {
  extern __shared__ uint32_t sT[];
  pdl_trigger();
  aes_fill_smem(sT, g_aes_img);
  __syncthreads();
  pdl_wait();
  uint4 *sF = reinterpret_cast<uint4 *>(reinterpret_cast<uint8_t *>(sT) + PRD_F_OFF);
  uint32_t *srk = reinterpret_cast<uint32_t *>(reinterpret_cast<uint8_t *>(sT) + PRD_RK_OFF(AS_SLOTS));
  const AesTab tab = aes_tab(sT);
  const uint32_t tid = threadIdx.x, warp = prd_warp(), lane = tid & 31, g = lane >> 2, t = lane & 3;
  const uint32_t n = a.n, nch = n / 8, tiles = (a.rows ? a.rows : n) / 16;
  const uint64_t units = (uint64_t)count * tiles;
  const uint64_t u0 = units * blockIdx.x / gridDim.x, u1 = units * (blockIdx.x + 1) / gridDim.x;
  for (uint64_t eb = u0 / tiles; eb * tiles < u1; eb += AS_SLOTS) {
    const uint32_t ne = (uint32_t)min((uint64_t)AS_SLOTS, (u1 + tiles - 1) / tiles - eb);
    __syncthreads();
    if (warp < ne)
      prd_expand_key(tab, a.seeds + (eb + warp) * a.seed_stride, srk + 44 * warp);
    __syncthreads();
    for (uint32_t k = 0; k < ne; k++) aes_f_fill(sF + AES_F_ENTRIES * k, tab, srk + 44 * k, 0, tid, 512);
    __syncthreads();
    const uint64_t last = min(u1, (eb + ne) * tiles);
    for (uint64_t u = max(u0, eb * tiles) + warp; u < last; u += 16) {
      const uint32_t e = (uint32_t)(u / tiles), rt = (uint32_t)(u % tiles), k = e - (uint32_t)eb;
      uint32_t rk[32];
      prd_load_rk(srk + 44 * k, rk);
      AesF F = aes_f_open(sF + AES_F_ENTRIES * k, srk + 44 * k);
      int sum[4] = {};
      as_gen_tile(tab, F, rk, a.St + (size_t)e * a.st_stride + (size_t)g * n, nch,
                  (a.row0 + 16 * rt) * nch, 0, 4, g, t, sum);
      as_store(a, e, 16 * rt, g, t, sum);
    }
  }
}

// Regenerated A, few row tiles: a cluster of R CTAs takes a 16-row tile, its
// 16 R warps split the columns, and the sums meet in shared memory (with R >
// 1 in the cluster's first CTA).  Clusters walk the tiles.
__global__ void __launch_bounds__(512, 1) k_mul_as_gen_split(MulAsArgs a) {
  extern __shared__ uint32_t sT[];
  __shared__ int red[2][128];
  pdl_trigger();
  const uint32_t R = gridDim.x, rank = blockIdx.x, e = blockIdx.z, tid = threadIdx.x;
  if (tid < 128) red[0][tid] = red[1][tid] = 0;
  aes_fill_smem(sT, g_aes_img);
  __syncthreads();
  pdl_wait();
  uint4 *sF = reinterpret_cast<uint4 *>(reinterpret_cast<uint8_t *>(sT) + PRD_F_OFF);
  uint32_t *srk = reinterpret_cast<uint32_t *>(reinterpret_cast<uint8_t *>(sT) + PRD_RK_OFF(1));
  const AesTab tab = aes_tab(sT);
  const uint32_t warp = prd_warp(), lane = tid & 31, g = lane >> 2, t = lane & 3;
  const uint32_t n = a.n, nch = n / 8, tiles = (a.rows ? a.rows : n) / 16;
  if (warp == 0) prd_expand_key(tab, a.seeds + (size_t)e * a.seed_stride, srk);
  __syncthreads();
  aes_f_fill(sF, tab, srk, 0, tid, 512);
  __syncthreads();
  uint32_t rk[32];
  prd_load_rk(srk, rk);
  AesF F = aes_f_open(sF, srk);
  const int8_t *St = a.St + (size_t)e * a.st_stride + (size_t)g * n;
  uint32_t buf = 0;
  for (uint32_t rt = blockIdx.y; rt < tiles; rt += gridDim.y, buf ^= 1) {
    int sum[4] = {};
    as_gen_tile(tab, F, rk, St, nch, (a.row0 + 16 * rt) * nch, 4 * (rank * 16 + warp), 64 * R, g, t,
                sum);
#pragma unroll
    for (int j = 0; j < 4; j++)
      atomicAdd(&red[buf][(g + 8 * (j >> 1)) * 8 + 2 * t + (j & 1)], sum[j]);
    __syncthreads();
    if (R > 1) cluster_barrier();  // every CTA's sums are there
    if (warp == 0 && rank == 0) {
      int v[4];
#pragma unroll
      for (int j = 0; j < 4; j++) {
        const uint32_t at = (g + 8 * (j >> 1)) * 8 + 2 * t + (j & 1);
        v[j] = red[buf][at];
        for (uint32_t r = 1; r < R; r++) v[j] += ld_cluster_s32(cluster_map(&red[buf][at], r));
      }
      as_store(a, e, 16 * rt, g, t, v);
    }
    // read: the buffer is cleared for the next tile but one (the next tile's
    // barrier lies between), and no CTA leaves while others read its sums
    if (R > 1) cluster_barrier();
    else __syncthreads();
    if (tid < 128) red[buf][tid] = 0;
  }
}

// ---------------------------------------------------------------------------
// S' A + E'.  M = columns of A, K = rows: lane (g, t) supplies chunk g (8
// columns) of rows 4 t .. 4 t + 3 of a 16-row step, four 16-byte loads or AES
// blocks.  For each word of the chunk (two columns, M rows g and g + 8) the
// bytes of two rows pair up in an f16 word, which is what m16n8k16 takes; S'
// enters as the 4 bytes of row g at the step's rows 4 t ...  A warp so covers
// 64 columns with 32 accumulators per lane.
//
// A CTA takes cgs groups of 64 columns (its warps split the rows of each) and
// one of R equal row ranges; R CTAs form a cluster whose partial sums are
// added through distributed shared memory, so no global workspace is needed.
// Where the call wants V = S' B + E'' too (Alg. 2), one more CTA column takes
// B, an n x 8 matrix, as a ninth-chunk-wide A and finishes C = V + Enc(mu):
// a launch of its own (one CTA per item walking n rows) took 175 us at n =
// 32768 and 9 us at n = 1344.
// ---------------------------------------------------------------------------
#define SA_RED_K 68    // row k of a 64-column group's sums: 64, and 4 so that a
#define SA_RED_CG 544  // warp's atomics fall in 32 banks; 8 rows per group

// One word column (two columns of the chunk) of four rows
LWE_DEV void sa_mma_word(float acc[2][4], uint32_t w0, uint32_t w1, uint32_t w2, uint32_t w3,
                         uint32_t b0, uint32_t b1) {
  const uint32_t p = __byte_perm(w0, w1, 0x5410), q = __byte_perm(w0, w1, 0x7632);
  const uint32_t r = __byte_perm(w2, w3, 0x5410), s = __byte_perm(w2, w3, 0x7632);
  mma_f16_k16(acc[0], f16_lo(p), f16_lo(q), f16_lo(r), f16_lo(s), b0, b1);
  mma_f16_k16(acc[1], f16_hi(p), f16_hi(q), f16_hi(r), f16_hi(s), b0, b1);
}

// the lane's sums into the CTA's: red[k][c][g] = row k, column 8 g + c; cleared
LWE_DEV void sa_reduce(int *red, uint32_t g, uint32_t t, float acc[4][2][4]) {
#pragma unroll
  for (int w = 0; w < 4; w++)
#pragma unroll
    for (int j = 0; j < 4; j++) {
      atomicAdd(&red[(2 * t + (j & 1)) * SA_RED_K + (2 * w + (j >> 1)) * 8 + g],
                limb_sum(acc[w][0][j], acc[w][1][j]));
      acc[w][0][j] = acc[w][1][j] = 0.f;
    }
}

// row steps st, st + inc, ... below se of a stored matrix (row i at A + i ld,
// this lane's chunk already added), two steps (eight loads) in flight; the
// sums go to red
LWE_DEV void sa_rows_stored(const uint16_t *A, size_t ld, bool valid, const int8_t *S, uint32_t st,
                            uint32_t se, uint32_t inc, uint32_t g, uint32_t t, int *red) {
  float acc[4][2][4] = {};
  uint32_t terms = 0;
  for (; st < se; st += 2 * inc) {
    uint4 x[2][4];
    uint32_t sw[2];
#pragma unroll
    for (int u = 0; u < 2; u++) {
      const uint32_t s = st + u * inc;
      const bool in = s < se;
#pragma unroll
      for (int q = 0; q < 4; q++)
        x[u][q] = in && valid ? ld_stream_u4(A + (size_t)(16 * s + 4 * t + q) * ld)
                              : make_uint4(0, 0, 0, 0);
      sw[u] = in ? ld_nc_u1(S + 16 * (size_t)s + 4 * t) : 0u;
    }
    if ((terms += 32) > PRD_EXACT_K) {
      sa_reduce(red, g, t, acc);
      terms = 32;
    }
#pragma unroll
    for (int u = 0; u < 2; u++) {
      uint32_t b0, b1;
      f16_of_s8(sw[u], b0, b1);
      sa_mma_word(acc[0], x[u][0].x, x[u][1].x, x[u][2].x, x[u][3].x, b0, b1);
      sa_mma_word(acc[1], x[u][0].y, x[u][1].y, x[u][2].y, x[u][3].y, b0, b1);
      sa_mma_word(acc[2], x[u][0].z, x[u][1].z, x[u][2].z, x[u][3].z, b0, b1);
      sa_mma_word(acc[3], x[u][0].w, x[u][1].w, x[u][2].w, x[u][3].w, b0, b1);
    }
  }
  sa_reduce(red, g, t, acc);
}

LWE_DEV uint32_t sa_total(int *red, uint32_t idx, uint32_t R) {
  if (R == 1) return (uint32_t)red[idx];
  uint32_t sum = 0;
  for (uint32_t r = 0; r < R; r++) sum += (uint32_t)ld_cluster_s32(cluster_map(red + idx, r));
  return sum;
}

// The cluster's sums are finished: + E' mod q (+ E'' + Enc(mu) for the V
// columns), stored or (CMP) compared with the received ciphertext.
template <bool CMP>
LWE_DEV void sa_epilogue(const MulSaArgs &a, int *red, bool vcols, uint32_t cgs, uint32_t rsplit,
                         uint32_t R, uint32_t e, uint32_t tid, uint32_t nt) {
  const uint32_t n = a.n, mq = (1u << a.logq) - 1u;
  uint32_t diff = 0;
  if (vcols) {
    for (uint32_t v = rsplit * nt + tid; v < 64; v += R * nt) {
      const uint32_t k = v >> 3, l = v & 7;
      uint32_t sum = sa_total(red, k * SA_RED_K + l * 8, R);
      const uint8_t *mu = a.mu + (size_t)e * 32 + k * a.B;
      uint32_t bits = 0;
      for (uint32_t b = 0; b < a.B; b++) bits |= (uint32_t)mu[b] << (8 * b);
      const uint32_t sym = (bits >> (l * a.B)) & ((1u << a.B) - 1u);
      sum += (uint32_t)(int)a.Epp[(size_t)e * a.epp_stride + v] + (sym << (a.logq - a.B));
      const uint32_t val = sum & mq;
      uint16_t *o = reinterpret_cast<uint16_t *>(a.out + (size_t)e * a.out_stride + 16 * (size_t)n) + v;
      if (CMP)
        diff |= val ^ (uint32_t)*o;
      else
        *o = (uint16_t)val;
    }
  } else {
    const uint32_t W = 64 * cgs, cells = 8 * W, share = (cells + R - 1) / R;
    const uint32_t end = min(cells, (rsplit + 1) * share);
    for (uint32_t v = rsplit * share + tid; v < end; v += nt) {
      const uint32_t k = v / W, col = v - k * W, j = blockIdx.x * W + col;
      if (j >= n) continue;
      uint32_t sum = sa_total(red, (col >> 6) * SA_RED_CG + k * SA_RED_K + (col & 7) * 8 + ((col >> 3) & 7), R);
      if (a.E) sum += (uint32_t)(int)a.E[(size_t)e * a.e_stride + (size_t)k * n + j];
      const uint32_t val = sum & mq;
      uint16_t *o = reinterpret_cast<uint16_t *>(a.out + (size_t)e * a.out_stride) + (size_t)k * n + j;
      if (CMP)
        diff |= val ^ (uint32_t)*o;
      else
        *o = (uint16_t)val;
    }
  }
  if (CMP) {
    diff = __reduce_or_sync(0xffffffffu, diff);
    if ((tid & 31) == 0 && diff) atomicOr(a.flags + e, 1u);
  }
}

// B of the item's public key, n x 8 entries
LWE_DEV const uint16_t *sa_pk_B(const MulSaArgs &a, uint32_t e) {
  const uint8_t *pk = a.key_ptrs ? a.key_ptrs[e] + a.key_off : a.pk;
  return reinterpret_cast<const uint16_t *>(pk + 16);
}

template <bool CMP>
__global__ void __launch_bounds__(256) k_sa(MulSaArgs a, uint32_t cgs) {
  __shared__ int red[4 * SA_RED_CG];
  pdl_trigger();
  const uint32_t tid = threadIdx.x, warp = prd_warp(), lane = tid & 31, g = lane >> 2, t = lane & 3;
  for (uint32_t i = tid; i < cgs * SA_RED_CG; i += 256) red[i] = 0;
  __syncthreads();
  pdl_wait();
  const uint32_t rsplit = blockIdx.y, R = gridDim.y, e = blockIdx.z, n = a.n;
  const bool vcols = a.vcols && blockIdx.x == gridDim.x - 1;
  const uint32_t s0 = a.row0 / 16, s1 = (a.row1 ? a.row1 : n) / 16;  // 16-row steps
  const uint32_t sb = s0 + (s1 - s0) * rsplit / R, se = s0 + (s1 - s0) * (rsplit + 1) / R;
  const int8_t *S = a.S + (size_t)e * a.s_stride + (size_t)g * n;
  if (vcols) {
    sa_rows_stored(sa_pk_B(a, e), 8, g == 0, S, sb + warp, se, 8, g, t, red);
  } else {
    const uint32_t wc = warp & (cgs - 1), rows_w = 8 / cgs, chunk = (blockIdx.x * cgs + wc) * 8 + g;
    const uint16_t *A = a.A_ptrs ? a.A_ptrs[e] : a.A;
    // a stored row block starts at row row0; chunks beyond n are never read
    const bool valid = 8 * chunk < n && LWE_BOUNDS(16 * se <= (a.row1 ? a.row1 : n), 110);
    A -= (size_t)a.row0 * n;
    sa_rows_stored(A + (valid ? 8 * (size_t)chunk : 0), n, valid, S, sb + warp / cgs, se, rows_w, g,
                   t, red + wc * SA_RED_CG);
  }
  __syncthreads();
  if (R > 1) cluster_barrier();  // every CTA of the cluster has its partial sum
  sa_epilogue<CMP>(a, red, vcols, cgs, rsplit, R, e, tid, 256);
  if (R > 1) cluster_barrier();  // no CTA leaves while others read its shared memory
}

// The same with A regenerated: 16 warps on one 64-column group, four AES
// blocks side by side per lane and step, whose last round delivers the byte
// pairs.  Bound by the shared-memory pipe: 128 table lookups a block, and 8
// wavefronts for rounds 1 and 2.  (A lane pair that swapped halves of two
// blocks, dp2a, and 160 lookups a block took 101.9 us at n = 4096 and 2.94 ms
// at 32768; this takes 45.1 us, on 128 of 152 SMs, and 2.1 ms, 1.02 TB/s of
// keystream.)
template <bool CMP>
__global__ void __launch_bounds__(512, 1) k_sa_gen(MulSaArgs a) {
  extern __shared__ uint32_t sT[];
  __shared__ int red[SA_RED_CG];
  pdl_trigger();
  const uint32_t tid = threadIdx.x, warp = prd_warp(), lane = tid & 31, g = lane >> 2, t = lane & 3;
  const uint32_t rsplit = blockIdx.y, R = gridDim.y, e = blockIdx.z, n = a.n, nch = n / 8;
  const bool vcols = a.vcols && blockIdx.x == gridDim.x - 1;
  for (uint32_t i = tid; i < SA_RED_CG; i += 512) red[i] = 0;
  if (!vcols) aes_fill_smem(sT, g_aes_img);
  __syncthreads();
  pdl_wait();
  const uint32_t s0 = a.row0 / 16, s1 = (a.row1 ? a.row1 : n) / 16;  // 16-row steps
  const uint32_t sb = s0 + (s1 - s0) * rsplit / R, se = s0 + (s1 - s0) * (rsplit + 1) / R;
  const int8_t *S = a.S + (size_t)e * a.s_stride + (size_t)g * n;
  if (vcols) {
    sa_rows_stored(sa_pk_B(a, e), 8, g == 0, S, sb + warp, se, 16, g, t, red);
  } else {
    uint4 *sF = reinterpret_cast<uint4 *>(reinterpret_cast<uint8_t *>(sT) + PRD_F_OFF);
    uint32_t *srk = reinterpret_cast<uint32_t *>(reinterpret_cast<uint8_t *>(sT) + PRD_RK_OFF(1));
    const AesTab tab = aes_tab(sT);
    if (warp == 0)
      prd_expand_key(tab, a.key_ptrs ? a.key_ptrs[e] + a.key_off : a.seedA, srk);
    __syncthreads();
    aes_f_fill(sF, tab, srk, 0, tid, 512);
    __syncthreads();
    uint32_t rk[32];
    prd_load_rk(srk, rk);
    AesF F = aes_f_open(sF, srk);
    const uint32_t chunk = blockIdx.x * 8 + g;
    float acc[4][2][4] = {};
    uint32_t terms = 0;
    for (uint32_t st = sb + warp; st < se; st += 16) {
      const uint32_t i = 16 * st + 4 * t;  // this lane's rows i .. i + 3
      const uint32_t sw = ld_nc_u1(S + i);
      uint32_t s[4][4];
#pragma unroll
      for (int q = 0; q < 4; q++) aes_f_start(F, tab, 0, (i + q) * nch + chunk, s[q]);
      aes_rounds_3_9<4>(tab, rk, s);
      if ((terms += 16) > PRD_EXACT_K) {
        sa_reduce(red, g, t, acc);
        terms = 16;
      }
      uint32_t b0, b1;
      f16_of_s8(sw, b0, b1);
#pragma unroll
      for (int w = 0; w < 4; w++) {
        const uint32_t k = rk[28 + w];
        const int w1 = (w + 1) & 3, w2 = (w + 2) & 3, w3 = (w + 3) & 3;
        const uint32_t k0 = __byte_perm(k, 0, 0x4040), k1 = __byte_perm(k, 0, 0x4141);
        const uint32_t k2 = __byte_perm(k, 0, 0x4242), k3 = __byte_perm(k, 0, 0x4343);
        mma_f16_k16(acc[w][0], aes_last2<0, 0>(tab, s[0][w], s[1][w], k0),
                    aes_last2<2, 2>(tab, s[0][w2], s[1][w2], k2),
                    aes_last2<0, 0>(tab, s[2][w], s[3][w], k0),
                    aes_last2<2, 2>(tab, s[2][w2], s[3][w2], k2), b0, b1);
        mma_f16_k16(acc[w][1], aes_last2<1, 1>(tab, s[0][w1], s[1][w1], k1),
                    aes_last2<3, 3>(tab, s[0][w3], s[1][w3], k3),
                    aes_last2<1, 1>(tab, s[2][w1], s[3][w1], k1),
                    aes_last2<3, 3>(tab, s[2][w3], s[3][w3], k3), b0, b1);
      }
    }
    sa_reduce(red, g, t, acc);
  }
  __syncthreads();
  if (R > 1) cluster_barrier();
  sa_epilogue<CMP>(a, red, vcols, 1, rsplit, R, e, tid, 512);
  if (R > 1) cluster_barrier();
}
