// Row-wise pair-biased attention on tcgen05 for samples whose whole key range fits one accumulator
// (N <= 224, pair order, head dim 16 or 32).
//
// Work item: one attention row (s, i), one head h, one block of 128 queries j.  The raw scores of the
// item, Q K^T (M = 128 queries, N = round_up(N_s, 16) keys, K = d), are one MMA group into a
// 224-column TMEM accumulator, so the softmax needs no running rescale:
//   pass 1  two threads per query read their halves of the row and take the maximum of the raw scores;
//           with the largest bias of the row (found once per (s, h) when the bias tile is loaded) it
//           bounds every biased score from above, which is all the reference value of a softmax needs
//           (the normalisation cancels it exactly);
//   pass 2  s = raw + bias (the bias tile of the (s, h, j block) is resident in shared memory, stored
//           times sqrt(d); key columns past N hold a large negative value so their weights are exact
//           zeros and no pass needs a mask), p = exp2((s - bound) log2(e) / sqrt(d)), summed in float
//           and written as packed bf16 pairs over half of each 16-key granule's own score columns,
//           from where the second MMA group takes P as its TMEM-resident A operand: O = P V (N = d)
//           into 32 columns of its own;
//   output  O / l, 16 channels per thread, stored row-major.
// The exponentials are the floor of this kernel (an SM retires 16 per clock); the bias addition rides
// in their shadow on the other pipes.
// Roles: warp 0 streams Q | K and warp 2 streams V of each item with TMA (32-row boxes, swizzle span =
// 2 d bytes) through two rings (a Q | K stage is free again as soon as the scores are computed), warp 1
// issues the MMAs (converged, one elected lane; the scores of item n + 1 before P V of item n), warps
// 3-10 and 11-18 are two softmax groups that own one TMEM buffer each and take alternate items.  Each
// CTA walks a contiguous range of the items ordered (s, h, i, j block), so the two query blocks of a
// row are neighbours (their K / V come from L2 the second time) and the bias tiles are reloaded only
// when (s, h) changes.
#include <cstring>

#include "fast.cuh"
#include "tc_common.cuh"

namespace ntp {

constexpr int TCA_THREADS = 96 + 512;
constexpr int TCA_NMAX = 224;      // keys per item: 224 score columns + 32 output columns = one 256-column TMEM buffer
constexpr int TCA_O_COL = 224;     // output accumulator (up to 32 columns)
constexpr float TCA_LOG2E = 1.4426950408889634f;

struct AttnTcParams {
  CUtensorMap qmap;       // flat {H d, rows}, box {d, 128}
  CUtensorMap kmap, vmap; // box {d, 32}
  // column mode (queries and keys run along the first pair index of a column): one map per sample,
  // {H d, first index (stride N H d), column (stride H d), which of q / k / v}, box {d, 32, 1, 1}
  CUtensorMap cmap[MAXB];
  BatchMeta m;
  long long item_off[MAXB + 1];   // prefix of N_s * H * ceil(N_s / 128) over the samples this kernel takes
  const __nv_bfloat16* bias;      // head-major channel-major, stored times sqrt(d); nullable
  __nv_bfloat16* o;
  long long row0;                 // first packed row the maps cover
  int H, nqk, nv, kv_rows;        // stages of the Q|K ring and of the V ring; rows reserved for K (and V) per stage
  int bias_tile_bytes;            // bytes reserved per resident bias tile
  int n_max;                      // samples with N > n_max are left to the other kernel
  int* status;
};

__host__ __device__ inline int tca_bias_stride(int nk) {   // bytes per resident bias row: an odd multiple of 16
  const int b = nk * 2;
  return (b / 16) % 2 == 0 ? b + 16 : b;
}

__device__ inline void tca_cp_async16(void* smem, const void* gmem, bool valid) {
  const unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
  const int sz = valid ? 16 : 0;
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(sa), "l"(gmem), "r"(sz));
}

// 16, 32 or 64 consecutive columns of this thread's row, landed: load and wait are one statement, so the compiler can neither use
// nor copy the registers in between, and ties no registers afterwards.
__device__ inline void tca_ld(unsigned t, unsigned (&a)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];\n\t"
      "tcgen05.wait::ld.sync.aligned;\n"
      : "=r"(a[0]), "=r"(a[1]), "=r"(a[2]), "=r"(a[3]), "=r"(a[4]), "=r"(a[5]), "=r"(a[6]), "=r"(a[7]), "=r"(a[8]), "=r"(a[9]), "=r"(a[10]), "=r"(a[11]), "=r"(a[12]), "=r"(a[13]), "=r"(a[14]), "=r"(a[15]) : "r"(t) : "memory");
}
__device__ inline void tca_ld(unsigned t, unsigned (&a)[16], unsigned (&b)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%32];\n\t"
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%33];\n\t"
      "tcgen05.wait::ld.sync.aligned;\n"
      : "=r"(a[0]), "=r"(a[1]), "=r"(a[2]), "=r"(a[3]), "=r"(a[4]), "=r"(a[5]), "=r"(a[6]), "=r"(a[7]), "=r"(a[8]), "=r"(a[9]), "=r"(a[10]), "=r"(a[11]), "=r"(a[12]), "=r"(a[13]), "=r"(a[14]), "=r"(a[15]),
        "=r"(b[0]), "=r"(b[1]), "=r"(b[2]), "=r"(b[3]), "=r"(b[4]), "=r"(b[5]), "=r"(b[6]), "=r"(b[7]), "=r"(b[8]), "=r"(b[9]), "=r"(b[10]), "=r"(b[11]), "=r"(b[12]), "=r"(b[13]), "=r"(b[14]), "=r"(b[15]) : "r"(t), "r"(t + 16) : "memory");
}
__device__ inline void tca_ld(unsigned t, unsigned (&a)[16], unsigned (&b)[16], unsigned (&c)[16], unsigned (&d)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%64];\n\t"
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%65];\n\t"
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%32,%33,%34,%35,%36,%37,%38,%39,%40,%41,%42,%43,%44,%45,%46,%47}, [%66];\n\t"
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%48,%49,%50,%51,%52,%53,%54,%55,%56,%57,%58,%59,%60,%61,%62,%63}, [%67];\n\t"
      "tcgen05.wait::ld.sync.aligned;\n"
      : "=r"(a[0]), "=r"(a[1]), "=r"(a[2]), "=r"(a[3]), "=r"(a[4]), "=r"(a[5]), "=r"(a[6]), "=r"(a[7]), "=r"(a[8]), "=r"(a[9]), "=r"(a[10]), "=r"(a[11]), "=r"(a[12]), "=r"(a[13]), "=r"(a[14]), "=r"(a[15]),
        "=r"(b[0]), "=r"(b[1]), "=r"(b[2]), "=r"(b[3]), "=r"(b[4]), "=r"(b[5]), "=r"(b[6]), "=r"(b[7]), "=r"(b[8]), "=r"(b[9]), "=r"(b[10]), "=r"(b[11]), "=r"(b[12]), "=r"(b[13]), "=r"(b[14]), "=r"(b[15]),
        "=r"(c[0]), "=r"(c[1]), "=r"(c[2]), "=r"(c[3]), "=r"(c[4]), "=r"(c[5]), "=r"(c[6]), "=r"(c[7]), "=r"(c[8]), "=r"(c[9]), "=r"(c[10]), "=r"(c[11]), "=r"(c[12]), "=r"(c[13]), "=r"(c[14]), "=r"(c[15]),
        "=r"(d[0]), "=r"(d[1]), "=r"(d[2]), "=r"(d[3]), "=r"(d[4]), "=r"(d[5]), "=r"(d[6]), "=r"(d[7]), "=r"(d[8]), "=r"(d[9]), "=r"(d[10]), "=r"(d[11]), "=r"(d[12]), "=r"(d[13]), "=r"(d[14]), "=r"(d[15])
      : "r"(t), "r"(t + 16), "r"(t + 32), "r"(t + 48) : "memory");
}

__device__ inline float tca_exp2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;\n" : "=f"(y) : "f"(x));
  return y;
}
__device__ inline float tca_max3(float a, float b, float c) {      // one instruction on sm_100
  float y;
  asm("max.f32 %0, %1, %2, %3;\n" : "=f"(y) : "f"(a), "f"(b), "f"(c));
  return y;
}
__device__ inline unsigned tca_pack(float lo, float hi) {
  unsigned y;
  asm("cvt.rn.bf16x2.f32 %0, %1, %2;\n" : "=r"(y) : "f"(hi), "f"(lo));
  return y;
}

// swizzled K-major / MN-major operand descriptor for a tile whose rows are `span` = 32, 64 or 128 bytes.  The start
// address sits in the low 14 bits in units of 16 bytes, so moving the operand by x bytes is adding x / 16.
__device__ inline unsigned long long tca_desc(unsigned saddr, int span) {
  unsigned long long d = 0;
  d |= (unsigned long long)((saddr & 0x3FFFFu) >> 4);
  d |= (unsigned long long)(((unsigned)(8 * span) >> 4) & 0x3FFF) << 16;   // leading byte offset (one block: unused)
  d |= (unsigned long long)(((unsigned)(8 * span) >> 4) & 0x3FFF) << 32;   // 8 rows further
  d |= (unsigned long long)1 << 46;
  d |= (unsigned long long)(span == 128 ? 2 : span == 64 ? 4 : 6) << 61;
  return d;
}

template <int D, bool COL>
__global__ void __launch_bounds__(TCA_THREADS, 1) attn_tc_kernel(const __grid_constant__ AttnTcParams p) {
  constexpr int SPAN = 2 * D;                 // bytes per tile row = swizzle span
  constexpr int Q_BYTES = 128 * SPAN;
  extern __shared__ unsigned char smem_raw[];
  __shared__ __align__(8) unsigned long long bars[12 + 8];
  __shared__ unsigned tmem_base_s;
  __shared__ int abort_flag;
  unsigned char* smem = smem_raw + ((1024 - (smem_u32(smem_raw) & 1023)) & 1023);
  const int kv_bytes = p.kv_rows * SPAN;
  const int qk_bytes = Q_BYTES + kv_bytes;
  unsigned char* sQK = smem;                                      // [nqk][Q | K]
  unsigned char* sV = sQK + p.nqk * qk_bytes;                     // [nv][V]
  float* xch = reinterpret_cast<float*>(sV + p.nv * kv_bytes);    // [2 groups][2 parities][max | sum][2 halves][128]
  unsigned char* sBias = reinterpret_cast<unsigned char*>(xch) + 2 * 2 * 2 * 2 * 128 * 4;   // [2 tiles][128 queries][stride]
  unsigned long long* qkfull = bars;          // [3]
  unsigned long long* qkempty = bars + 3;     // [3] the score MMAs that read the stage are done
  unsigned long long* vfull = bars + 6;       // [3]
  unsigned long long* vempty = bars + 9;      // [3] the P V MMAs that read the stage are done
  unsigned long long* sfull = bars + 12;      // [2] scores of the group's item are in TMEM
  unsigned long long* sempty = bars + 14;     // [2] P V has consumed the weights: the score columns are free
  unsigned long long* pfull = bars + 16;      // [2] P written
  unsigned long long* ofull = bars + 18;      // [2] P V complete

  const BatchMeta& m = p.m;
  const int H = p.H, Hd = H * D;
  const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;   // warp-uniform for the compiler too
  if (threadIdx.x == 0) {
    abort_flag = 0;
    for (int s = 0; s < 12; ++s) mbar_init(&bars[s], 1);
    for (int b = 0; b < 2; ++b) {
      mbar_init(&sfull[b], 1);
      mbar_init(&sempty[b], 1);
      mbar_init(&pfull[b], 8);
      mbar_init(&ofull[b], 1);
    }
    mbar_fence_init();
  }
  if (warp == 1) tmem_alloc(&tmem_base_s, 512);
  fence_proxy_async_smem();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  pdl_begin();
  const unsigned tmem_base = __shfl_sync(0xffffffffu, tmem_base_s, 0);
  AbortCtx ab{p.status, &abort_flag};
  const float sc2 = rsqrtf((float)D) * TCA_LOG2E;
  const bool has_bias = p.bias != nullptr;

  const long long total = p.item_off[m.B];
  long long r = total * blockIdx.x / gridDim.x;
  const long long r_end = total * (blockIdx.x + 1) / gridDim.x;
  unsigned it0 = 0;                           // items this CTA has finished (drives every ring position / parity)

  while (r < r_end) {
    // ------------------------------------------------------------ segment: items of one (s, h)
    int s = 0;
    while (s + 1 < m.B && r >= p.item_off[s + 1]) ++s;
    const int N = m.N[s], ld = round_up8(N), Nk = (N + 15) & ~15;
    const int njb = (N + 127) / 128;
    const unsigned rem0 = (unsigned)(r - p.item_off[s]);           // ((h N + i) njb + jb)
    const int h = (int)(rem0 / (unsigned)(N * njb));
    const unsigned in_head0 = rem0 - (unsigned)h * (unsigned)(N * njb);   // i njb + jb of the first item
    const long long left = (long long)N * njb - in_head0;
    const int cnt = (int)(left < r_end - r ? left : r_end - r);
    const __nv_bfloat16* bias_h = has_bias ? p.bias + (long long)H * m.cm_off[s] + (long long)h * N * ld : nullptr;
    const long long row_base = m.pair_off[s] - p.row0;            // packed row of (i = 0, j = 0) relative to the maps
    const int nb = (N + 31) / 32;                                  // 32-row boxes of K (and V)
    const int ng = Nk / 16;                                        // 16-key granules

    const int bstride = tca_bias_stride(Nk);
    float bmax[2] = {0.f, 0.f};                                    // largest bias of this thread's query row, per j block
    if (warp >= 3) {
      // bias tile of query block t: row-major, query q at t * tile + (q % 128) * stride.  Key columns N .. Nk - 1
      // (rows of K that belong to other pair rows) get a large negative bias, so their weights come out as exact
      // zeros and neither softmax pass needs a mask.
      const int chunks = Nk / 8;
      if (COL) {
        // the bias of (query q, key k) is element [k][q] of the plane: read 8 consecutive queries of a key row,
        // scatter them into the 8 query rows of the tile
        const int qchunks = ld / 8;
        for (int idx = threadIdx.x - 96; idx < N * qchunks; idx += 512) {
          const int k = idx / qchunks, c = idx - k * qchunks;
          uint4 val = make_uint4(0, 0, 0, 0);
          if (has_bias) val = *reinterpret_cast<const uint4*>(bias_h + (long long)k * ld + c * 8);
          const unsigned w4[4] = {val.x, val.y, val.z, val.w};
#pragma unroll
          for (int e = 0; e < 8; ++e) {
            const int q = c * 8 + e;
            if (q < njb * 128)
              *reinterpret_cast<unsigned short*>(sBias + (q >> 7) * p.bias_tile_bytes + (q & 127) * bstride + k * 2) =
                  (unsigned short)(e & 1 ? w4[e >> 1] >> 16 : w4[e >> 1] & 0xffffu);
          }
        }
      } else {
        for (int idx = threadIdx.x - 96; idx < njb * 128 * chunks; idx += 512) {
          const int q = idx / chunks, c = idx - q * chunks;
          const bool ok = has_bias && q < N && c * 8 < ld;
          tca_cp_async16(sBias + (q >> 7) * p.bias_tile_bytes + (q & 127) * bstride + c * 16,
                         ok ? bias_h + (long long)q * ld + c * 8 : p.o, ok);
        }
      }
      asm volatile("cp.async.wait_all;\n" ::: "memory");
      named_bar_sync(3, 512);
      const int tail = Nk - N;                                     // 0 .. 15 masked key columns
      for (int idx = threadIdx.x - 96; idx < njb * 128 * tail; idx += 512) {
        const int q = idx / tail, k = N + idx - q * tail;
        *reinterpret_cast<unsigned short*>(sBias + (q >> 7) * p.bias_tile_bytes + (q & 127) * bstride + k * 2) = 0xC6EAu;   // bf16 -29952
      }
      named_bar_sync(3, 512);
      const int qrow = (warp & 3) * 32 + lane;
      for (int t = 0; t < njb; ++t) {
        const unsigned char* br = sBias + t * p.bias_tile_bytes + qrow * bstride;
        float mb = -INFINITY;
        for (int c = 0; c < chunks; ++c) {
          const uint4 v = *reinterpret_cast<const uint4*>(br + c * 16);
          const unsigned w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
          for (int e = 0; e < 4; ++e) mb = fmaxf(mb, fmaxf(__uint_as_float(w[e] << 16), __uint_as_float(w[e] & 0xffff0000u)));
        }
        bmax[t] = mb;
      }
    }
    __syncthreads();

    if (warp == 0) {
      // -------------------------------------------------------------- Q | K producer
      unsigned st = it0 % (unsigned)p.nqk, k = it0 / (unsigned)p.nqk;
      for (int n = 0; n < cnt; ++n) {
        const unsigned ih = in_head0 + n;
        const int i = (int)(ih / (unsigned)njb), jb = (int)(ih - (unsigned)i * njb);
        const int base = (int)(row_base + (long long)i * N);
        unsigned char* stg = sQK + st * qk_bytes;
        if (lane == 0) {
          mbar_wait(&qkempty[st], (k & 1) ^ 1, ab);
          mbar_expect_tx(&qkfull[st], Q_BYTES + nb * 32 * SPAN);
        }
        __syncwarp();
        if (COL) {     // i is the column; the query block and the keys run along the first pair index
          if (lane < 4) tma_load_4d(stg + lane * 32 * SPAN, &p.cmap[s], &qkfull[st], h * D, jb * 128 + lane * 32, i, 0);
          else if (lane < 4 + nb) tma_load_4d(stg + Q_BYTES + (lane - 4) * 32 * SPAN, &p.cmap[s], &qkfull[st], h * D, (lane - 4) * 32, i, 1);
        } else {
          if (lane == 0) tma_load_2d(stg, &p.qmap, &qkfull[st], h * D, base + jb * 128);
          else if (lane <= nb) tma_load_2d(stg + Q_BYTES + (lane - 1) * 32 * SPAN, &p.kmap, &qkfull[st], h * D, base + (lane - 1) * 32);
        }
        if (++st == (unsigned)p.nqk) { st = 0; ++k; }
      }
    } else if (warp == 2) {
      // -------------------------------------------------------------- V producer
      unsigned st = it0 % (unsigned)p.nv, k = it0 / (unsigned)p.nv;
      for (int n = 0; n < cnt; ++n) {
        const unsigned ih = in_head0 + n;
        const int i = (int)(ih / (unsigned)njb);
        const int base = (int)(row_base + (long long)i * N);
        if (lane == 0) {
          mbar_wait(&vempty[st], (k & 1) ^ 1, ab);
          mbar_expect_tx(&vfull[st], nb * 32 * SPAN);
        }
        __syncwarp();
        if (lane < nb) {
          if (COL) tma_load_4d(sV + st * kv_bytes + lane * 32 * SPAN, &p.cmap[s], &vfull[st], h * D, lane * 32, i, 2);
          else tma_load_2d(sV + st * kv_bytes + lane * 32 * SPAN, &p.vmap, &vfull[st], h * D, base + lane * 32);
        }
        if (++st == (unsigned)p.nv) { st = 0; ++k; }
      }
    } else if (warp == 1) {
      // -------------------------------------------------------------- MMA issuer (whole warp, one elected lane issues)
      const unsigned idesc_s = idesc_f16(128, Nk, 0, 0, FMT_BF16, FMT_BF16);
      const unsigned idesc_o = idesc_f16(128, D, 0, 1, FMT_BF16, FMT_BF16);      // B = V, MN-major
      unsigned sq = it0 % (unsigned)p.nqk, kq = it0 / (unsigned)p.nqk;           // ring position of the next score item
      unsigned sv = it0 % (unsigned)p.nv, kv = it0 / (unsigned)p.nv;             // ... of the next P V item
      for (int n = 0; n <= cnt; ++n) {
        if (n < cnt) {
          const unsigned it = it0 + n, b = it & 1, u = it >> 1;
          mbar_wait(&qkfull[sq], kq & 1, ab);
          mbar_wait(&sempty[b], (u & 1) ^ 1, ab);
          tc_fence_after();
          const unsigned q_addr = smem_u32(sQK + sq * qk_bytes);
          const unsigned long long qd = tca_desc(q_addr, SPAN), kd = tca_desc(q_addr + Q_BYTES, SPAN);
          if (elect_one()) {
#pragma unroll
            for (int ks = 0; ks < D / 16; ++ks) umma_bf16(tmem_base + b * 256, qd + ks * 2, kd + ks * 2, idesc_s, ks);
            tc_commit(&sfull[b]);
            tc_commit(&qkempty[sq]);
          }
          __syncwarp();
          if (++sq == (unsigned)p.nqk) { sq = 0; ++kq; }
        }
        if (n >= 1) {
          const unsigned it = it0 + n - 1, b = it & 1, u = it >> 1;
          mbar_wait(&vfull[sv], kv & 1, ab);
          mbar_wait(&pfull[b], u & 1, ab);
          tc_fence_after();
          const unsigned long long vd = tca_desc(smem_u32(sV + sv * kv_bytes), SPAN);
          const unsigned a_p = tmem_base + b * 256, d_o = a_p + TCA_O_COL;
#pragma unroll
          for (int kk = 0; kk < TCA_NMAX / 16; ++kk)
            if (kk < ng && elect_one())
              umma_ts(d_o, a_p + kk * 16 + (kk & 1) * 8, vd + kk * SPAN, idesc_o, kk);   // 16 rows of V further: 16 SPAN bytes
          if (elect_one()) {
            tc_commit(&ofull[b]);
            tc_commit(&sempty[b]);
            tc_commit(&vempty[sv]);
          }
          __syncwarp();
          if (++sv == (unsigned)p.nv) { sv = 0; ++kv; }
        }
      }
    } else {
      // -------------------------------------------------------------- softmax groups
      const int sw = warp - 3, wg = sw >> 3, hf = (sw >> 2) & 1, quarter = warp & 3;
      const int row = quarter * 32 + lane;                          // query inside the 128-block = TMEM lane
      const unsigned t_row = tmem_base + ((unsigned)(quarter * 32) << 16) + wg * 256;
      for (int n = (int)((wg ^ it0) & 1); n < cnt; n += 2) {
        const unsigned it = it0 + n, u = it >> 1;
        const unsigned ih = in_head0 + n;
        const int i = (int)(ih / (unsigned)njb), jb = (int)(ih - (unsigned)i * njb);
        const int j = jb * 128 + row;
        const bool warp_live = jb * 128 + quarter * 32 < N;        // this warp owns at least one real query
        float* xm = xch + (wg * 2 + (u & 1)) * 4 * 128;             // [max | sum][2 halves][128]
        unsigned ra[16], rb[16];
        mbar_wait(&sfull[wg], u & 1, ab);      // a failed probe parks the warp in hardware: every warp may watch the barrier
        tc_fence_after();
        // Each thread owns a contiguous half of the row: granules [gb, ge), read 32 columns at a time where a pair
        // of granules starts on an even index, 16 otherwise.
        const int gh = (ng + 1) >> 1, gb = hf ? gh : 0, ge = hf ? ng : gh;
        // ---- pass 1: row maximum
        float mx = -INFINITY;
        if (warp_live) {
          float m4[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
          int g = gb;
          // reading needs no alignment of the granule index: four granules (64 columns) per wait while they last
#pragma unroll 1
          for (; g + 4 <= ge; g += 4) {
            unsigned rc[16], rd[16];
            tca_ld(t_row + g * 16, ra, rb, rc, rd);
#pragma unroll
            for (int e = 0; e < 16; ++e)
              m4[e & 3] = tca_max3(tca_max3(m4[e & 3], __uint_as_float(ra[e]), __uint_as_float(rb[e])), __uint_as_float(rc[e]), __uint_as_float(rd[e]));
          }
#pragma unroll 1
          for (; g + 2 <= ge; g += 2) {
            tca_ld(t_row + g * 16, ra, rb);
#pragma unroll
            for (int e = 0; e < 16; ++e) m4[e & 3] = tca_max3(m4[e & 3], __uint_as_float(ra[e]), __uint_as_float(rb[e]));
          }
          if (g < ge) {
            tca_ld(t_row + g * 16, ra);
#pragma unroll
            for (int e = 0; e < 16; ++e) m4[e & 3] = fmaxf(m4[e & 3], __uint_as_float(ra[e]));
          }
          mx = fmaxf(fmaxf(m4[0], m4[1]), fmaxf(m4[2], m4[3]));
        }
        xm[hf * 128 + row] = mx;
        named_bar_sync(1 + wg, 256);
        mx = fmaxf(mx, xm[(hf ^ 1) * 128 + row]) + (jb ? bmax[1] : bmax[0]);       // upper bound of the biased scores of the row
        // ---- pass 2: weights, their sum, and P as packed bf16 pairs written over the first (even granules) or
        // second (odd granules) half of the granule's own score columns, which only this thread reads
        float lsum = 0.f;
        if (warp_live) {
          const float ms = -mx * sc2;
          // packed float pairs (add / fma on two floats per instruction) for everything around the exponentials
          float2 l2[2] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
          const float2 sc22 = make_float2(sc2, sc2), ms2 = make_float2(ms, ms);
          const unsigned char* brow = sBias + jb * p.bias_tile_bytes + row * bstride;
          auto pass2 = [&](int gg, const unsigned (&rr)[16]) {
            const uint4 b0 = *reinterpret_cast<const uint4*>(brow + gg * 32), b1 = *reinterpret_cast<const uint4*>(brow + gg * 32 + 16);
            const unsigned bw[8] = {b0.x, b0.y, b0.z, b0.w, b1.x, b1.y, b1.z, b1.w};
            unsigned pk[8];
#pragma unroll
            for (int e = 0; e < 8; ++e) {
              const float2 sv = make_float2(__uint_as_float(rr[2 * e]), __uint_as_float(rr[2 * e + 1]));
              const float2 bv = make_float2(__uint_as_float(bw[e] << 16), __uint_as_float(bw[e] & 0xffff0000u));
              const float2 x = __ffma2_rn(__fadd2_rn(sv, bv), sc22, ms2);
              const float2 pv = make_float2(tca_exp2(x.x), tca_exp2(x.y));
              l2[e & 1] = __fadd2_rn(l2[e & 1], pv);
              pk[e] = tca_pack(pv.x, pv.y);
            }
            tmem_st8(t_row + gg * 16 + (gg & 1) * 8, pk);
          };
          int g = gb;
          if ((g & 1) && g < ge) {
            tca_ld(t_row + g * 16, ra);
            pass2(g, ra);
            ++g;
          }
#pragma unroll 1
          for (; g + 2 <= ge; g += 2) {
            tca_ld(t_row + g * 16, ra, rb);
            pass2(g, ra);
            pass2(g + 1, rb);
          }
          if (g < ge) {
            tca_ld(t_row + g * 16, ra);
            pass2(g, ra);
          }
          lsum = (l2[0].x + l2[0].y) + (l2[1].x + l2[1].y);
          tmem_st_wait();
        }
        xm[256 + hf * 128 + row] = lsum;
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&pfull[wg]);
        // ---- output: O / l
        if ((sw & 7) == 0) mbar_wait(&ofull[wg], u & 1, ab);
        named_bar_sync(1 + wg, 256);                               // also: the partner's half of the row sum is visible
        tc_fence_after();
        if (warp_live && (D >= 32 || hf == 0)) {
          constexpr int CPT = D >= 32 ? D / 2 : D;                 // output channels per thread (16)
          const float inv = 1.0f / (xm[256 + row] + xm[256 + 128 + row]);
          tca_ld(t_row + TCA_O_COL + hf * CPT, ra);
          const long long orow = COL ? (long long)j * N + i : (long long)i * N + j;
          if (j < N && NT_IN(row_base + orow, m.pair_off[m.B] - p.row0, NT_SITE_ROW_ATTN_OUT)) {
            __nv_bfloat16* op = p.o + (p.row0 + row_base + orow) * Hd + h * D + hf * CPT;
            unsigned w[8];
#pragma unroll
            for (int e = 0; e < 8; ++e) w[e] = tca_pack(__uint_as_float(ra[2 * e]) * inv, __uint_as_float(ra[2 * e + 1]) * inv);
            // (one 32-byte store instead of two of 16: 206 -> 198 us at eight samples of 215)
            store_32b(op, w, ((unsigned long long)p.o & 31) == 0);
          }
        }
      }
    }
    it0 += (unsigned)cnt;
    r += cnt;
    __syncthreads();   // every role has finished the segment: the bias tiles may be replaced
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  abort_linger(ab);
  if (warp == 1) tmem_dealloc(tmem_base, 512);
}

static size_t tca_smem_bytes(int D, int n_max, bool has_bias, int nqk, int nv, int* kv_rows, int* tile_bytes) {
  const int rows = (n_max + 31) & ~31;
  *kv_rows = rows;
  *tile_bytes = 128 * tca_bias_stride((n_max + 15) & ~15) + 64;
  const int njb = (n_max + 127) / 128;
  return (size_t)nqk * (128 * 2 * D + rows * 2 * D) + (size_t)nv * rows * 2 * D + 2 * 2 * 2 * 2 * 128 * 4 +
         (size_t)njb * *tile_bytes + 1024;
}

template <int D, bool COL>
static nt_status launch_attn_tc(const __nv_bfloat16* q, const __nv_bfloat16* k, const __nv_bfloat16* v,
                                const __nv_bfloat16* bias, __nv_bfloat16* o, int H, const BatchMeta& m, int n_max,
                                int* status, cudaStream_t st) {
  AttnTcParams p;
  memset(&p, 0, sizeof(p));
  p.m = m;
  p.bias = bias;
  p.o = o;
  p.H = H;
  p.n_max = n_max;
  p.status = status;
  p.row0 = m.pair_off[0];
  const long long rows = m.pair_off[m.B] - p.row0;
  if (rows <= 0) return NT_OK;
  if (rows > 0x7FFFFF00ll) return NT_ERR_UNSUPPORTED;
  int longest = 0;
  p.item_off[0] = 0;
  for (int s = 0; s < m.B; ++s) {
    const int N = m.N[s];
    const bool take = N >= 1 && N <= n_max;
    if (take && N > longest) longest = N;
    p.item_off[s + 1] = p.item_off[s] + (take ? (long long)N * H * ((N + 127) / 128) : 0);
  }
  const long long total = p.item_off[m.B];
  if (total == 0) return NT_OK;
  const size_t limit = 232448;
  size_t smem = 0;
  const int tries[3][2] = {{3, 3}, {3, 2}, {2, 2}};
  for (int t = 0; t < 3; ++t) {
    p.nqk = tries[t][0];
    p.nv = tries[t][1];
    smem = tca_smem_bytes(D, longest, bias != nullptr, p.nqk, p.nv, &p.kv_rows, &p.bias_tile_bytes);
    if (smem <= limit) break;
  }
  if (smem > limit) return NT_ERR_UNSUPPORTED;
  const int Hd = H * D;
  if (COL) {
    // q, k, v must be three equally spaced buffers (they are carved that way): the map's outermost dimension picks one
    const long long gap = (const char*)k - (const char*)q;
    if (gap <= 0 || (const char*)v - (const char*)k != gap || gap % 16 != 0) return NT_ERR_UNSUPPORTED;
    for (int s = 0; s < m.B; ++s) {
      const int N = m.N[s];
      if (N < 1 || N > n_max) continue;
      const unsigned long long dims[4] = {(unsigned long long)Hd, (unsigned long long)N, (unsigned long long)N, 3};
      const unsigned long long strides[3] = {(unsigned long long)N * Hd * 2, (unsigned long long)Hd * 2, (unsigned long long)gap};
      const unsigned box[4] = {(unsigned)D, 32, 1, 1};
      if (!make_tmap_16bit(&p.cmap[s], q + m.pair_off[s] * Hd, 4, dims, strides, box, 2 * D, 2 * D >= 128 ? 128 : 2 * D))
        return cuda_fail("attn tc column map");
    }
  } else {
    const unsigned long long dims[2] = {(unsigned long long)Hd, (unsigned long long)rows};
    const unsigned long long strides[1] = {(unsigned long long)Hd * 2};
    const unsigned qbox[2] = {(unsigned)D, 128}, kbox[2] = {(unsigned)D, 32};
    if (!make_tmap_16bit(&p.qmap, q + p.row0 * Hd, 2, dims, strides, qbox, 2 * D, 2 * D >= 128 ? 128 : 2 * D)) return cuda_fail("attn tc q map");
    if (!make_tmap_16bit(&p.kmap, k + p.row0 * Hd, 2, dims, strides, kbox, 2 * D, 2 * D >= 128 ? 128 : 2 * D)) return cuda_fail("attn tc k map");
    if (!make_tmap_16bit(&p.vmap, v + p.row0 * Hd, 2, dims, strides, kbox, 2 * D, 2 * D >= 128 ? 128 : 2 * D)) return cuda_fail("attn tc v map");
  }
  // the attribute belongs to a (kernel, device) pair: one flag per device
  static bool attr_set_dev[64] = {};
  int attr_dev = 0;
  cudaGetDevice(&attr_dev);
  bool& attr_set = attr_set_dev[attr_dev & 63];
  if (!attr_set) {
    if (cudaFuncSetAttribute(attn_tc_kernel<D, COL>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)limit - 1024) != cudaSuccess)
      return cuda_fail("attention tc smem attribute");
    attr_set = true;
  }
  const unsigned grid = (unsigned)(total < sm_count() ? total : sm_count());
  {
    LaunchScope ls(COL ? "attn_core_col" : "attn_core", st);
    launch_kernel(attn_tc_kernel<D, COL>, grid, TCA_THREADS, smem, st, p);
  }
  return cuda_ok("attention tc launch");
}

int fast_attn_tc_max_n(int d, bool has_bias) {
  if (d != 16 && d != 32) return 0;
  int kv_rows, tile;
  int n = TCA_NMAX;
  while (n > 0 && tca_smem_bytes(d, n, has_bias, 2, 2, &kv_rows, &tile) > 232448 - 1024) n -= 8;
  return n;
}

nt_status fast_attn_core_tc(const void* q, const void* k, const void* v, const void* bias, void* o, int H, int d,
                            const BatchMeta& m, int n_max, int* status, cudaStream_t st, bool col) {
  const __nv_bfloat16* qq = (const __nv_bfloat16*)q;
  const __nv_bfloat16* kk = (const __nv_bfloat16*)k;
  const __nv_bfloat16* vv = (const __nv_bfloat16*)v;
  const __nv_bfloat16* bb = (const __nv_bfloat16*)bias;
  __nv_bfloat16* oo = (__nv_bfloat16*)o;
  if (col) {
    if (d == 16) return launch_attn_tc<16, true>(qq, kk, vv, bb, oo, H, m, n_max, status, st);
    if (d == 32) return launch_attn_tc<32, true>(qq, kk, vv, bb, oo, H, m, n_max, status, st);
    return NT_ERR_UNSUPPORTED;
  }
  if (d == 16) return launch_attn_tc<16, false>(qq, kk, vv, bb, oo, H, m, n_max, status, st);
  if (d == 32) return launch_attn_tc<32, false>(qq, kk, vv, bb, oo, H, m, n_max, status, st);
  return NT_ERR_UNSUPPORTED;
}

}  // namespace ntp
