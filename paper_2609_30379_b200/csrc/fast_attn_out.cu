// Attention output stage on tcgen05 (bf16, float accumulate), in place on the pair state:
//   z += (sigmoid(LN(z) W_g^T) * o) W_o^T
// The gate is recomputed from z here (LayerNorm folded into W_g: W_g' = bf16(W_g gamma) meets the bf16 state
// directly, the row statistics are taken beside the MMA and enter it as one more K step, ln_aug_row) instead of
// being written by the input projection.  Per 128-position tile: TMA brings the z tile and the o tile; the gate MMAs
// run as soon as they land; eight gate warps turn the result into sigmoid(.) * o, written back over the o tile in
// shared memory; the output MMAs multiply that by W_o; eight output warps add the residual into the z tile, and a
// warp of its own stores it.
// Bound: the life of a tile -- load, gate MMA, gate warps, output MMA, output warps, store -- with room for two of them
// beside the weights.  With one group of warps for both stages, the two tiles' lives did not overlap at all.
// Measured at eight samples of about 215 positions: 79 us with one group of eight warps, 66 us so.
//
// Optional fused reduction (the mean over j that follows the attention in the block): while the finished tile is
// still in shared memory the epilogue threads add up its columns per group of 32 positions, split at the one pair
// row boundary such a group can contain (every sample of the batch has N >= 32 or is empty), and write the two
// partial sums to a scratch array; a second small kernel adds the partials of every pair row in a fixed order.  The
// state is then never read back for the reduction.
#include <cstring>

#include "fast.cuh"
#include "tc_common.cuh"

namespace ntp {

// producer, gate MMAs, 4 statistics warps, 8 gate warps, 8 output warps, store, output MMAs
constexpr int AO_GATE = 6, AO_OUT = 14, AO_STORE = 22, AO_MMA2 = 23;
constexpr int AO_THREADS = 32 * 24;

struct AttnOutParams {
  CUtensorMap zmap;              // {c, rows}, box {64, 128}: load and store
  CUtensorMap omap;              // {Hd, rows}, box {64, 128}
  CUtensorMap wgmap;             // {c, Hd}, box {64, Hd}
  CUtensorMap womap;             // {Hd, c}, box {64, c}
  int c, Hd;
  long long rows;
  float eps;
  const float2* c01g;            // [Hd]
  int* status;
  const float2* zstats;          // nullable: (mean, rstd) of every z row, left by the input projection
  float* partial;                // nullable: [ceil(rows / 32)][2][c] column sums of 32-position groups
  long long P0;                  // packed position of row 0 of the maps
  BatchMeta m;                   // read only when partial != nullptr
};

__device__ inline float ao_tanh(float x) {
  float t;
  asm("tanh.approx.f32 %0, %1;\n" : "=f"(t) : "f"(x));
  return t;
}

__global__ void __launch_bounds__(AO_THREADS, 1) attn_out_kernel(const __grid_constant__ AttnOutParams p) {
  extern __shared__ unsigned char smem_raw[];
  __shared__ __align__(8) unsigned long long bars[17];
  __shared__ float sStats[2][128];         // per stage: rstd / 2 of every z row
  __shared__ unsigned tmem_base_s;
  __shared__ int abort_flag;
  unsigned char* smem = smem_raw + ((1024 - (smem_u32(smem_raw) & 1023)) & 1023);
  const int c = p.c, Hd = p.Hd;
  const int zslab = c / 64, oslab = Hd / 64;
  const int slab = 128 * 128;
  const int wg_slab = Hd * 128, wo_slab = c * 128;
  const int stage_bytes = (zslab + oslab) * slab;
  unsigned char* sWg = smem;                          // zslab slabs of [Hd rows][64]
  unsigned char* sWo = sWg + zslab * wg_slab;         // oslab slabs of [c rows][64]
  unsigned char* sSt = sWo + oslab * wo_slab;         // 2 stages: z slabs then o slabs
  unsigned char* sAx = sSt + 2 * stage_bytes;         // [2 stages][2][128][8] bf16: augmentation columns 0-7, 8-15 of the rows
  unsigned char* sBx = sAx + 2 * 4096;                // [2][Hd][8] bf16: the same of W_g
  unsigned long long* afull = bars;        // [2]
  unsigned long long* aempty = bars + 2;   // [2]
  unsigned long long* gfull = bars + 4;    // [2]
  unsigned long long* ogated = bars + 6;   // [2]
  unsigned long long* ofull = bars + 8;    // [2]
  unsigned long long* tempty = bars + 10;  // [2]
  unsigned long long* wfull = bars + 12;
  unsigned long long* aconv = bars + 13;   // [2]
  unsigned long long* zdone = bars + 15;   // [2] the new z is in the tile

  const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;   // warp-uniform for the compiler too
  if (threadIdx.x == 0) {
    abort_flag = 0;
    for (int s = 0; s < 2; ++s) {
      mbar_init(&afull[s], 1);
      mbar_init(&aempty[s], p.partial ? 2 + 8 : 2);   // output MMAs, store, + the output warps that read the tile for the column sums
      mbar_init(&gfull[s], 1);
      mbar_init(&ogated[s], 8);
      mbar_init(&ofull[s], 1);
      mbar_init(&tempty[s], 8);
      mbar_init(&aconv[s], 4);
      mbar_init(&zdone[s], 8);
    }
    mbar_init(wfull, 1);
    mbar_fence_init();
  }
  if (warp == 1) tmem_alloc(&tmem_base_s, 512);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  pdl_begin();
  for (int n = threadIdx.x; n < Hd; n += AO_THREADS) ln_aug_weight(sBx + n * 16, Hd * 16, p.c01g[n]);
  fence_proxy_async_smem();
  __syncthreads();
  const unsigned tmem_base = __shfl_sync(0xffffffffu, tmem_base_s, 0);
  AbortCtx ab{p.status, &abort_flag};
  const long long ntiles = (p.rows + 127) / 128;

  if (warp == 0) {
    // ------------------------------------------------------------------ producer
    if (lane == 0) {
      mbar_expect_tx(wfull, zslab * wg_slab + oslab * wo_slab);
      for (int sl = 0; sl < zslab; ++sl) tma_load_2d(sWg + sl * wg_slab, &p.wgmap, wfull, sl * 64, 0);
      for (int sl = 0; sl < oslab; ++sl) tma_load_2d(sWo + sl * wo_slab, &p.womap, wfull, sl * 64, 0);
      int stage = 0;
      unsigned phase = 0;
      for (long long t = blockIdx.x; t < ntiles; t += gridDim.x) {
        mbar_wait(&aempty[stage], phase ^ 1, ab);
        mbar_expect_tx(&afull[stage], stage_bytes);
        unsigned char* st = sSt + stage * stage_bytes;
        for (int sl = 0; sl < zslab; ++sl) tma_load_2d(st + sl * slab, &p.zmap, &afull[stage], sl * 64, (int)(t * 128));
        for (int sl = 0; sl < oslab; ++sl)
          tma_load_2d(st + (zslab + sl) * slab, &p.omap, &afull[stage], sl * 64, (int)(t * 128));
        if (++stage == 2) { stage = 0; phase ^= 1; }
      }
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------------ gate MMAs (whole warp, one elected lane issues)
    mbar_wait(wfull, 0, ab);
    int stage = 0;
    unsigned phase = 0;
    const unsigned idesc_g = idesc_f16(128, Hd, 0, 0, FMT_BF16, FMT_BF16);  // the bf16 z tile, folded W_g bf16
    const unsigned long long wg_desc = desc_kmajor_sw128(smem_u32(sWg));
    const unsigned slab16 = (unsigned)slab >> 4, wg16 = (unsigned)wg_slab >> 4;
    const unsigned long long bx_desc = desc_kmajor_nosw(smem_u32(sBx), Hd * 16, 128);
    for (long long t = blockIdx.x; t < ntiles; t += gridDim.x) {
      mbar_wait(&tempty[stage], phase ^ 1, ab);              // accumulators and stages advance together
      mbar_wait(&afull[stage], phase, ab);
      tc_fence_after();
      const unsigned long long st_desc = desc_kmajor_sw128(smem_u32(sSt + stage * stage_bytes));
      const unsigned dg = tmem_base + stage * 256;
#pragma unroll
      for (int sl = 0; sl < 2; ++sl)
        if (sl < zslab) umma_k4(dg, st_desc + sl * slab16, wg_desc + sl * wg16, idesc_g, sl);
      mbar_wait(&aconv[stage], phase, ab);                   // the rows' augmentation columns are written
      tc_fence_after();
      if (elect_one()) {
        umma_bf16(dg, desc_kmajor_nosw(smem_u32(sAx + stage * 4096), 2048, 128), bx_desc, idesc_g, 1);
        tc_commit(&gfull[stage]);
      }
      __syncwarp();
      if (++stage == 2) { stage = 0; phase ^= 1; }
    }
  } else if (warp == AO_MMA2) {
    // ------------------------------------------------------------------ output MMAs: an issuer of their own, so that they
    // never wait for the next tile's load and its gate MMAs never for this tile's gate warps
    mbar_wait(wfull, 0, ab);
    int stage = 0;
    unsigned phase = 0;
    const unsigned idesc_o = idesc_f16(128, c, 0, 0, FMT_BF16, FMT_BF16);   // gated o bf16, W_o as given (bf16)
    const unsigned long long wo_desc = desc_kmajor_sw128(smem_u32(sWo));
    const unsigned slab16 = (unsigned)slab >> 4, wo16 = (unsigned)wo_slab >> 4;
    for (long long t = blockIdx.x; t < ntiles; t += gridDim.x) {
      mbar_wait(&ogated[stage], phase, ab);
      tc_fence_after();
      const unsigned long long o_desc = desc_kmajor_sw128(smem_u32(sSt + stage * stage_bytes + zslab * slab));
      const unsigned dout = tmem_base + stage * 256 + Hd;
#pragma unroll
      for (int sl = 0; sl < 2; ++sl)
        if (sl < oslab) umma_k4(dout, o_desc + sl * slab16, wo_desc + sl * wo16, idesc_o, sl);
      if (elect_one()) {
        tc_commit(&ofull[stage]);
        tc_commit(&aempty[stage]);
      }
      __syncwarp();
      if (++stage == 2) { stage = 0; phase ^= 1; }
    }
  } else if (warp >= 2 && warp < 6) {
    // ------------------------------------------------------------------ row statistics (4 warps, one row per thread),
    // beside the gate MMA
    const int row = (warp - 2) * 32 + lane;
    int stage = 0;
    unsigned phase = 0;
    for (long long t = blockIdx.x; t < ntiles; t += gridDim.x) {
      if (p.zstats) {                       // the input projection normalised the same rows: take its statistics
        const float2 zst = t * 128 + row < p.rows ? *(p.zstats + t * 128 + row) : make_float2(0.f, 1.f);
        mbar_wait(&afull[stage], phase, ab);
        sStats[stage][row] = 0.5f * ln_aug_row(sAx + stage * 4096 + row * 16, 2048, zst.x, zst.y);
        fence_proxy_async_smem();
        __syncwarp();
        if (lane == 0) mbar_arrive(&aconv[stage]);
        if (++stage == 2) { stage = 0; phase ^= 1; }
        continue;
      }
      mbar_wait(&afull[stage], phase, ab);
      float s4[4] = {0.f, 0.f, 0.f, 0.f}, q4[4] = {0.f, 0.f, 0.f, 0.f};
      const unsigned char* zt = sSt + stage * stage_bytes;
      for (int g8 = 0; g8 < c / 8; ++g8) {
        const uint4 v = *reinterpret_cast<const uint4*>(zt + (g8 >> 3) * slab + sw128_off(row, g8 & 7));
        const unsigned w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const float lo = __uint_as_float(w[e] << 16), hi = __uint_as_float(w[e] & 0xffff0000u);
          s4[e] += lo + hi;
          q4[e] = fmaf(lo, lo, q4[e]);
          q4[e] = fmaf(hi, hi, q4[e]);
        }
      }
      const float sum = (s4[0] + s4[1]) + (s4[2] + s4[3]), sq = (q4[0] + q4[1]) + (q4[2] + q4[3]);
      const float mean = sum / (float)c;
      const float rstd = rsqrtf(fmaxf(sq / (float)c - mean * mean, 0.f) + p.eps);
      sStats[stage][row] = 0.5f * ln_aug_row(sAx + stage * 4096 + row * 16, 2048, mean, rstd);
      fence_proxy_async_smem();
      __syncwarp();
      if (lane == 0) mbar_arrive(&aconv[stage]);
      if (++stage == 2) { stage = 0; phase ^= 1; }
    }
  } else if (warp < AO_OUT) {
    // ------------------------------------------------------------------ gate warps: o <- sigmoid(gate) * o, in place in shared memory
    const int quarter = warp & 3;
    const int half = (warp - AO_GATE) >> 2;
    const int row = quarter * 32 + lane;
    int stage = 0;
    unsigned phase = 0;
    for (long long t = blockIdx.x; t < ntiles; t += gridDim.x) {
      unsigned char* st = sSt + stage * stage_bytes;
      mbar_wait(&gfull[stage], phase, ab);
      mbar_wait(&aconv[stage], phase, ab);   // (long complete: orders the read of what the statistics warps left)
      tc_fence_after();
      // sigmoid(x) o = tanh(x / 2) (o / 2) + o / 2 with x / 2 = (rstd / 2) acc, on packed float pairs
      const float rh = sStats[stage][row];
      const float2 rh2 = make_float2(rh, rh), half2 = make_float2(0.5f, 0.5f);
      const unsigned taddr = tmem_base + ((unsigned)(quarter * 32) << 16) + stage * 256;
#pragma unroll 1
      for (int c0 = half * (Hd / 2); c0 < (half + 1) * (Hd / 2); c0 += 32) {
        unsigned r[32];
        tmem_ld32(taddr + c0, r);
        tmem_ld_wait();
        unsigned char* op = st + (zslab + (c0 >> 6)) * slab;
#pragma unroll
        for (int ch = 0; ch < 4; ++ch) {
          uint4* ptr = reinterpret_cast<uint4*>(op + sw128_off(row, ((c0 & 63) >> 3) + ch));
          const uint4 v = *ptr;
          unsigned w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            const int n0 = ch * 8 + e * 2;
            const float2 xh = __fmul2_rn(rh2, make_float2(__uint_as_float(r[n0]), __uint_as_float(r[n0 + 1])));
            const float2 oh = __fmul2_rn(half2, make_float2(__uint_as_float(w[e] << 16), __uint_as_float(w[e] & 0xffff0000u)));
            const float2 go = __ffma2_rn(make_float2(ao_tanh(xh.x), ao_tanh(xh.y)), oh, oh);
            __nv_bfloat162 hh = __floats2bfloat162_rn(go.x, go.y);
            w[e] = *reinterpret_cast<unsigned*>(&hh);
          }
          *ptr = make_uint4(w[0], w[1], w[2], w[3]);
        }
      }
      tc_fence_before();
      fence_proxy_async_smem();
      __syncwarp();
      if (lane == 0) mbar_arrive(&ogated[stage]);
      if (++stage == 2) { stage = 0; phase ^= 1; }
    }
  } else if (warp < AO_STORE) {
    // ------------------------------------------------------------------ output warps: z += (gated o) W_o^T, in place in the z tile
    const int quarter = warp & 3;
    const int half = (warp - AO_OUT) >> 2;
    const int row = quarter * 32 + lane;
    const int ep_tid = threadIdx.x - AO_OUT * 32;
    int stage = 0;
    unsigned phase = 0;
    for (long long t = blockIdx.x; t < ntiles; t += gridDim.x) {
      unsigned char* st = sSt + stage * stage_bytes;
      const unsigned taddr = tmem_base + ((unsigned)(quarter * 32) << 16) + stage * 256;
      mbar_wait(&ofull[stage], phase, ab);
      tc_fence_after();
#pragma unroll 1
      for (int c0 = half * (c / 2); c0 < (half + 1) * (c / 2); c0 += 32) {
        unsigned r[32];
        tmem_ld32(taddr + Hd + c0, r);
        tmem_ld_wait();
        unsigned char* zp = st + (c0 >> 6) * slab;
#pragma unroll
        for (int ch = 0; ch < 4; ++ch) {
          uint4* ptr = reinterpret_cast<uint4*>(zp + sw128_off(row, ((c0 & 63) >> 3) + ch));
          const uint4 v = *ptr;
          unsigned w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            const int n0 = ch * 8 + e * 2;
            const float2 zn = __fadd2_rn(make_float2(__uint_as_float(w[e] << 16), __uint_as_float(w[e] & 0xffff0000u)),   // the bf16 state
                                         make_float2(__uint_as_float(r[n0]), __uint_as_float(r[n0 + 1])));
            __nv_bfloat162 hh = __floats2bfloat162_rn(zn.x, zn.y);
            w[e] = *reinterpret_cast<unsigned*>(&hh);
          }
          *ptr = make_uint4(w[0], w[1], w[2], w[3]);
        }
      }
      tc_fence_before();
      fence_proxy_async_smem();
      __syncwarp();
      if (lane == 0) {
        mbar_arrive(&tempty[stage]);
        mbar_arrive(&zdone[stage]);
      }
      if (p.partial) {
        named_bar_sync(1, 256);
        // thread = (channel pair, quarter of the tile): column sums of 32 positions, split at the pair row boundary
        const int cp = ep_tid & 63, q = ep_tid >> 6;
        const long long p0 = t * 128 + q * 32;
        if (cp < c / 2 && p0 < p.rows) {
          const int nvalid = (int)min(32ll, p.rows - p0);
          const int s = find_sample(p.m.pair_off, p.m.B, p.P0 + p0);
          const unsigned N = (unsigned)p.m.N[s];
          const unsigned rem = (unsigned)(p.P0 + p0 - p.m.pair_off[s]) % N;        // N^2 < 2^32 on this path
          const int br = rem == 0 ? nvalid : (int)min((unsigned)nvalid, N - rem);   // positions of the row that holds p0
          const unsigned char* zt = st + (cp >> 5) * slab + (cp & 3) * 4;
          const int chunk = (cp & 31) >> 2;
          float2 a0 = make_float2(0.f, 0.f), a1 = make_float2(0.f, 0.f);
          if (br == 32) {                    // no boundary inside: four independent chains
            float2 b0 = a0, b1 = a0, b2 = a0;
#pragma unroll
            for (int r = 0; r < 32; r += 4) {
              const unsigned w0 = *reinterpret_cast<const unsigned*>(zt + sw128_off(q * 32 + r, chunk));
              const unsigned w1 = *reinterpret_cast<const unsigned*>(zt + sw128_off(q * 32 + r + 1, chunk));
              const unsigned w2 = *reinterpret_cast<const unsigned*>(zt + sw128_off(q * 32 + r + 2, chunk));
              const unsigned w3 = *reinterpret_cast<const unsigned*>(zt + sw128_off(q * 32 + r + 3, chunk));
              a0 = __fadd2_rn(a0, make_float2(__uint_as_float(w0 << 16), __uint_as_float(w0 & 0xffff0000u)));
              b0 = __fadd2_rn(b0, make_float2(__uint_as_float(w1 << 16), __uint_as_float(w1 & 0xffff0000u)));
              b1 = __fadd2_rn(b1, make_float2(__uint_as_float(w2 << 16), __uint_as_float(w2 & 0xffff0000u)));
              b2 = __fadd2_rn(b2, make_float2(__uint_as_float(w3 << 16), __uint_as_float(w3 & 0xffff0000u)));
            }
            a0 = __fadd2_rn(__fadd2_rn(a0, b0), __fadd2_rn(b1, b2));
          } else {
            for (int r = 0; r < br; ++r) {
              const unsigned w = *reinterpret_cast<const unsigned*>(zt + sw128_off(q * 32 + r, chunk));
              a0.x += __uint_as_float(w << 16);
              a0.y += __uint_as_float(w & 0xffff0000u);
            }
            for (int r = br; r < nvalid; ++r) {
              const unsigned w = *reinterpret_cast<const unsigned*>(zt + sw128_off(q * 32 + r, chunk));
              a1.x += __uint_as_float(w << 16);
              a1.y += __uint_as_float(w & 0xffff0000u);
            }
          }
          float2* dst = reinterpret_cast<float2*>(p.partial + ((t * 4 + q) * 2) * (long long)c) + cp;
          dst[0] = a0;
          dst[c / 2] = a1;
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(&aempty[stage]);      // this warp has read what it needs of the tile
      }
      if (++stage == 2) { stage = 0; phase ^= 1; }
    }
  } else if (warp == AO_STORE) {
    // ------------------------------------------------------------------ store: lane l takes slab l
    int stage = 0;
    unsigned phase = 0;
    for (long long t = blockIdx.x; t < ntiles; t += gridDim.x) {
      mbar_wait(&zdone[stage], phase, ab);
      if (lane < zslab) tma_store_2d(&p.zmap, sSt + stage * stage_bytes + lane * slab, lane * 64, (int)(t * 128));
      tma_store_commit();
      tma_store_wait_read0();
      __syncwarp();
      if (lane == 0) mbar_arrive(&aempty[stage]);
      if (++stage == 2) { stage = 0; phase ^= 1; }
    }
    tma_store_wait_all0();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  abort_linger(ab);
  if (warp == 1) tmem_dealloc(tmem_base, 512);
}

// Adds the partial column sums of every pair row (= token row g of the group) in ascending position order.  Group
// mt of 32 positions keeps the sum of the row that holds its first position in slot 0 and of the row that starts
// inside it in slot 1.
__global__ void __launch_bounds__(128) segment_partials_kernel(const float* partial, BatchMeta m,
                                                               long long P0, int C, int mean,
                                                               __nv_bfloat16* out) {
  pdl_begin();
  const long long g = m.tok_off[0] + blockIdx.x;
  const int s = find_sample(m.tok_off, m.B, g);
  const long long N = m.N[s];
  const long long lo = m.pair_off[s] + (g - m.tok_off[s]) * N - P0, hi = lo + N;
  const float sc = mean ? 1.0f / (float)N : 1.0f;
  const long long mt0 = lo >> 5, mt1 = (hi - 1) >> 5;
  for (int c = threadIdx.x; c < C; c += 128) {
    float tot = 0.f;
    for (long long mb = mt0; mb <= mt1; mb += 8) {     // eight loads in flight, added in ascending order
      float v[8];
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        const long long mt = mb + k;
        v[k] = mt <= mt1 ? partial[(mt * 2 + (lo > (mt << 5) ? 1 : 0)) * C + c] : 0.f;
      }
#pragma unroll
      for (int k = 0; k < 8; ++k) tot += v[k];
    }
    out[g * C + c] = __float2bfloat16_rn(tot * sc);
  }
}

// The fused reduction needs every 32 consecutive positions to meet at most one pair row boundary.
bool fast_attn_out_reduce_supported(const BatchMeta& m) {
  for (int s = 0; s < m.B; ++s)
    if (m.N[s] > 0 && m.N[s] < 32) return false;
  return true;
}

size_t fast_attn_out_partial_bytes(long long rows, int c) { return (size_t)((rows + 31) / 32) * 2 * c * sizeof(float); }

nt_status fast_segment_partials(const float* partial, const BatchMeta& m, int C, int mean, void* out, cudaStream_t st) {
  const long long G = m.tok_off[m.B] - m.tok_off[0];
  if (G <= 0) return NT_OK;
  if (G > 0x7FFFFFFFll) return NT_ERR_UNSUPPORTED;
  {
    LaunchScope ls("segment_partials", st);
    launch_kernel(segment_partials_kernel, (unsigned)G, 128, 0, st, partial, m, m.pair_off[0], C, mean, (__nv_bfloat16*)out);
  }
  return cuda_ok();
}

bool fast_attn_out_supported(int c, int H, int d) {
  const int Hd = H * d;
  // the prepared weights place the folded gate rows behind 16 bias rows (H of them real): more heads than that
  // would overlap the two
  return (c == 64 || c == 128) && (Hd == 64 || Hd == 128) && H <= 16;
}

nt_status fast_attn_out(void* z, const void* o, const void* W_o, const AttnPrep& ap, float eps, int c, int H, int d,
                        const BatchMeta& m, int* status, cudaStream_t st, float* partial, const float2* zstats) {
  const int Hd = H * d;
  const void* wg = ap.wg;
  const float2* c01g = (const float2*)ap.c01g;
  const int zslab = c / 64, oslab = Hd / 64;
  const size_t smem = (size_t)zslab * Hd * 128 + (size_t)oslab * c * 128 + 2 * (size_t)(zslab + oslab) * 128 * 128 +
                      2 * 4096 + (size_t)Hd * 32 + 1024;
  // the attribute belongs to a (kernel, device) pair: one flag per device
  static bool attr_set_dev[64] = {};
  int attr_dev = 0;
  cudaGetDevice(&attr_dev);
  bool& attr_set = attr_set_dev[attr_dev & 63];
  if (!attr_set) {
    if (cudaFuncSetAttribute(attn_out_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 220 * 1024) != cudaSuccess)
      return cuda_fail("attn_out smem attribute");
    attr_set = true;
  }
  AttnOutParams p;
  memset(&p, 0, sizeof(p));
  const long long P0 = m.pair_off[0];
  p.rows = m.pair_off[m.B] - P0;
  if (p.rows == 0) return NT_OK;
  if (p.rows > 0x7FFFFF00ll) return NT_ERR_UNSUPPORTED;
  p.c = c;
  p.Hd = Hd;
  p.eps = eps;
  p.c01g = c01g;
  p.status = status;
  p.partial = partial;
  p.zstats = zstats ? zstats + P0 : nullptr;
  p.P0 = P0;
  if (partial) p.m = m;
  {
    const unsigned box[2] = {64, 128};
    const unsigned long long zdims[2] = {(unsigned long long)c, (unsigned long long)p.rows};
    const unsigned long long zstr[1] = {(unsigned long long)c * 2};
    if (!make_tmap_bf16(&p.zmap, (char*)z + (size_t)P0 * c * 2, 2, zdims, zstr, box)) return cuda_fail("attn_out z map");
    const unsigned long long odims[2] = {(unsigned long long)Hd, (unsigned long long)p.rows};
    const unsigned long long ostr[1] = {(unsigned long long)Hd * 2};
    if (!make_tmap_bf16(&p.omap, (const char*)o + (size_t)P0 * Hd * 2, 2, odims, ostr, box))
      return cuda_fail("attn_out o map");
    const unsigned long long gdims[2] = {(unsigned long long)c, (unsigned long long)Hd};
    const unsigned gbox[2] = {64, (unsigned)Hd};
    if (!make_tmap_bf16(&p.wgmap, wg, 2, gdims, zstr, gbox)) return cuda_fail("attn_out W_g map");
    const unsigned long long wdims[2] = {(unsigned long long)Hd, (unsigned long long)c};
    const unsigned wbox[2] = {64, (unsigned)c};
    if (!make_tmap_bf16(&p.womap, W_o, 2, wdims, ostr, wbox)) return cuda_fail("attn_out W_o map");
  }
  const long long ntiles = (p.rows + 127) / 128;
  const unsigned grid = (unsigned)(ntiles < sm_count() ? ntiles : sm_count());
  {
    LaunchScope ls("attn_out", st);
    launch_kernel(attn_out_kernel, grid, AO_THREADS, smem, st, p);
  }
  if (cudaPeekAtLastError() != cudaSuccess) return cuda_fail("attn_out launch");
  return NT_OK;
}

}  // namespace ntp
