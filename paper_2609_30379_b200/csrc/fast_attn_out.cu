// Attention output stage on tcgen05 (bf16, float accumulate), in place on the pair state:
//   z += (sigmoid(LN(z) W_g^T) * o) W_o^T
// The gate is recomputed from z here (LayerNorm folded into W_g: W_g' = bf16(W_g gamma) meets the bf16 state
// directly, the row statistics are taken beside the MMA and applied in the epilogue) instead of
// being written by the input projection.  Per 128-position tile: TMA brings the z tile and the o
// tile; the MMA warp computes the gate pre-activation into TMEM as soon as they land; the epilogue warps turn it
// into sigmoid(.) * o, written back over the o tile in shared memory; the MMA warp multiplies that by
// W_o; the epilogue adds the residual into the z tile and TMA-stores it.
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

constexpr int AO_THREADS = 64 + 128 + 256;   // producer, MMA, 4 statistics warps, 8 epilogue warps

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
  __shared__ __align__(8) unsigned long long bars[15];
  __shared__ float2 sStats[2][128];        // per stage: (mean, rstd) of every z row
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
  float* sC0 = reinterpret_cast<float*>(sSt + 2 * stage_bytes);   // c0 / 2 per gate channel
  float* sC1 = sC0 + Hd;                                          // c1 per gate channel
  unsigned long long* afull = bars;        // [2]
  unsigned long long* aempty = bars + 2;   // [2]
  unsigned long long* gfull = bars + 4;    // [2]
  unsigned long long* ogated = bars + 6;   // [2]
  unsigned long long* ofull = bars + 8;    // [2]
  unsigned long long* tempty = bars + 10;  // [2]
  unsigned long long* wfull = bars + 12;
  unsigned long long* aconv = bars + 13;   // [2]

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    abort_flag = 0;
    for (int s = 0; s < 2; ++s) {
      mbar_init(&afull[s], 1);
      mbar_init(&aempty[s], p.partial ? 2 + 8 : 2);   // + the epilogue warps that read the tile for the column sums
      mbar_init(&gfull[s], 1);
      mbar_init(&ogated[s], 8);
      mbar_init(&ofull[s], 1);
      mbar_init(&tempty[s], 8);
      mbar_init(&aconv[s], 4);
    }
    mbar_init(wfull, 1);
    mbar_fence_init();
  }
  if (warp == 1) tmem_alloc(&tmem_base_s, 512);
  for (int n = threadIdx.x; n < Hd; n += AO_THREADS) {
    sC0[n] = 0.5f * p.c01g[n].x;
    sC1[n] = p.c01g[n].y;
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  pdl_begin();
  const unsigned tmem_base = tmem_base_s;
  AbortCtx ab{p.status, &abort_flag};
  const long long ntiles = (p.rows + 127) / 128;

  if (warp == 0 && lane == 0) {
    // ------------------------------------------------------------------ producer
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
  } else if (warp == 1) {
    // ------------------------------------------------------------------ MMA issuer (whole warp, one elected lane issues)
    mbar_wait(wfull, 0, ab);
    int stage = 0;
    unsigned phase = 0, tph0 = 0, tph1 = 0, gph0 = 0, gph1 = 0;
    unsigned n = 0;
    const unsigned idesc_g = idesc_f16(128, Hd, 0, 0, FMT_BF16, FMT_BF16);  // the bf16 z tile, folded W_g bf16
    const unsigned idesc_o = idesc_f16(128, c, 0, 0, FMT_BF16, FMT_BF16);   // gated o bf16, W_o as given (bf16)
    const unsigned long long wg_desc = desc_kmajor_sw128(smem_u32(sWg)), wo_desc = desc_kmajor_sw128(smem_u32(sWo));
    const unsigned slab16 = (unsigned)slab >> 4, wg16 = (unsigned)wg_slab >> 4, wo16 = (unsigned)wo_slab >> 4;
    for (long long t = blockIdx.x; t < ntiles; t += gridDim.x, ++n) {
      const unsigned buf = n & 1;
      if (buf == 0) { mbar_wait(&tempty[0], tph0 ^ 1, ab); tph0 ^= 1; }
      else { mbar_wait(&tempty[1], tph1 ^ 1, ab); tph1 ^= 1; }
      mbar_wait(&afull[stage], phase, ab);
      tc_fence_after();
      const unsigned long long st_desc = desc_kmajor_sw128(smem_u32(sSt + stage * stage_bytes));
      const unsigned dg = tmem_base + buf * 256, dout = dg + Hd;
#pragma unroll
      for (int ks = 0; ks < 8; ++ks)
        if (ks < c / 16 && elect_one())
          umma_bf16(dg, st_desc + ((ks >> 2) * slab16 + (ks & 3) * 2), wg_desc + ((ks >> 2) * wg16 + (ks & 3) * 2), idesc_g, ks != 0);
      if (elect_one()) tc_commit(&gfull[buf]);
      __syncwarp();
      // gated o tile written back by the epilogue warps
      if (buf == 0) { mbar_wait(&ogated[0], gph0, ab); gph0 ^= 1; }
      else { mbar_wait(&ogated[1], gph1, ab); gph1 ^= 1; }
      tc_fence_after();
#pragma unroll
      for (int ks = 0; ks < 8; ++ks)
        if (ks < Hd / 16 && elect_one())
          umma_bf16(dout, st_desc + ((zslab + (ks >> 2)) * slab16 + (ks & 3) * 2), wo_desc + ((ks >> 2) * wo16 + (ks & 3) * 2),
                    idesc_o, ks != 0);
      if (elect_one()) {
        tc_commit(&ofull[buf]);
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
        sStats[stage][row] = zst;
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
      sStats[stage][row] = make_float2(mean, rsqrtf(fmaxf(sq / (float)c - mean * mean, 0.f) + p.eps));
      __syncwarp();
      if (lane == 0) mbar_arrive(&aconv[stage]);
      if (++stage == 2) { stage = 0; phase ^= 1; }
    }
  } else if (warp >= 6) {
    // ------------------------------------------------------------------ epilogue (8 warps)
    const int quarter = warp & 3;
    const int half = (warp - 6) >> 2;
    const int row = quarter * 32 + lane;
    const int ep_tid = threadIdx.x - 192;
    int stage = 0;
    unsigned gph[2] = {0, 0}, oph[2] = {0, 0};
    long long n = 0;
    for (long long t = blockIdx.x; t < ntiles; t += gridDim.x, ++n) {
      const int buf = (int)(n & 1);
      unsigned char* st = sSt + stage * stage_bytes;
      // ---- phase 1: o <- sigmoid(gate) * o, in place in shared memory
      mbar_wait(&aconv[stage], (unsigned)((n >> 1) & 1), ab);   // the row statistics are published
      mbar_wait(&gfull[buf], gph[buf], ab);
      gph[buf] ^= 1;
      tc_fence_after();
      // sigmoid(x) = tanh(x / 2) / 2 + 1 / 2 with x / 2 = (rstd / 2) acc + (c0 / 2 - mean (rstd / 2) c1), on packed float pairs
      const float rh = 0.5f * sStats[stage][row].y, mh = -sStats[stage][row].x * rh;
      const float2 rh2 = make_float2(rh, rh), mh2 = make_float2(mh, mh), half2 = make_float2(0.5f, 0.5f);
      const unsigned taddr = tmem_base + ((unsigned)(quarter * 32) << 16) + buf * 256;
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
            const float2 k0 = *reinterpret_cast<const float2*>(sC0 + c0 + n0), k1 = *reinterpret_cast<const float2*>(sC1 + c0 + n0);
            const float2 xh = __ffma2_rn(rh2, make_float2(__uint_as_float(r[n0]), __uint_as_float(r[n0 + 1])), __ffma2_rn(mh2, k1, k0));
            const float2 g = __ffma2_rn(half2, make_float2(ao_tanh(xh.x), ao_tanh(xh.y)), half2);
            const float2 go = __fmul2_rn(g, make_float2(__uint_as_float(w[e] << 16), __uint_as_float(w[e] & 0xffff0000u)));
            __nv_bfloat162 hh = __floats2bfloat162_rn(go.x, go.y);
            w[e] = *reinterpret_cast<unsigned*>(&hh);
          }
          *ptr = make_uint4(w[0], w[1], w[2], w[3]);
        }
      }
      tc_fence_before();
      fence_proxy_async_smem();
      __syncwarp();
      if (lane == 0) mbar_arrive(&ogated[buf]);
      // ---- phase 2: z += (gated o) W_o^T, in place in the z tile, then store
      mbar_wait(&ofull[buf], oph[buf], ab);
      oph[buf] ^= 1;
      tc_fence_after();
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
      __syncwarp();
      if (lane == 0) mbar_arrive(&tempty[buf]);
      fence_proxy_async_smem();
      named_bar_sync(1, 256);
      if (ep_tid == 0) {
        for (int sl = 0; sl < zslab; ++sl) tma_store_2d(&p.zmap, st + sl * slab, sl * 64, (int)(t * 128));
        tma_store_commit();
      }
      if (p.partial) {
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
      if (ep_tid == 0) {
        tma_store_wait_read0();
        mbar_arrive(&aempty[stage]);
      }
      if (++stage == 2) stage = 0;
    }
    if (ep_tid == 0) tma_store_wait_all0();
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
                      (size_t)Hd * 8 + 1024;
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
