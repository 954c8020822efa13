// SwiGLU pair transition on tcgen05, fused so that the expanded hidden activation never leaves the SM:
//   zh = LN(z);  z += (silu(zh W_a^T) * (zh W_b^T)) W_2^T          (position-wise on packed rows)
//
// A persistent CTA per SM walks PAIRS of tiles of 128 consecutive packed rows; the two tiles of a pair share every
// weight slice that streams in from L2 (the weights, 3 c hidden elements, do not fit in shared memory), which halves
// that traffic.  The hidden width is processed in chunks of 64 units, two halves of 32; per tile and chunk
//   GEMM 1  [128 rows x c] x [32 gate | 32 value | 32 gate | 32 value rows of the folded W_a / W_b]^T -> 128 TMEM columns
//   gate    h = silu(g) * v in registers (g arrives halved: silu(g) = g' tanh(g') + g' with g' = g / 2), packed bf16
//           and stored back over the gate columns it came from; each half has four warps of its own
//   GEMM 2  out[128 rows x c] += h[128 x 32](TMEM) x W_2[:, half]^T per half, accumulated over the chunks in TMEM
// and at the end of the tile out + z goes back through the z tile in shared memory and TMA stores.
// What bounds it: shared-memory reads of the MMAs.  An MMA of N columns and 16 K values reads 4 KB of rows and 32 N bytes of
// weights at 128 bytes per clock and needs N / 2 clocks of the tensor pipe, so N = 64 runs at two thirds of the
// tensor rate (measured 48 clocks for 32) and leaves no bandwidth for anything else, while N = 128 runs at the full
// rate (64 clocks).  Hence one GEMM 1 of 128 columns per tile rather than two accumulator buffers of 64; while one tile
// is in its gate stage the other tile's MMAs fill the tensor pipe.  GEMM 1 of the next chunk overwrites the columns that
// GEMM 2 has just read and waits for it to be complete: the order in which MMAs are issued is only guaranteed to be
// kept between those of one shape into one accumulator.  TMEM columns:
// [0, 256) two tiles x two halves x (32 gate | 32 value), [256, 512) two output accumulators.
// Measured (256,653 rows, c = 128, hidden 512): 155 us with two buffers of 64 columns, 107 us so (99 without the wait for
// GEMM 2); c = 64, hidden 256: 71 and 50 us.
// LayerNorm is folded into the weights (W' = W gamma, fp16); its mean and offset ride in GEMM 1 as one more K step:
// (-mean_hi, -mean_lo, -mean_hi, s_hi, s_hi, s_lo, 4096 s_rest, 0) per row, s = 1 / rstd split into fp16 parts, against
// (c1_hi, c1_hi, c1_lo, c0_hi, c0_lo, c0_hi, c0_hi / 4096, 0) per weight row, so that rstd times the accumulator is
// the normalised projection; the z tile itself is only converted bf16 -> fp16 (exact), because it is also the residual.
// The state tiles are double buffered per tile of the pair: the next pair loads and converts while this one computes.
// Roles: warp 0 producer (W_1 ring, state tiles), warp 22 producer (W_2 ring), warp 1 MMA issuer (converged, one
// elected lane), warps 2-5 converters (one row per thread), warps 6-21 gate and output stage: two groups
// of four per tile.  All waits are bounded.
#include <cstring>

#include "fast.cuh"
#include "tc_common.cuh"

namespace ntp {

constexpr int TR_HALF = 32;                   // hidden units per half: one gate group, one GEMM 2
constexpr int TR_CHUNK = 2 * TR_HALF;         // hidden units per GEMM 1
constexpr int TR_WST = 2;                     // stages of either weight ring: W_1 by chunk, W_2 by half
constexpr int TR_GATE_WARPS = 16;             // two groups of four per tile: first and second half of a chunk
constexpr int TR_W2PROD = 6 + TR_GATE_WARPS;  // warp that loads W_2
constexpr int TR_THREADS = 32 * (TR_W2PROD + 1);
constexpr int TR_SMEM_MAX = 224 * 1024;       // dynamic; c = 128 needs 228352 bytes

struct TransParams {
  CUtensorMap zmap;      // state {c, rows}, box {64, 128} (loads)
  CUtensorMap zsmap;     // same tensor, box {64, 32} (stores, one per warp and slab)
  CUtensorMap w1map;     // folded [W_a / 2; W_b] {c, 2 hidden} fp16, box {64, 32}
  CUtensorMap w1xmap;    // augmentation columns {8, 2 * 2 hidden} fp16, box {8, 32}, no swizzle
  CUtensorMap w2map;     // W_2 {hidden, c} bf16, box {32, c}, 64-byte swizzle (one half)
  long long rows;
  int c, hidden;
  float eps;
  int* status;
};

__device__ inline float tr_tanh(float x) {
  float t;
  asm("tanh.approx.f32 %0, %1;\n" : "=f"(t) : "f"(x));
  return t;
}

// K-major operand whose rows are 64 bytes (32 elements), 64-byte swizzle: 8 rows form a 512-byte atom
__device__ inline unsigned long long tr_desc_sw64(unsigned saddr) {
  unsigned long long d = 0;
  d |= (unsigned long long)((saddr & 0x3FFFFu) >> 4);
  d |= (unsigned long long)(512 >> 4) << 16;
  d |= (unsigned long long)(512 >> 4) << 32;
  d |= (unsigned long long)1 << 46;
  d |= (unsigned long long)4 << 61;
  return d;
}

__global__ void __launch_bounds__(TR_THREADS, 1) transition_kernel(const __grid_constant__ TransParams p) {
  extern __shared__ unsigned char smem_raw[];
  __shared__ __align__(8) unsigned long long bars[30];
  __shared__ float sRstd[4][128];
  __shared__ unsigned tmem_base_s;
  __shared__ int abort_flag;
  unsigned char* smem = smem_raw + ((1024 - (smem_u32(smem_raw) & 1023)) & 1023);
  const int c = p.c, hidden = p.hidden;
  const int nslab = c / 64;
  const int nhalf = hidden / TR_HALF;                // an odd count leaves the second half of the last chunk unused
  const int nchunk = (nhalf + 1) / 2;
  const int slab = 128 * 128;                        // [128 rows][64 channels] of 16-bit elements, either operand
  const int z_stage = nslab * slab;
  const int w1_bytes = nslab * slab;                 // [gate | value | gate | value][32 rows] x c
  const int w1_stage = w1_bytes + 2048;              // + augmentation columns 0-7 of the 128 weight rows
  const int w2_bytes = c * 2 * TR_HALF;              // [c rows][32 hidden units] of bf16
  unsigned char* sZ = smem;                          // 4 buffers, index tile * 2 + pair parity
  unsigned char* sW1 = sZ + 4 * z_stage;             // ring: [W1 chunk | its augmentation]; free once both GEMM 1s ran
  unsigned char* sW2 = sW1 + TR_WST * w1_stage;      // ring of W_2 slices; free once both GEMM 2s ran
  unsigned char* sZx = sW2 + TR_WST * w2_bytes;      // 4 x [128][8] fp16: augmentation columns 0-7 of the rows
  unsigned char* sZero = sZx + 4 * 2048;             // [128][8] zeros: augmentation columns 8-15 of either operand
  unsigned long long* zfull = bars;         // [4]
  unsigned long long* zempty = bars + 4;    // [4] the tile's stores have read the buffer
  unsigned long long* zconv = bars + 8;     // [4]
  unsigned long long* w1full = bars + 12;   // [2]
  unsigned long long* w1empty = bars + 14;  // [2] both tiles' GEMM 1s have read the stage
  unsigned long long* w2full = bars + 16;   // [2]
  unsigned long long* w2empty = bars + 18;  // [2]
  unsigned long long* ofull = bars + 20;    // [2] output accumulator of a tile is complete
  unsigned long long* oempty = bars + 22;   // [2]
  unsigned long long* gvfull = bars + 24;   // [2] gate | value accumulators of a tile complete
  unsigned long long* hfull = bars + 26;    // [2] hidden slices of a tile stored over them
  unsigned long long* hread = bars + 28;    // [2] GEMM 2 has read them

  const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;   // warp-uniform for the compiler too
  if (threadIdx.x == 0) {
    abort_flag = 0;
    for (int s = 0; s < 4; ++s) {
      mbar_init(&zfull[s], 1);
      mbar_init(&zempty[s], 8);
      mbar_init(&zconv[s], 4);
    }
    for (int s = 0; s < 2; ++s) {
      mbar_init(&gvfull[s], 1);
      mbar_init(&hfull[s], 8);
      mbar_init(&hread[s], 1);
      mbar_init(&ofull[s], 1);
      mbar_init(&oempty[s], 8);
    }
    for (int s = 0; s < TR_WST; ++s) {
      mbar_init(&w1full[s], 1);
      mbar_init(&w1empty[s], 1);
      mbar_init(&w2full[s], 1);
      mbar_init(&w2empty[s], 1);
    }
    mbar_fence_init();
  }
  if (warp == 1) tmem_alloc(&tmem_base_s, 512);
  for (int idx = threadIdx.x; idx < (4 * 2048 + 2048) / 16; idx += TR_THREADS)      // augmentation tiles start as zeros
    *reinterpret_cast<uint4*>(sZx + idx * 16) = make_uint4(0, 0, 0, 0);
  fence_proxy_async_smem();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  pdl_begin();
  const unsigned tmem_base = __shfl_sync(0xffffffffu, tmem_base_s, 0);
  AbortCtx ab{p.status, &abort_flag};
  const long long ntiles = (p.rows + 127) / 128;
  const long long npairs = (ntiles + 1) / 2;
  const int npass = (int)((npairs - blockIdx.x + gridDim.x - 1) / gridDim.x);   // pairs of this CTA

  if (warp == 0) {
    // ------------------------------------------------------------------ producer: lane l issues load l of a group
    auto load_pair = [&](int pass) {          // both state tiles of a pair, into the buffers of its parity
      const int pb = pass & 1;
      if (lane < 2) {
        mbar_wait(&zempty[lane * 2 + pb], ((pass >> 1) & 1) ^ 1, ab);
        mbar_expect_tx(&zfull[lane * 2 + pb], z_stage);
      }
      __syncwarp();
      if (lane < 2 * nslab) {
        const int r = lane / nslab, sl = lane % nslab;
        const long long t = 2 * ((long long)blockIdx.x + (long long)pass * gridDim.x) + r;
        tma_load_2d(sZ + (r * 2 + pb) * z_stage + sl * slab, &p.zmap, &zfull[r * 2 + pb], sl * 64, (int)(t * 128));
      }
    };
    if (npass > 0) load_pair(0);
    unsigned st = 0, ph = 0;
    for (int pass = 0; pass < npass; ++pass)
      for (int q = 0; q < nchunk; ++q) {
        unsigned char* wst = sW1 + st * w1_stage;
        if (lane == 0) {
          mbar_wait(&w1empty[st], ph ^ 1, ab);
          mbar_expect_tx(&w1full[st], w1_stage);
        }
        __syncwarp();
        // rows of either region: 32 gate rows and 32 value rows of the first half, then of the second (rows that an odd
        // half count leaves over are zero or belong to other units; nothing reads their accumulators)
        const int part = lane & 3, row = (part & 1) * hidden + q * TR_CHUNK + (part >> 1) * TR_HALF;
        if (lane < 4 * nslab) {
          const int sl = lane >> 2;
          tma_load_2d(wst + sl * slab + part * TR_HALF * 128, &p.w1map, &w1full[st], sl * 64, row);
        } else if (lane < 4 * nslab + 4) {      // augmentation columns 0-7 of the same rows (region 0 of the table)
          tma_load_2d(wst + w1_bytes + part * TR_HALF * 16, &p.w1xmap, &w1full[st], 0, row);
        }
        // the next pair, into the buffers that the pair before this one has stored from; behind this chunk's weights,
        // because those buffers are given back in the course of this pair
        if (q == nchunk / 2 && pass + 1 < npass) load_pair(pass + 1);
        if (++st == TR_WST) { st = 0; ph ^= 1; }
      }
  } else if (warp == TR_W2PROD) {
    if (lane == 0) {
      unsigned st = 0, ph = 0;
      for (int pass = 0; pass < npass; ++pass)
        for (int h = 0; h < nhalf; ++h) {
          mbar_wait(&w2empty[st], ph ^ 1, ab);
          mbar_expect_tx(&w2full[st], w2_bytes);
          tma_load_2d(sW2 + st * w2_bytes, &p.w2map, &w2full[st], h * TR_HALF, 0);
          if (++st == TR_WST) { st = 0; ph ^= 1; }
        }
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------------ MMA issuer (whole warp, one elected lane)
    // One issuer for both tiles, in the order GEMM 2 and the next GEMM 1 of tile 0, then of tile 1: the tensor pipe takes
    // MMAs as they are issued, so that tile 1's follow tile 0's as a block and one tile's gate stage lies under the
    // other's MMAs.  An issuer per tile interleaves them: both GEMM 1s end together and both gate stages run together.
    const unsigned idesc1 = idesc_f16(128, 2 * TR_CHUNK, 0, 0, FMT_F16, FMT_F16);   // rows x 2 x (32 gate | 32 value)
    const unsigned idesc2 = idesc_f16(128, c, 0, 0, FMT_BF16, FMT_BF16);            // rows x c, A = hidden slice (TMEM)
    const unsigned zero_addr = smem_u32(sZero);
    const int total = npass * nchunk;                      // chunks of this CTA
    int q1 = 0, pass1 = 0, q2 = 0, pass2 = 0;              // chunk and pair of the next GEMM 1 / GEMM 2
    unsigned st1 = 0, ph1 = 0, st2 = 0, ph2 = 0;           // their ring positions
    auto gemm1 = [&](int r) {
      const int zb = r * 2 + (pass1 & 1);
      const unsigned d_gv = tmem_base + r * 128;
      if (q1 == 0) mbar_wait(&zconv[zb], (pass1 >> 1) & 1, ab);
      if (r == 0) mbar_wait(&w1full[st1], ph1, ab);    // tile 1 follows on the same stage
      tc_fence_after();
      const unsigned w_addr = smem_u32(sW1 + st1 * w1_stage);
      const unsigned long long w1_desc = desc_kmajor_sw128(w_addr);
      const unsigned wx_addr = w_addr + w1_bytes;
      const unsigned long long wx_desc = desc_kmajor_nosw(wx_addr, zero_addr - wx_addr, 128);
      const unsigned long long z_desc = desc_kmajor_sw128(smem_u32(sZ + zb * z_stage));
      const unsigned zx_addr = smem_u32(sZx + zb * 2048);
      const unsigned long long zx_desc = desc_kmajor_nosw(zx_addr, zero_addr - zx_addr, 128);
#pragma unroll
      for (int sl = 0; sl < 2; ++sl)
        if (sl < nslab) umma_k4(d_gv, z_desc + sl * (slab >> 4), w1_desc + sl * (slab >> 4), idesc1, sl);
      if (elect_one()) {
        umma_bf16(d_gv, zx_desc, wx_desc, idesc1, 1);   // mean and offset
        tc_commit(&gvfull[r]);
        if (r == 1) tc_commit(&w1empty[st1]);
      }
      __syncwarp();
      if (r == 1) {
        if (++q1 == nchunk) { q1 = 0; ++pass1; }
        if (++st1 == TR_WST) { st1 = 0; ph1 ^= 1; }
      }
    };
    auto gemm2 = [&](int r, unsigned phh) {
      const unsigned d_gv = tmem_base + r * 128;
      const unsigned d_out = tmem_base + 256 + r * 128;
      unsigned st = st2, ph = ph2;
      if (q2 == 0) mbar_wait(&oempty[r], (pass2 & 1) ^ 1, ab);
      mbar_wait(&hfull[r], phh, ab);
      tc_fence_after();
#pragma unroll
      for (int b = 0; b < 2; ++b)
        if (2 * q2 + b < nhalf) {
          if (r == 0) mbar_wait(&w2full[st], ph, ab);
          const unsigned long long w2_desc = tr_desc_sw64(smem_u32(sW2 + st * w2_bytes));
#pragma unroll
          for (int ks = 0; ks < 2; ++ks)
            if (elect_one()) umma_ts(d_out, d_gv + b * 64 + ks * 8, w2_desc + ks * 2, idesc2, (q2 | b | ks) != 0);
          if (r == 1) {
            if (elect_one()) tc_commit(&w2empty[st]);
          }
          if (++st == TR_WST) { st = 0; ph ^= 1; }
        }
      if (elect_one()) tc_commit(&hread[r]);
      if (q2 == nchunk - 1) {
        if (elect_one()) tc_commit(&ofull[r]);
      }
      __syncwarp();
      if (r == 1) {
        st2 = st;
        ph2 = ph;
        if (++q2 == nchunk) { q2 = 0; ++pass2; }
      }
    };
    if (total > 0) {
      gemm1(0);
      gemm1(1);
    }
    for (int g = 0; g < total; ++g)
#pragma unroll
      for (int r = 0; r < 2; ++r) {
        gemm2(r, g & 1);
        if (g + 1 < total) {
          mbar_wait(&hread[r], g & 1, ab);                 // the next chunk's accumulators go over the slices just read
          gemm1(r);
        }
      }
  } else if (warp < 6) {
    // ------------------------------------------------------------------ converters (4 warps, one row per thread)
    const int row = (warp - 2) * 32 + lane;
    for (int pass = 0; pass < npass; ++pass) {
      for (int r = 0; r < 2; ++r) {
        const int zb = r * 2 + (pass & 1);
        mbar_wait(&zfull[zb], (pass >> 1) & 1, ab);
        float sum, sq;
        convert_row_bf16_to_f16(sZ + zb * z_stage, nslab, slab, row, sum, sq);
        const float mean = sum / (float)c;
        const float ve = fmaxf(sq / (float)c - mean * mean, 0.f) + p.eps, rstd = rsqrtf(ve);
        sRstd[zb][row] = rstd;
        const float s = fminf(ve * rstd, 65504.f);        // above that the tile's own fp16 values have overflowed
        const __half sh = __float2half_rn(s);
        const float s1 = s - __half2float(sh);
        const __half sl = __float2half_rn(s1), sr = __float2half_rn((s1 - __half2float(sl)) * 4096.f);
        const __half zh = __float2half_rn(-mean), zl = __float2half_rn(-mean - __half2float(zh));
        __half2 a[4] = {__halves2half2(zh, zl), __halves2half2(zh, sh), __halves2half2(sh, sl), __halves2half2(sr, __float2half_rn(0.f))};
        *reinterpret_cast<uint4*>(sZx + zb * 2048 + row * 16) = *reinterpret_cast<const uint4*>(a);
        fence_proxy_async_smem();
        __syncwarp();
        if (lane == 0) mbar_arrive(&zconv[zb]);
      }
    }
  } else {
    // ------------------------------------------------------------------ gate stage and output stage: eight warps per tile
    // of the pair, in two groups that take the first and the second half of every chunk; a warp covers 32 rows (its TMEM
    // lane quarter).  A half is a chain of TMEM read, 32 units of arithmetic, TMEM write and two barrier hops.
    const int quarter = warp & 3, r = ((warp - 6) >> 2) & 1, b = (warp - 6) >> 3;
    const int row = quarter * 32 + lane;
    const unsigned t_lane = tmem_base + ((unsigned)(quarter * 32) << 16);
    const unsigned t_gv = t_lane + r * 128 + b * 64;
    const int cpg = c / 2;                                   // output channels of this group
    unsigned phg = 0;
    int zgive = -1;                                          // buffer whose store this warp still has to wait for
    auto give_back = [&]() {                                 // off the chain from one pair to the next: after its first chunk
      if (zgive >= 0 && lane == 0) {
        tma_store_wait_read0();
        mbar_arrive(&zempty[zgive]);
      }
      zgive = -1;
    };
    for (int pass = 0; pass < npass; ++pass) {
      const int zb = r * 2 + (pass & 1);
      float rstd = 0.f;
      for (int q = 0; q < nchunk; ++q) {
        mbar_wait(&gvfull[r], phg, ab);                      // GEMM 1 has run, so the converters' statistics are published
        phg ^= 1;
        if (2 * q + b >= nhalf) {
          if (lane == 0) mbar_arrive(&hfull[r]);           // a half that is not there
          continue;
        }
        tc_fence_after();
        if (q == 0) rstd = sRstd[zb][row];
#pragma unroll
        for (int half = 0; half < 2; ++half) {               // 16 units at a time: fewer registers, room for 16 warps
          unsigned rg[16], rv[16];
          tmem_ld16(t_gv + half * 16, rg);
          tmem_ld16(t_gv + 32 + half * 16, rv);
          tmem_ld_wait2(rg, rv);
          unsigned w[8];
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            const float2 r2 = make_float2(rstd, rstd);
            const float2 ga = __fmul2_rn(r2, make_float2(__uint_as_float(rg[4 * e]), __uint_as_float(rg[4 * e + 1])));
            const float2 gb = __fmul2_rn(r2, make_float2(__uint_as_float(rg[4 * e + 2]), __uint_as_float(rg[4 * e + 3])));
            const float2 va = __fmul2_rn(r2, make_float2(__uint_as_float(rv[4 * e]), __uint_as_float(rv[4 * e + 1])));
            const float2 vb = __fmul2_rn(r2, make_float2(__uint_as_float(rv[4 * e + 2]), __uint_as_float(rv[4 * e + 3])));
            // g arrives halved: silu(2 g') = g' tanh(g') + g'
            const float2 ha = __fmul2_rn(__ffma2_rn(ga, make_float2(tr_tanh(ga.x), tr_tanh(ga.y)), ga), va);
            const float2 hb = __fmul2_rn(__ffma2_rn(gb, make_float2(tr_tanh(gb.x), tr_tanh(gb.y)), gb), vb);
            __nv_bfloat162 pa = __floats2bfloat162_rn(ha.x, ha.y), pb = __floats2bfloat162_rn(hb.x, hb.y);
            w[2 * e] = *reinterpret_cast<unsigned*>(&pa);
            w[2 * e + 1] = *reinterpret_cast<unsigned*>(&pb);
          }
          tmem_st8(t_gv + half * 8, w);       // over gate columns that are already in registers
        }
        tmem_st_wait();
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&hfull[r]);
        if (q == 0) give_back();
      }
      // ---- output stage: out + z through the z tile, half of the channels per group, then one TMA store per 64-channel slab
      const long long t = 2 * ((long long)blockIdx.x + (long long)pass * gridDim.x) + r;
      give_back();
      mbar_wait(&ofull[r], pass & 1, ab);
      tc_fence_after();
      unsigned char* zt = sZ + zb * z_stage;
      for (int c0 = b * cpg; c0 < (b + 1) * cpg; c0 += 16) {
        unsigned rr[16];
        tmem_ld16(t_lane + 256 + r * 128 + c0, rr);
        tmem_ld_wait16(rr);
        unsigned char* zp = zt + (c0 >> 6) * slab;
#pragma unroll
        for (int ch = 0; ch < 2; ++ch) {
          uint4* ptr = reinterpret_cast<uint4*>(zp + sw128_off(row, ((c0 & 63) >> 3) + ch));
          const uint4 v = *ptr;
          unsigned wz[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            const float2 zo = unpack_h2(wz[e]);           // the tile holds the exact fp16 copy of z
            __nv_bfloat162 hv = __floats2bfloat162_rn(__uint_as_float(rr[ch * 8 + 2 * e]) + zo.x, __uint_as_float(rr[ch * 8 + 2 * e + 1]) + zo.y);
            wz[e] = *reinterpret_cast<unsigned*>(&hv);
          }
          *ptr = make_uint4(wz[0], wz[1], wz[2], wz[3]);
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&oempty[r]);
      fence_proxy_async_smem();
      // two slabs: each group stores its own; one slab: the two warps of a lane quarter share it and the first stores
      if (nslab == 1) named_bar_sync(1 + r * 4 + quarter, 64);
      else __syncwarp();
      if (lane == 0) {
        const long long r0 = t * 128 + quarter * 32;
        if (r0 < p.rows && (nslab == 2 || b == 0))
          tma_store_2d(&p.zsmap, zt + (nslab == 2 ? b : 0) * slab + quarter * 32 * 128, (nslab == 2 ? b : 0) * 64, (int)r0);
        tma_store_commit();
      }
      zgive = zb;
    }
    if (lane == 0) tma_store_wait_all0();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  abort_linger(ab);
  if (warp == 1) tmem_dealloc(tmem_base, 512);
}

bool fast_transition_supported(int c, int hidden) {
  return (c == 64 || c == 128) && hidden % TR_HALF == 0 && hidden >= TR_HALF && hidden <= 1024;
}

nt_status fast_transition(void* z, const nt_transition_weights* W, float eps, int c, int hidden, long long rows,
                          void* prep, int* status, cudaStream_t st) {
  if (rows > 0x7FFFFF00ll) return NT_ERR_UNSUPPORTED;
  TransPrep tp{};
  nt_status r0 = fast_transition_prep(W, c, hidden, prep, tp, st);
  if (r0 != NT_OK) return r0;
  const int nslab = c / 64;
  const size_t smem = (4 + TR_WST) * (size_t)nslab * 16384 + TR_WST * (2048 + (size_t)c * 2 * TR_HALF) + 5 * 2048 + 1024;
  // the attribute belongs to a (kernel, device) pair: one flag per device
  static bool attr_set_dev[64] = {};
  int attr_dev = 0;
  cudaGetDevice(&attr_dev);
  bool& attr_set = attr_set_dev[attr_dev & 63];
  if (!attr_set) {
    if (cudaFuncSetAttribute(transition_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, TR_SMEM_MAX) != cudaSuccess)
      return cuda_fail("transition smem attribute");
    attr_set = true;
  }
  if (smem > TR_SMEM_MAX) return NT_ERR_UNSUPPORTED;
  TransParams p;
  memset(&p, 0, sizeof(p));
  p.rows = rows;
  p.c = c;
  p.hidden = hidden;
  p.eps = eps;
  p.status = status;
  {
    const unsigned long long dims[2] = {(unsigned long long)c, (unsigned long long)rows};
    const unsigned long long strides[1] = {(unsigned long long)c * 2};
    const unsigned box[2] = {64, 128}, sbox[2] = {64, 32};
    if (!make_tmap_bf16(&p.zmap, z, 2, dims, strides, box)) return cuda_fail("transition z map");
    if (!make_tmap_bf16(&p.zsmap, z, 2, dims, strides, sbox)) return cuda_fail("transition z store map");
    const unsigned long long wdims[2] = {(unsigned long long)c, (unsigned long long)2 * hidden};
    const unsigned wbox[2] = {64, TR_HALF};
    if (!make_tmap_bf16(&p.w1map, tp.w1, 2, wdims, strides, wbox)) return cuda_fail("transition W1 map");
    const unsigned long long xdims[2] = {8, (unsigned long long)2 * tp.rows};
    const unsigned long long xstr[1] = {16};
    const unsigned xbox[2] = {8, TR_HALF};
    if (!make_tmap_16bit(&p.w1xmap, tp.aug, 2, xdims, xstr, xbox, 0)) return cuda_fail("transition augmentation map");
    const unsigned long long w2dims[2] = {(unsigned long long)hidden, (unsigned long long)c};
    const unsigned long long w2str[1] = {(unsigned long long)hidden * 2};
    const unsigned w2box[2] = {TR_HALF, (unsigned)c};
    if (!make_tmap_16bit(&p.w2map, W->W_2, 2, w2dims, w2str, w2box, 64)) return cuda_fail("transition W2 map");
  }
  const long long ntiles = (rows + 127) / 128;
  const long long npairs = (ntiles + 1) / 2;
  const unsigned grid = (unsigned)(npairs < sm_count() ? npairs : sm_count());
  {
    LaunchScope ls("transition", st);
    launch_kernel(transition_kernel, grid, TR_THREADS, smem, st, p);
  }
  return cuda_ok("transition launch");
}

}  // namespace ntp
