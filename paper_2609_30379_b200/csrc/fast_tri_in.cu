// Triangle-update input projection on tcgen05 (fp16 operands, float accumulate):
//   zh = LN(z);  a = sigmoid(zh W_ag^T) * (zh W_ap^T);  b = sigmoid(zh W_bg^T) * (zh W_bp^T)
// written channel-major in fp16 (a[c][i][k], k contiguous) so the contraction's operands are K-major.
//
// The product is computed transposed, D^T[channel][position] = W' z'^T: the accumulator row (TMEM
// lane) is the output channel and the columns are positions, so a thread that reads 32 columns
// holds 32 consecutive k of one channel -- exactly a 64-byte channel-major run, stored with four
// 16-byte stores and no transposition.
//
// LayerNorm is folded completely into the MMA.  With W' = W * gamma (fp16), c1[n] = sum_k W'[n][k],
// c0[n] = sum_k W[n][k] beta[k]:
//   (LN(z) W^T)[n] = (rstd z) . W'[n] + (-mean rstd) c1[n] + c0[n].
// Eight converter warps (two threads per position) rewrite the bf16 z tile as fp16 scaled by the row's rstd and append five
// extra K columns (m_hi, m_lo, m_hi, 1, 1), m = -mean rstd, that meet (c1_hi, c1_hi, c1_lo, c0_hi,
// c0_lo) on the weight side (hi / lo halves keep ~22 bits), so the accumulator already holds the
// normalised projection and the epilogue is sigmoid * value, convert, store.
//
// A tile is 128 packed positions made of four 32-position chunks, each a run of consecutive k inside
// one pair row (s, i) taken from the offset table.  The weights (4 c_h x c_z) stay resident in
// shared memory; the pair state is read exactly once.
#include <cstring>

#include "fast.cuh"
#include "tc_common.cuh"

namespace ntp {

constexpr int TI_CH = 32;                       // positions per chunk
constexpr int TI_CONV_WARPS = 8;
constexpr int TI_EPI_WARP0 = 2 + TI_CONV_WARPS; // first epilogue warp (a multiple of 4 plus 2: see the lane quarters below)
constexpr int TI_THREADS = 64 + 32 * TI_CONV_WARPS + 256;   // producer warp, MMA warp, converter warps, 8 epilogue warps
constexpr int TI_MAXB = 12;

struct TriInParams {
  CUtensorMap zmap[TI_MAXB];               // {c_z, N (k), N (i), 1}, box {64, 32, 1, 1}
  CUtensorMap omap[TI_MAXB];               // outputs {ld (k), N (i), c_h, 2 (a | b)}, box {32, 1, 32, 1}, 64-byte swizzle
  CUtensorMap wmap;                        // {c_z, 4 c_h}, box {64, 128}
  CUtensorMap xmap;                        // augmentation columns {8, 2 * aug_rows}, box {8, 256}, no swizzle
  long long chunk_off[TI_MAXB + 1];
  long long cm_off[TI_MAXB];
  int N[TI_MAXB];
  int B, c_z, c_h, aug_rows;
  int split;                               // CTAs 2 k and 2 k + 1 share tile k, one unit each
  float eps;
  int* status;
  float2* zstats;                          // nullable: (mean, rstd) of every row of z, by packed position, for the output stage
  long long pos_off[TI_MAXB];              // packed position of the first cell of the sample
};

__device__ inline bool ti_decode(const TriInParams& p, long long q, int& s, int& i, int& jc) {
  if (q >= p.chunk_off[p.B]) return false;
  s = 0;
  while (s + 1 < p.B && q >= p.chunk_off[s + 1]) ++s;
  const int cpr = (p.N[s] + TI_CH - 1) / TI_CH;
  // a sample's chunk count N * ceil(N / chunk) is far below 2^32 (N < 2^20 is checked on the host): 32-bit division
  const unsigned r = (unsigned)(q - p.chunk_off[s]);
  i = (int)(r / (unsigned)cpr);
  jc = (int)(r - (unsigned)i * (unsigned)cpr) * TI_CH;
  return true;
}

__device__ inline float tanh_fast(float x) {
  float t;
  asm("tanh.approx.f32 %0, %1;\n" : "=f"(t) : "f"(x));
  return t;
}

__global__ void __launch_bounds__(TI_THREADS, 1) tri_in_kernel(const __grid_constant__ TriInParams p) {
  extern __shared__ unsigned char smem_raw[];
  __shared__ __align__(8) unsigned long long bars[11];
  __shared__ unsigned tmem_base_s;
  __shared__ int abort_flag;
  __shared__ int4 tinfo[8][4];             // ring of decoded chunks {s, i, k0, valid} per tile, written by the producer up to
                                           // five tiles ahead of the epilogue that reads it
  unsigned char* smem = smem_raw + ((1024 - (smem_u32(smem_raw) & 1023)) & 1023);
  const int c_z = p.c_z, c_h = p.c_h;
  const int nslab = c_z / 64;
  const int wrows = 4 * c_h;
  const int w_slab_bytes = wrows * 128;            // one 64-channel slab of all weight rows
  const int w_bytes = nslab * w_slab_bytes;
  const int wx_region = wrows * 16;                // one 8-column region of the weight augmentation
  const int z_slab_bytes = 128 * 128;
  const int z_stage_bytes = nslab * z_slab_bytes;
  const int zx_region = 128 * 16;                  // one 8-column region of the activation augmentation
  unsigned char* sW = smem;
  unsigned char* sWx = sW + w_bytes;               // [wrows][8] fp16, no swizzle: augmentation columns 0-7 of the weights
  unsigned char* sZ = sWx + wx_region;             // 2 stages of the z tile
  unsigned char* sZx = sZ + 2 * z_stage_bytes;     // 2 stages x [128][8] fp16: augmentation columns 0-7 of the activations
  unsigned char* sZero = sZx + 2 * zx_region;      // [128][8] zeros: augmentation columns 8-15 of either operand
  unsigned char* sOut = sZero + zx_region;         // per epilogue warp: 2 x [32 channels][16 positions] fp16 staged for TMA stores
  unsigned long long* afull = bars;        // [2] TMA landed
  unsigned long long* aempty = bars + 2;   // [2] MMAs that read the stage are done
  unsigned long long* tfull = bars + 4;    // [2] accumulator buffer ready
  unsigned long long* tempty = bars + 6;   // [2] accumulator buffer drained
  unsigned long long* wfull = bars + 8;
  unsigned long long* aconv = bars + 9;    // [2] tile normalised / converted, augmentation written

  const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;   // warp-uniform for the compiler too
  if (threadIdx.x == 0) {
    abort_flag = 0;
    for (int s = 0; s < 2; ++s) {
      mbar_init(&afull[s], 1);
      mbar_init(&aempty[s], 1);
      mbar_init(&tfull[s], 1);
      mbar_init(&tempty[s], 8);
      mbar_init(&aconv[s], TI_CONV_WARPS);
    }
    mbar_init(wfull, 1);
    mbar_fence_init();
  }
  if (warp == 1) tmem_alloc(&tmem_base_s, 512);
  // the second 8-column region of the activation augmentation is always zero
  for (int idx = threadIdx.x; idx < zx_region / 16; idx += TI_THREADS)
    *reinterpret_cast<uint4*>(sZero + idx * 16) = make_uint4(0, 0, 0, 0);
  fence_proxy_async_smem();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  pdl_begin();
  const unsigned tmem_base = __shfl_sync(0xffffffffu, tmem_base_s, 0);
  AbortCtx ab{p.status, &abort_flag};
  const long long nchunks = p.chunk_off[p.B];
  const long long ntiles = (nchunks + 3) / 4;
  const int nunits = c_h == 128 ? 2 : 1;           // accumulator units per tile: (gate rows | value rows) of 128 each
  // split: a CTA takes one unit of a tile and fetches only that unit's weights
  const int u0 = p.split ? (int)(blockIdx.x & 1) : 0, u1 = p.split ? u0 + 1 : nunits;
  const long long t0 = p.split ? blockIdx.x >> 1 : blockIdx.x, tstep = p.split ? gridDim.x >> 1 : gridDim.x;

  if (warp == 0) {
    // ------------------------------------------------------------------ producer (lane q decodes and loads chunk q)
    if (lane == 0) {
      mbar_expect_tx(wfull, (u1 - u0) * 256 * (nslab * 128 + 16));
      for (int sl = 0; sl < nslab; ++sl)
        for (int rb = 2 * u0; rb < 2 * u1; ++rb)
          tma_load_2d(sW + sl * w_slab_bytes + rb * 128 * 128, &p.wmap, wfull, sl * 64, rb * 128);
      for (int rb = u0; rb < u1; ++rb) tma_load_2d(sWx + rb * 256 * 16, &p.xmap, wfull, 0, rb * 256);
    }
    int stage = 0, tn = 0;
    unsigned phase = 0;
    for (long long t = t0; t < ntiles; t += tstep, ++tn) {
      int s = 0, i = 0, jc = 0;
      bool valid = false;
      if (lane < 4) {
        valid = ti_decode(p, 4 * t + lane, s, i, jc);
        tinfo[tn & 7][lane] = make_int4(s, i, jc, valid ? 1 : 0);
      }
      __syncwarp();
      if (lane == 0) {
        const long long left = nchunks - 4 * t;
        const int nvalid = left < 4 ? (int)left : 4;
        mbar_wait(&aempty[stage], phase ^ 1, ab);
        mbar_expect_tx(&afull[stage], nvalid * nslab * TI_CH * 128);
      }
      __syncwarp();
      if (valid)
        for (int sl = 0; sl < nslab; ++sl)
          tma_load_4d(sZ + stage * z_stage_bytes + sl * z_slab_bytes + lane * TI_CH * 128, &p.zmap[s], &afull[stage],
                      sl * 64, jc, i, 0);
      if (++stage == 2) { stage = 0; phase ^= 1; }
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------------ MMA issuer: the whole warp runs the loop and
    // one elected lane issues, with descriptors derived from per-CTA bases by adding constants
    mbar_wait(wfull, 0, ab);
    int stage = 0;
    unsigned phase = 0, tph0 = 0, tph1 = 0;
    unsigned unit = 0;
    const unsigned idesc = idesc_f16(128, 128, 0, 0, FMT_F16, FMT_F16);   // M = 128 channels, N = 128 positions
    const unsigned long long w_desc = desc_kmajor_sw128(smem_u32(sW));
    const unsigned wx_addr = smem_u32(sWx), zero_addr = smem_u32(sZero);   // columns 8-15 of both operands: the zero region
    const unsigned w_slab16 = (unsigned)w_slab_bytes >> 4, z_slab16 = (unsigned)z_slab_bytes >> 4;
    for (long long t = t0; t < ntiles; t += tstep) {
      mbar_wait(&aconv[stage], phase, ab);
      tc_fence_after();
      const unsigned long long z_desc = desc_kmajor_sw128(smem_u32(sZ + stage * z_stage_bytes));
      const unsigned zx_addr = smem_u32(sZx + stage * zx_region);
      const unsigned long long zx_desc = desc_kmajor_nosw(zx_addr, zero_addr - zx_addr, 128);
      for (int u = u0; u < u1; ++u, ++unit) {
        const unsigned buf = unit & 1;
        if (buf == 0) { mbar_wait(&tempty[0], tph0 ^ 1, ab); tph0 ^= 1; }
        else { mbar_wait(&tempty[1], tph1 ^ 1, ab); tph1 ^= 1; }
        tc_fence_after();
#pragma unroll
        for (int part = 0; part < 2; ++part) {                 // 0 = gate rows, 1 = value rows
          const unsigned row16 = (unsigned)(u * 256 + part * 128) * 8;        // row offset in units of 16 bytes (128-byte rows)
          const unsigned d_tmem = tmem_base + buf * 256 + part * 128;
#pragma unroll
          for (int sl = 0; sl < 2; ++sl) {
            if (sl < nslab) umma_k4(d_tmem, w_desc + (sl * w_slab16 + row16), z_desc + sl * z_slab16, idesc, sl);
          }
          // augmentation K step: c1 / c0 columns against the (-mean rstd, 1) columns (16-byte rows)
          const unsigned wxa = wx_addr + (unsigned)(u * 256 + part * 128) * 16;
          if (elect_one()) umma_bf16(d_tmem, desc_kmajor_nosw(wxa, zero_addr - wxa, 128), zx_desc, idesc, 1);
        }
        if (elect_one()) tc_commit(&tfull[buf]);
        __syncwarp();
      }
      if (elect_one()) tc_commit(&aempty[stage]);
      __syncwarp();
      if (++stage == 2) { stage = 0; phase ^= 1; }
    }
  } else if (warp >= 2 && warp < TI_EPI_WARP0) {
    // ------------------------------------------------------------------ converters: two threads per position, each
    // owning four of the eight 16-byte chunks of every 64-channel slab
    const int row = (warp - 2) * 16 + (lane >> 1), hf = lane & 1;
    int stage = 0, tn = 0;
    unsigned phase = 0;
    for (long long t = t0; t < ntiles; t += tstep, ++tn) {
      mbar_wait(&afull[stage], phase, ab);
      unsigned char* tile = sZ + stage * z_stage_bytes;
      uint4 raw[2][4];
#pragma unroll
      for (int sl = 0; sl < 2; ++sl)
#pragma unroll
        for (int j = 0; j < 4; ++j)
          raw[sl][j] = sl < nslab ? *reinterpret_cast<const uint4*>(tile + sl * z_slab_bytes + sw128_off(row, hf * 4 + j))
                                  : make_uint4(0, 0, 0, 0);
      float s4[4] = {0.f, 0.f, 0.f, 0.f}, q4[4] = {0.f, 0.f, 0.f, 0.f};   // four independent chains
#pragma unroll
      for (int sl = 0; sl < 2; ++sl)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const unsigned w[4] = {raw[sl][j].x, raw[sl][j].y, raw[sl][j].z, raw[sl][j].w};
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            const float lo = __uint_as_float(w[e] << 16), hi = __uint_as_float(w[e] & 0xffff0000u);
            s4[e] += lo + hi;
            q4[e] = fmaf(lo, lo, q4[e]);
            q4[e] = fmaf(hi, hi, q4[e]);
          }
        }
      float sum = (s4[0] + s4[1]) + (s4[2] + s4[3]), sq = (q4[0] + q4[1]) + (q4[2] + q4[3]);
      sum += __shfl_xor_sync(0xffffffffu, sum, 1);
      sq += __shfl_xor_sync(0xffffffffu, sq, 1);
      const float mean = sum / (float)c_z;
      const float rstd = rsqrtf(fmaxf(sq / (float)c_z - mean * mean, 0.f) + p.eps);
#pragma unroll
      for (int sl = 0; sl < 2; ++sl)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          if (sl < nslab) {
            unsigned w[4] = {raw[sl][j].x, raw[sl][j].y, raw[sl][j].z, raw[sl][j].w};
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              __half2 h =
                  __floats2half2_rn(__uint_as_float(w[e] << 16) * rstd, __uint_as_float(w[e] & 0xffff0000u) * rstd);
              w[e] = *reinterpret_cast<unsigned*>(&h);
            }
            *reinterpret_cast<uint4*>(tile + sl * z_slab_bytes + sw128_off(row, hf * 4 + j)) =
                make_uint4(w[0], w[1], w[2], w[3]);
          }
        }
      if (p.zstats && hf == 0 && u0 == 0) {             // the output stage normalises the same rows: hand the statistics over
        const int4 info = tinfo[tn & 7][row / TI_CH];
        const int j = info.z + (row % TI_CH);
        if (info.w && j < p.N[info.x])
          p.zstats[p.pos_off[info.x] + (long long)info.y * p.N[info.x] + j] = make_float2(mean, rstd);
      }
      if (hf == 0) {
        const float mm = -mean * rstd;
        const __half mh = __float2half_rn(mm), ml = __float2half_rn(mm - __half2float(mh));
        const __half one = __float2half_rn(1.0f), zero = __float2half_rn(0.0f);
        __half2 p0 = __halves2half2(mh, ml), p1 = __halves2half2(mh, one), p2 = __halves2half2(one, zero),
                p3 = __halves2half2(zero, zero);
        *reinterpret_cast<uint4*>(sZx + stage * zx_region + row * 16) =
            make_uint4(*reinterpret_cast<unsigned*>(&p0), *reinterpret_cast<unsigned*>(&p1),
                       *reinterpret_cast<unsigned*>(&p2), *reinterpret_cast<unsigned*>(&p3));
      }
      fence_proxy_async_smem();
      __syncwarp();
      if (lane == 0) mbar_arrive(&aconv[stage]);
      if (++stage == 2) { stage = 0; phase ^= 1; }
    }
  } else if (warp >= TI_EPI_WARP0) {
    // ------------------------------------------------------------------ epilogue (8 warps)
    const int quarter = warp & 3;                  // TMEM lane quarter = 32 output channels
    const int half = (warp - TI_EPI_WARP0) >> 2;   // which two of the tile's four chunks this warp stores
    const __half2 hmax2 = __float2half2_rn(65504.f), hmin2 = __float2half2_rn(-65504.f);
    unsigned tph[2] = {0, 0};
    long long unit = 0;
    int tn = 0;
    for (long long t = t0; t < ntiles; t += tstep, ++tn) {
      for (int u = u0; u < u1; ++u, ++unit) {
        const int buf = (int)(unit & 1);
        mbar_wait(&tfull[buf], tph[buf], ab);
        tph[buf] ^= 1;
        tc_fence_after();
        // c_h = 128: unit 0 -> a, unit 1 -> b, channel = accumulator row; c_h = 64: rows 0-63 -> a, 64-127 -> b
        const int which = c_h == 128 ? u : (quarter >> 1);
        const int ch0 = c_h == 128 ? quarter * 32 : (quarter & 1) * 32;          // first channel of this warp
        unsigned char* stg0 = sOut + (warp - TI_EPI_WARP0) * 2048;
        const unsigned taddr = tmem_base + ((unsigned)(quarter * 32) << 16) + buf * 256 + half * 64;
        // four steps of 16 positions; the TMEM loads of step k + 1 are in flight while step k is computed.  A step's
        // 32 channels x 16 positions go through a 1 KB staging tile and out with one TMA store (runs of 32 bytes per
        // channel row, clipped at the row end), which keeps the scattered writes off the load / store units.
        unsigned rg[2][16], rv[2][16], w[2][8];
        tmem_ld16(taddr, rg[0]);
        tmem_ld16(taddr + 128, rv[0]);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          tmem_ld_wait2(rg[k & 1], rv[k & 1]);
          if (k < 3) {
            tmem_ld16(taddr + (k + 1) * 16, rg[(k + 1) & 1]);
            tmem_ld16(taddr + 128 + (k + 1) * 16, rv[(k + 1) & 1]);
          }
          const int4 info = tinfo[tn & 7][half * 2 + (k >> 1)];
#pragma unroll
          for (int e = 0; e < 8; ++e) {
            // the gate and value weight rows were folded times 1/2, so with g' = g / 2, v' = v / 2:
            // sigmoid(g) * v = (tanh(g') + 1) * v' = fma(v', tanh(g'), v')
            const float h0 = __uint_as_float(rv[k & 1][2 * e]), h1 = __uint_as_float(rv[k & 1][2 * e + 1]);
            const float v0 = fmaf(h0, tanh_fast(__uint_as_float(rg[k & 1][2 * e])), h0);
            const float v1 = fmaf(h1, tanh_fast(__uint_as_float(rg[k & 1][2 * e + 1])), h1);
            __half2 h = __floats2half2_rn(v0, v1);          // overflow gives inf, clamped below
            h = __hmax2(__hmin2(h, hmax2), hmin2);
            w[k & 1][e] = *reinterpret_cast<unsigned*>(&h);
          }
          // a chunk (two steps, 32 positions) is staged as 32 channel rows of 64 bytes and leaves with one TMA store:
          // the store engine's cost is per row, so rows should be as long as the tile geometry allows
          if (k & 1) {
            // The store of the chunk before has had two steps of arithmetic to read the staging tile.  (Waiting after the first
            // step: 83.3 us per launch at eight samples of about 215 positions, 76.9 so.)
            if (lane == 0) tma_store_wait_read0();
            __syncwarp();
            // 64-byte swizzle of the store map: the 16-byte pieces of a row are XOR-ed with the row's bits 1-2, so eight
            // lanes cover all banks
            unsigned char* rowp = stg0 + lane * 64;
            const int sw = (lane >> 1) & 3;
#pragma unroll
            for (int e = 0; e < 4; ++e)
              *reinterpret_cast<uint4*>(rowp + ((e ^ sw) << 4)) =
                  make_uint4(w[e >> 1][(e & 1) * 4], w[e >> 1][(e & 1) * 4 + 1], w[e >> 1][(e & 1) * 4 + 2], w[e >> 1][(e & 1) * 4 + 3]);
            fence_proxy_async_smem();
            __syncwarp();
            if (lane == 0 && info.w) {
              if (info.z < round_up8(p.N[info.x])) tma_store_4d(&p.omap[info.x], stg0, info.z, info.y, ch0, which);
              tma_store_commit();
            }
          }
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&tempty[buf]);
      }
    }
    if (lane == 0) tma_store_wait_all0();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  abort_linger(ab);
  if (warp == 1) tmem_dealloc(tmem_base, 512);
}

bool fast_tri_in_supported(int c_z, int c_h) { return (c_z == 64 || c_z == 128) && (c_h == 64 || c_h == 128); }

nt_status fast_tri_in(const void* z, const TriPrep& tp, float eps, int c_z, int c_h, void* a, void* b,
                      const BatchMeta& m, int* status, cudaStream_t st, float2* zstats) {
  const int nslab = c_z / 64;
  const int wrows = 4 * c_h;
  const size_t smem = (size_t)nslab * wrows * 128 + (size_t)wrows * 16 + 2 * (size_t)nslab * 128 * 128 +
                      3 * (size_t)128 * 16 + 16 * 1024 + 1024;
  if (((const char*)b - (const char*)a) % 16 != 0 || b <= a) return NT_ERR_UNSUPPORTED;   // a | b form one 4-D tensor
  // the attribute belongs to a (kernel, device) pair: one flag per device
  static bool attr_set_dev[64] = {};
  int attr_dev = 0;
  cudaGetDevice(&attr_dev);
  bool& attr_set = attr_set_dev[attr_dev & 63];
  if (!attr_set) {
    if (cudaFuncSetAttribute(tri_in_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 231424) != cudaSuccess)
      return cuda_fail("tri_in smem attribute");
    attr_set = true;
  }
  for (int g0 = 0; g0 < m.B; g0 += TI_MAXB) {
    TriInParams p;
    memset(&p, 0, sizeof(p));
    p.B = m.B - g0 < TI_MAXB ? m.B - g0 : TI_MAXB;
    p.c_z = c_z;
    p.c_h = c_h;
    p.aug_rows = tp.aug1_rows;
    p.eps = eps;
    p.status = status;
    {
      const unsigned long long dims[2] = {(unsigned long long)c_z, (unsigned long long)wrows};
      const unsigned long long strides[1] = {(unsigned long long)c_z * 2};
      const unsigned box[2] = {64, 128};
      if (!make_tmap_bf16(&p.wmap, tp.w1, 2, dims, strides, box)) return cuda_fail("tri_in weight map");
      const unsigned long long xdims[2] = {8, (unsigned long long)2 * tp.aug1_rows};
      const unsigned long long xstr[1] = {16};
      const unsigned xbox[2] = {8, 256};
      if (!make_tmap_16bit(&p.xmap, tp.aug1, 2, xdims, xstr, xbox, 0)) return cuda_fail("tri_in augmentation map");
    }
    p.zstats = zstats;
    p.chunk_off[0] = 0;
    for (int l = 0; l < TI_MAXB; ++l) {
      const int N = l < p.B ? m.N[g0 + l] : 0;
      p.N[l] = N;
      p.cm_off[l] = l < p.B ? m.cm_off[g0 + l] : 0;
      p.pos_off[l] = l < p.B ? m.pair_off[g0 + l] : 0;
      p.chunk_off[l + 1] = p.chunk_off[l] + (long long)N * ((N + TI_CH - 1) / TI_CH);
      if (N > 0) {
        const unsigned long long dims[4] = {(unsigned long long)c_z, (unsigned long long)N, (unsigned long long)N, 1};
        const unsigned long long strides[3] = {(unsigned long long)c_z * 2, (unsigned long long)N * c_z * 2,
                                               (unsigned long long)N * N * c_z * 2};
        const unsigned box[4] = {64, TI_CH, 1, 1};
        const char* base = (const char*)z + (size_t)m.pair_off[g0 + l] * c_z * 2;
        if (!make_tmap_bf16(&p.zmap[l], base, 4, dims, strides, box)) return cuda_fail("tri_in z map");
        const int ld = round_up8(N);
        const unsigned long long odims[4] = {(unsigned long long)ld, (unsigned long long)N, (unsigned long long)c_h, 2};
        const unsigned long long ostr[3] = {(unsigned long long)ld * 2, (unsigned long long)N * ld * 2,
                                            (unsigned long long)((const char*)b - (const char*)a)};
        const unsigned obox[4] = {32, 1, 32, 1};
        const char* obase = (const char*)a + (size_t)c_h * m.cm_off[g0 + l] * 2;
        if (!make_tmap_16bit(&p.omap[l], obase, 4, odims, ostr, obox, 64)) return cuda_fail("tri_in output map");
      }
    }
    const long long ntiles = (p.chunk_off[p.B] + 3) / 4;
    if (ntiles == 0) continue;
    // Few tiles leave most SMs idle and the launch is one tile's latency: 128 KB of weights, then two units one after the other.
    // With an SM for either unit both parts halve (the line is where a CTA would have to come back for a second tile).
    p.split = c_h == 128 && 2 * ntiles <= sm_count();
    const long long nwork = p.split ? 2 * ntiles : ntiles;
    const unsigned grid = (unsigned)(nwork < sm_count() ? nwork : sm_count());
    {
      LaunchScope ls("tri_in", st);
      launch_kernel(tri_in_kernel, grid, TI_THREADS, smem, st, p);
    }
    if (cudaPeekAtLastError() != cudaSuccess) return cuda_fail("tri_in launch");
  }
  return NT_OK;
}

}  // namespace ntp
