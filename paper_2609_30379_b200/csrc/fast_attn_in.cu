// Attention input projection on tcgen05 (bf16, float accumulate):
//   zh = LN(z);  q, k, v = zh W_{q,k,v}^T  (row-major [T2, H d]);  bias = zh W_b^T  (head-major, channel-major)
// LayerNorm is folded into the weights (see fast_tri_in.cu).  The gate sigmoid(zh W_g^T) is not
// produced here: the output projection recomputes it from z, which saves a [T2, H d] write and read.
//
// Tiles are 128 consecutive packed positions (the outputs are row-major, so no row alignment is
// needed); the (3 H d + 16) x c_z weights stay resident in shared memory.  Accumulator units per
// tile: [q | k], [v], [bias padded to 16 columns].  Eight epilogue warps apply the LayerNorm
// correction, stage each output as swizzled 64-channel panels and TMA-store them; the bias values
// are scattered per head as 2-byte stores that coalesce across the warp (consecutive k of a row).
#include <cstring>

#include "fast.cuh"
#include "tc_common.cuh"

namespace ntp {

constexpr int AI_CONV_WARPS = 8;
constexpr int AI_EPI_WARP0 = 2 + AI_CONV_WARPS;
constexpr int AI_THREADS = 64 + 32 * AI_CONV_WARPS + 256;   // producer, MMA, 8 converter warps, 8 epilogue warps
constexpr int AI_MAXB = 16;

struct AttnInParams {
  CUtensorMap zmap;              // {c, rows}, box {64, 128}
  CUtensorMap wmap;              // {c, 3 Hd + 16}, box {64, 128} (q, k, v rows)
  CUtensorMap wbmap;             // same tensor, box {64, 16} (bias rows)
  CUtensorMap omap[3];           // q, k, v: {Hd, rows}, box {64, 32}: one epilogue warp's rows
  long long pair_off[AI_MAXB + 1];   // relative to the first position of the group
  long long cm_off[AI_MAXB];
  int N[AI_MAXB];
  int B, c, H, Hd;
  long long rows;                // positions in the group
  float eps;
  CUtensorMap xmap;              // augmentation columns {8, 2 * aug_rows}, box {8, 16}, no swizzle
  int aug_rows;
  __nv_bfloat16* bias;           // nullable
  int* status;
  float2* zstats;                // nullable: (mean, rstd) of every row of the group, for the output stage
  long long bias_elems;          // elements of the bias buffer the group may touch (checked build)
  int bias_tr_above;             // samples longer than this get their bias planes transposed ([h][j][i]: column-wise attention)
};

template <bool SPLIT>   // a parameter of the code: with the units of a tile known, the loops over them keep their constants
__global__ void __launch_bounds__(AI_THREADS, 1) attn_in_kernel(const __grid_constant__ AttnInParams p) {
  extern __shared__ unsigned char smem_raw[];
  __shared__ __align__(8) unsigned long long bars[11];
  __shared__ unsigned tmem_base_s;
  __shared__ int abort_flag;
  unsigned char* smem = smem_raw + ((1024 - (smem_u32(smem_raw) & 1023)) & 1023);
  const int c = p.c, Hd = p.Hd;
  const int nslab = c / 64;
  const int wrows = 3 * Hd + 16;
  const int w_slab = wrows * 128;
  const int a_slab = 128 * 128;
  const int a_stage = nslab * a_slab;
  const int npanel = Hd / 64 > 0 ? Hd / 64 : 1;
  const int wx_region = wrows * 16;                      // one 8-column region of the weight augmentation
  const int zx_region = 128 * 16;                        // one 8-column region of the activation augmentation
  unsigned char* sW = smem;
  unsigned char* sA = sW + nslab * w_slab;               // 2 stages
  unsigned char* sOut = sA + 2 * a_stage;                // npanel panels of [128][64]
  unsigned char* sWx = sOut + npanel * a_slab;           // [2 regions][wrows][8] fp16, no swizzle
  unsigned char* sAx = sWx + 2 * wx_region;              // 2 stages x [2 regions][128][8] fp16
  unsigned long long* afull = bars;
  unsigned long long* aempty = bars + 2;
  unsigned long long* tfull = bars + 4;
  unsigned long long* tempty = bars + 6;
  unsigned long long* wfull = bars + 8;
  unsigned long long* aconv = bars + 9;    // [2]

  const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;   // warp-uniform for the compiler too
  if (threadIdx.x == 0) {
    abort_flag = 0;
    for (int s = 0; s < 2; ++s) {
      mbar_init(&afull[s], 1);
      mbar_init(&aempty[s], 1);
      mbar_init(&tfull[s], 1);
      mbar_init(&tempty[s], 8);
      mbar_init(&aconv[s], AI_CONV_WARPS);
    }
    mbar_init(wfull, 1);
    mbar_fence_init();
  }
  if (warp == 1) tmem_alloc(&tmem_base_s, 512);
  // the second 8-column region of the activation augmentation is always zero
  for (int idx = threadIdx.x; idx < 2 * zx_region / 16; idx += AI_THREADS) {
    const int st = idx / (zx_region / 16), r = idx % (zx_region / 16);
    *reinterpret_cast<uint4*>(sAx + st * 2 * zx_region + zx_region + r * 16) = make_uint4(0, 0, 0, 0);
  }
  fence_proxy_async_smem();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  pdl_begin();
  const unsigned tmem_base = __shfl_sync(0xffffffffu, tmem_base_s, 0);
  AbortCtx ab{p.status, &abort_flag};
  const long long ntiles = (p.rows + 127) / 128;
  const int nunits = p.bias ? 3 : 2;
  // split: a CTA takes q | k of a tile or v and the bias, and fetches only those weights
  const int u0 = SPLIT ? (int)(blockIdx.x & 1) : 0, u1 = SPLIT && u0 == 0 ? 1 : nunits;
  const long long t0 = SPLIT ? blockIdx.x >> 1 : blockIdx.x, tstep = SPLIT ? gridDim.x >> 1 : gridDim.x;
  // unit u: weight row offset and accumulator width
  const int u_row[3] = {0, 2 * Hd, 3 * Hd};
  const int u_n[3] = {2 * Hd, Hd, 16};

  if (warp == 0 && lane == 0) {
    // ------------------------------------------------------------------ producer
    const int row0 = u0 == 0 ? 0 : 2 * Hd, row1 = u1 == 1 ? 2 * Hd : wrows;      // weight rows of this CTA's units
    mbar_expect_tx(wfull, (row1 - row0) * (nslab * 128 + 2 * 16));
    for (int reg = 0; reg < 2; ++reg)
      for (int r16 = row0; r16 < row1; r16 += 16)
        tma_load_2d(sWx + reg * wx_region + r16 * 16, &p.xmap, wfull, 0, reg * p.aug_rows + r16);
    for (int sl = 0; sl < nslab; ++sl)
      for (int r = row0; r < row1;) {
        const bool big = r + 128 <= 3 * Hd && r + 128 <= row1;   // 128-row boxes where they fit, 16-row boxes for the rest
        tma_load_2d(sW + sl * w_slab + r * 128, big ? &p.wmap : &p.wbmap, wfull, sl * 64, r);
        r += big ? 128 : 16;
      }
    int stage = 0;
    unsigned phase = 0;
    for (long long t = t0; t < ntiles; t += tstep) {
      mbar_wait(&aempty[stage], phase ^ 1, ab);
      mbar_expect_tx(&afull[stage], a_stage);
      for (int sl = 0; sl < nslab; ++sl)
        tma_load_2d(sA + stage * a_stage + sl * a_slab, &p.zmap, &afull[stage], sl * 64, (int)(t * 128));
      if (++stage == 2) { stage = 0; phase ^= 1; }
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------------ MMA issuer (whole warp, one elected lane issues)
    mbar_wait(wfull, 0, ab);
    int stage = 0;
    unsigned phase = 0, tph0 = 0, tph1 = 0;
    unsigned unit = 0;
    const unsigned long long w_desc = desc_kmajor_sw128(smem_u32(sW));
    const unsigned w16 = (unsigned)w_slab >> 4, a16 = (unsigned)a_slab >> 4;
    const unsigned long long wx_desc = desc_kmajor_nosw(smem_u32(sWx), wx_region, 128);
    for (long long t = t0; t < ntiles; t += tstep) {
      mbar_wait(&aconv[stage], phase, ab);
      tc_fence_after();
      const unsigned long long a_desc = desc_kmajor_sw128(smem_u32(sA + stage * a_stage));
      const unsigned long long ax_desc = desc_kmajor_nosw(smem_u32(sAx + stage * 2 * zx_region), zx_region, 128);
      for (int u = u0; u < u1; ++u, ++unit) {
        const unsigned buf = unit & 1;
        if (buf == 0) { mbar_wait(&tempty[0], tph0 ^ 1, ab); tph0 ^= 1; }
        else { mbar_wait(&tempty[1], tph1 ^ 1, ab); tph1 ^= 1; }
        tc_fence_after();
        const unsigned idesc = idesc_f16(128, u_n[u], 0, 0, FMT_F16, FMT_F16);   // z tile converted to fp16, folded weights fp16
        const unsigned d_tmem = tmem_base + buf * 256;
        const unsigned row16 = (unsigned)u_row[u] * 8;                           // 128-byte rows in units of 16 bytes
#pragma unroll
        for (int sl = 0; sl < 2; ++sl)
          if (sl < nslab) {
            umma_k4(d_tmem, a_desc + sl * a16, w_desc + (sl * w16 + row16), idesc, sl);
          }
        // augmentation K step: (-mean rstd, 1) columns against the c1 / c0 columns (16-byte rows)
        if (elect_one()) umma_bf16(d_tmem, ax_desc, wx_desc + (unsigned)u_row[u], idesc, 1);
        if (elect_one()) tc_commit(&tfull[buf]);
        __syncwarp();
      }
      if (elect_one()) tc_commit(&aempty[stage]);
      __syncwarp();
      if (++stage == 2) { stage = 0; phase ^= 1; }
    }
  } else if (warp >= 2 && warp < AI_EPI_WARP0) {
    // ------------------------------------------------------------------ converters (8 warps, two threads per row):
    // the tile becomes fp16 scaled by the row's rstd, with the augmentation columns that complete the LayerNorm
    const int row = (warp - 2) * 16 + (lane >> 1), hf = lane & 1;
    int stage = 0;
    unsigned phase = 0;
    for (long long t = t0; t < ntiles; t += tstep) {
      mbar_wait(&afull[stage], phase, ab);
      convert_row_ln_fp16(sA + stage * a_stage, nslab, a_slab, sAx + stage * 2 * zx_region + row * 16, row, hf, c, p.eps,
                          p.zstats && u0 == 0 && t * 128 + row < p.rows ? p.zstats + t * 128 + row : nullptr);
      fence_proxy_async_smem();
      __syncwarp();
      if (lane == 0) mbar_arrive(&aconv[stage]);
      if (++stage == 2) { stage = 0; phase ^= 1; }
    }
  } else if (warp >= AI_EPI_WARP0) {
    // ------------------------------------------------------------------ epilogue (8 warps): the accumulators already hold
    // the normalised projections
    const int quarter = warp & 3;
    const int half = (warp - AI_EPI_WARP0) >> 2;
    const int row = quarter * 32 + lane;
    const int cpw = Hd / 2;                         // channels of one output handled by this warp
    unsigned tph[2] = {0, 0};
    long long unit = 0;
    bool store_pending = false;
    int tn = 0;
    for (long long t = t0; t < ntiles; t += tstep, ++tn) {
      for (int u = u0; u < u1; ++u, ++unit) {
        const int buf = (int)(unit & 1);
        mbar_wait(&tfull[buf], tph[buf], ab);
        tph[buf] ^= 1;
        tc_fence_after();
        const unsigned taddr = tmem_base + ((unsigned)(quarter * 32) << 16) + buf * 256;
        if (u < 2) {
          const int nout = u == 0 ? 2 : 1;
          for (int oi = 0; oi < nout; ++oi) {
            const int o = u == 0 ? oi : 2;          // 0 = q, 1 = k, 2 = v
            // Every warp stores its own 32 positions x 64 channels as soon as it has written them (Hd = 64: the two
            // warps of a lane quarter share the slab and meet at a barrier of their own), so no store waits for the
            // other warps and only the warp's own previous store has to have read its corner of the panels.
            const bool storer = lane == 0 && (npanel == 2 || half == 0);
            // The output before has the time of this one's loads and conversions to leave the panels.  (Waiting first: 83 us
            // per launch at eight samples of about 215 positions, 77 so; line stores from registers instead of the copy engine: 86.)
            unsigned w[32];
#pragma unroll
            for (int ci = 0; ci < 2; ++ci)
              if (ci * 32 < cpw) {
                unsigned r[32];
                tmem_ld32(taddr + oi * Hd + half * cpw + ci * 32, r);
                tmem_ld_wait();
#pragma unroll
                for (int e = 0; e < 16; ++e) {
                  __nv_bfloat162 hh = __floats2bfloat162_rn(__uint_as_float(r[2 * e]), __uint_as_float(r[2 * e + 1]));
                  w[ci * 16 + e] = *reinterpret_cast<unsigned*>(&hh);
                }
              }
            if (oi == nout - 1) {                           // the accumulator has been read
              tc_fence_before();
              __syncwarp();
              if (lane == 0) mbar_arrive(&tempty[buf]);
            }
            if (store_pending) {
              if (storer) tma_store_wait_read0();
              if (npanel == 1) named_bar_sync(2 + quarter, 64);
              else __syncwarp();
            }
#pragma unroll
            for (int ci = 0; ci < 2; ++ci)
              if (ci * 32 < cpw) {
                const int c0 = half * cpw + ci * 32;
                unsigned char* panel = sOut + (c0 >> 6) * a_slab;
#pragma unroll
                for (int ch = 0; ch < 4; ++ch)
                  *reinterpret_cast<uint4*>(panel + sw128_off(row, ((c0 & 63) >> 3) + ch)) =
                      make_uint4(w[ci * 16 + ch * 4], w[ci * 16 + ch * 4 + 1], w[ci * 16 + ch * 4 + 2], w[ci * 16 + ch * 4 + 3]);
              }
            fence_proxy_async_smem();
            if (npanel == 1) named_bar_sync(2 + quarter, 64);
            else __syncwarp();
            if (storer) {
              const int pn = npanel == 2 ? half : 0;
              if (t * 128 + quarter * 32 < p.rows)
                tma_store_2d(&p.omap[o], sOut + pn * a_slab + quarter * 32 * 128, pn * 64, (int)(t * 128 + quarter * 32));
              tma_store_commit();
            }
            store_pending = true;
          }
        } else if (half == (tn & 1)) {                       // the two halves take the bias in turn
          // bias: H values per position, written head-major / channel-major
          unsigned r[16];
          tmem_ld16(taddr, r);
          tmem_ld_wait16(r);
          const long long P = t * 128 + row;
          if (P < p.rows) {
            int s = 0;
            while (s + 1 < p.B && P >= p.pair_off[s + 1]) ++s;
            const int N = p.N[s], ld = round_up8(N);
            const unsigned rr = (unsigned)(P - p.pair_off[s]);      // N^2 < 2^32 (N < 2^16 for this path)
            const unsigned i = rr / (unsigned)N, j = rr - i * (unsigned)N;
            // (transposed planes: the register-fragment core reads a query's keys contiguously, and in column-wise attention
            // the bias of (query i, key k) is the plane's element [k][i])
            __nv_bfloat16* bp = p.bias + (long long)p.H * p.cm_off[s] + (N > p.bias_tr_above ? (long long)j * ld + i : (long long)i * ld + j);
#pragma unroll
            for (int h = 0; h < 16; ++h)
              if (h < p.H && NT_IN((bp - p.bias) + (long long)h * N * ld, p.bias_elems, NT_SITE_ATTN_IN_BIAS))
                bp[(long long)h * N * ld] = __float2bfloat16_rn(__uint_as_float(r[h]));
          }
        }
        if (u == 2) {
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(&tempty[buf]);
        }
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

bool fast_attn_in_supported(int c, int H, int d) {
  const int Hd = H * d;
  return (c == 64 || c == 128) && (Hd == 64 || Hd == 128) && H <= 16;
}

nt_status fast_attn_in(const void* z, const AttnPrep& ap, float eps, int c, int H, int d, void* q, void* k, void* v,
                       void* bias, const BatchMeta& m, int* status, cudaStream_t st, float2* zstats, int bias_tr_above) {
  const int Hd = H * d;
  const int wrows = 3 * Hd + 16;
  const void* wprime = ap.w;
  const int nslab = c / 64;
  const int npanel = Hd / 64;
  const size_t smem = (size_t)nslab * wrows * 128 + 2 * (size_t)nslab * 128 * 128 + (size_t)npanel * 128 * 128 +
                      2 * (size_t)wrows * 16 + 2 * 2 * (size_t)128 * 16 + 1024;
  // the attribute belongs to a (kernel, device) pair: one flag per device
  static bool attr_set_dev[64] = {};
  int attr_dev = 0;
  cudaGetDevice(&attr_dev);
  bool& attr_set = attr_set_dev[attr_dev & 63];
  if (!attr_set) {
    if (cudaFuncSetAttribute(attn_in_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, 220 * 1024) != cudaSuccess ||
        cudaFuncSetAttribute(attn_in_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, 220 * 1024) != cudaSuccess)
      return cuda_fail("attn_in smem attribute");
    attr_set = true;
  }
  for (int g0 = 0; g0 < m.B; g0 += AI_MAXB) {
    AttnInParams p;
    memset(&p, 0, sizeof(p));
    p.B = m.B - g0 < AI_MAXB ? m.B - g0 : AI_MAXB;
    p.c = c;
    p.H = H;
    p.Hd = Hd;
    p.eps = eps;
    p.aug_rows = ap.aug_rows;
    p.bias = (__nv_bfloat16*)bias;
    p.status = status;
    const long long P0 = m.pair_off[g0];
    p.zstats = zstats ? zstats + P0 : nullptr;
    p.bias_tr_above = bias_tr_above;
    p.bias_elems = (long long)H * m.cm_off[m.B];
    p.pair_off[0] = 0;
    for (int l = 0; l < AI_MAXB; ++l) {
      const int N = l < p.B ? m.N[g0 + l] : 0;
      p.N[l] = N;
      p.cm_off[l] = l < p.B ? m.cm_off[g0 + l] : 0;
      p.pair_off[l + 1] = p.pair_off[l] + (long long)N * N;
    }
    p.rows = p.pair_off[p.B];
    if (p.rows == 0) continue;
    if (p.rows > 0x7FFFFF00ll) return NT_ERR_UNSUPPORTED;
    {
      const unsigned long long dims[2] = {(unsigned long long)c, (unsigned long long)p.rows};
      const unsigned long long strides[1] = {(unsigned long long)c * 2};
      const unsigned box[2] = {64, 128};
      if (!make_tmap_bf16(&p.zmap, (const char*)z + (size_t)P0 * c * 2, 2, dims, strides, box))
        return cuda_fail("attn_in z map");
      const unsigned long long wdims[2] = {(unsigned long long)c, (unsigned long long)wrows};
      if (!make_tmap_bf16(&p.wmap, wprime, 2, wdims, strides, box)) return cuda_fail("attn_in w map");
      const unsigned long long xdims[2] = {8, (unsigned long long)2 * ap.aug_rows};
      const unsigned long long xstr[1] = {16};
      const unsigned xbox[2] = {8, 16};
      if (!make_tmap_16bit(&p.xmap, ap.aug, 2, xdims, xstr, xbox, 0)) return cuda_fail("attn_in augmentation map");
      const unsigned bbox[2] = {64, 16};
      if (!make_tmap_bf16(&p.wbmap, wprime, 2, wdims, strides, bbox)) return cuda_fail("attn_in wb map");
      const unsigned long long odims[2] = {(unsigned long long)Hd, (unsigned long long)p.rows};
      const unsigned long long ostr[1] = {(unsigned long long)Hd * 2};
      void* outs[3] = {q, k, v};
      const unsigned obox[2] = {64, 32};
      for (int o = 0; o < 3; ++o)
        if (!make_tmap_bf16(&p.omap[o], (char*)outs[o] + (size_t)P0 * Hd * 2, 2, odims, ostr, obox))
          return cuda_fail("attn_in out map");
    }
    const long long ntiles = (p.rows + 127) / 128;
    // few tiles: an SM for q | k and one for v and the bias of each halve the weights to wait for and the units to go through
    // (as in the triangle's input projection)
    const bool split = 2 * ntiles <= sm_count();
    const long long nwork = split ? 2 * ntiles : ntiles;
    const unsigned grid = (unsigned)(nwork < sm_count() ? nwork : sm_count());
    {
      LaunchScope ls("attn_in", st);
      launch_kernel(split ? attn_in_kernel<true> : attn_in_kernel<false>, grid, AI_THREADS, smem, st, p);
    }
    if (cudaPeekAtLastError() != cudaSuccess) return cuda_fail("attn_in launch");
  }
  return NT_OK;
}

}  // namespace ntp
