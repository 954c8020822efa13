// Token-side projection GEMMs on tcgen05: out[r][n] (+)= sum_k A[r][k] W[n][k] for up to two (W, out) pairs that
// share the activation A (q | k, v | g, the output projection accumulated into the residual stream).
//
// These are plain dense GEMMs over the packed token rows ([T1, K] x [N, K]^T): where the token axis is the whole
// workload (the single-ragged special case: T1 ~ 6 400, K = N = 768) they are most of the step.  A persistent CTA per
// SM walks (128-row block, BN-column block) tiles:
//   warp 0    TMA producer: 64-wide K slabs of the A rows and of the W rows into a 4-stage ring (both K-major,
//             128-byte swizzle); rows past the end of A are zero-filled by TMA
//   warp 1    MMA issuer: 128 x BN x 16 steps into one of two TMEM accumulators (the epilogue of a tile overlaps
//             the MMAs of the next)
//   warps 2-9 epilogue, two per TMEM lane quarter on alternate 64-column groups: TMEM -> registers -> bf16 or float,
//             added to the old value when accumulating, stored row-major (a thread owns a row: 128-byte runs)
#include <cstring>

#include "fast.cuh"
#include "tc_common.cuh"

namespace ntp {

constexpr int TG_STAGES = 4;
constexpr int TG_A_BYTES = 128 * 128;            // 128 rows x 64 bf16
constexpr int TG_THREADS = 64 + 256;

struct TokGemmTcParams {
  CUtensorMap amap;        // {K, rows}, box {64, 128}
  CUtensorMap wmap[TOK_SEGS];   // {K, N_i}, box {64, BN}
  void* out[TOK_SEGS];
  int N[TOK_SEGS];
  long long rows;
  int K, BN, out_f32, accumulate;
  int ntile[TOK_SEGS];     // column tiles of each output
  int ncol;                // of all of them
  int* status;
};

template <int BN>
__global__ void __launch_bounds__(TG_THREADS, 1) token_gemm_tc_kernel(const __grid_constant__ TokGemmTcParams p) {
  constexpr int B_BYTES = BN * 128;
  constexpr int STAGE_BYTES = TG_A_BYTES + B_BYTES;
  extern __shared__ unsigned char smem_raw[];
  __shared__ __align__(8) unsigned long long bars[2 * TG_STAGES + 4];
  __shared__ unsigned tmem_base_s;
  __shared__ int abort_flag;
  unsigned char* smem = smem_raw + ((1024 - (smem_u32(smem_raw) & 1023)) & 1023);
  unsigned long long* full = bars;
  unsigned long long* empty = bars + TG_STAGES;
  unsigned long long* tfull = bars + 2 * TG_STAGES;
  unsigned long long* tempty = bars + 2 * TG_STAGES + 2;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    abort_flag = 0;
    for (int s = 0; s < TG_STAGES; ++s) { mbar_init(&full[s], 1); mbar_init(&empty[s], 1); }
    for (int b = 0; b < 2; ++b) { mbar_init(&tfull[b], 1); mbar_init(&tempty[b], 8); }
    mbar_fence_init();
  }
  if (warp == 1) tmem_alloc(&tmem_base_s, 512);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  pdl_begin();
  const unsigned tmem_base = tmem_base_s;
  AbortCtx ab{p.status, &abort_flag};
  const int ncol = p.ncol;
  const long long nrow = (p.rows + 127) / 128;
  const long long njobs = nrow * ncol;
  const int nkc = (p.K + 63) / 64;
  // job -> (row block, output, column block): the column tiles of one row block are neighbours, so its A slabs are
  // fetched from L2 by CTAs running at the same time

  if (warp == 0 && lane == 0) {
    // ------------------------------------------------------------------ TMA producer
    int stage = 0;
    unsigned phase = 0;
    for (long long job = blockIdx.x; job < njobs; job += gridDim.x) {
      const long long rb = job / ncol;
      int cb = (int)(job - rb * ncol), which = 0;
      while (cb >= p.ntile[which]) cb -= p.ntile[which++];
      for (int kc = 0; kc < nkc; ++kc) {
        mbar_wait(&empty[stage], phase ^ 1, ab);
        unsigned char* As = smem + stage * STAGE_BYTES;
        mbar_expect_tx(&full[stage], STAGE_BYTES);
        tma_load_2d(As, &p.amap, &full[stage], kc * 64, (int)(rb * 128));
        tma_load_2d(As + TG_A_BYTES, &p.wmap[which], &full[stage], kc * 64, cb * BN);
        if (++stage == TG_STAGES) { stage = 0; phase ^= 1; }
      }
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------------ MMA issuer (whole warp, one elected lane issues)
    int stage = 0;
    unsigned phase = 0, tph[2] = {0, 0};
    unsigned n = 0;
    const unsigned idesc = idesc_f16(128, BN, 0, 0, FMT_BF16, FMT_BF16);
    for (long long job = blockIdx.x; job < njobs; job += gridDim.x, ++n) {
      const unsigned buf = n & 1;
      mbar_wait(&tempty[buf], tph[buf] ^ 1, ab);
      tph[buf] ^= 1;
      tc_fence_after();
      const unsigned d_tmem = tmem_base + buf * 256;
      for (int kc = 0; kc < nkc; ++kc) {
        mbar_wait(&full[stage], phase, ab);
        tc_fence_after();
        const unsigned a_addr = smem_u32(smem + stage * STAGE_BYTES);
        const unsigned long long a_desc = desc_kmajor_sw128(a_addr), b_desc = desc_kmajor_sw128(a_addr + TG_A_BYTES);
        const int ksteps = min(4, (p.K - kc * 64 + 15) / 16);
        if (elect_one()) {
          if (ksteps == 4) {
#pragma unroll
            for (int k4 = 0; k4 < 4; ++k4) umma_bf16(d_tmem, a_desc + k4 * 2, b_desc + k4 * 2, idesc, (kc | k4) != 0);
          } else {
            for (int k4 = 0; k4 < ksteps; ++k4) umma_bf16(d_tmem, a_desc + k4 * 2, b_desc + k4 * 2, idesc, (kc | k4) != 0);
          }
          tc_commit(&empty[stage]);
        }
        __syncwarp();
        if (++stage == TG_STAGES) { stage = 0; phase ^= 1; }
      }
      if (elect_one()) tc_commit(&tfull[buf]);
      __syncwarp();
    }
  } else if (warp >= 2) {
    // ------------------------------------------------------------------ epilogue
    const int quarter = warp & 3, half = (warp - 2) >> 2;
    const int row = quarter * 32 + lane;
    unsigned tph[2] = {0, 0};
    long long n = 0;
    for (long long job = blockIdx.x; job < njobs; job += gridDim.x, ++n) {
      const long long rb = job / ncol;
      int cb = (int)(job - rb * ncol), which = 0;
      while (cb >= p.ntile[which]) cb -= p.ntile[which++];
      const int buf = (int)(n & 1);
      mbar_wait(&tfull[buf], tph[buf], ab);
      tph[buf] ^= 1;
      tc_fence_after();
      const unsigned taddr = tmem_base + ((unsigned)(quarter * 32) << 16) + buf * 256;
      const long long r = rb * 128 + row;
      const int Nout = p.N[which];
      for (int cg = half; cg < BN / 64; cg += 2) {
        unsigned r0[32], r1[32];
        tmem_ld32(taddr + cg * 64, r0);
        tmem_ld32(taddr + cg * 64 + 32, r1);
        tmem_ld_wait();
        if (r < p.rows && NT_IN(cb * BN + cg * 64 + 63, Nout, NT_SITE_TOKEN_GEMM_OUT)) {
          const long long off = r * Nout + cb * BN + cg * 64;
          // 32-byte stores: a thread's columns are whole sectors, which 16-byte stores each write in part
          const bool wide = ((unsigned long long)p.out[which] & 31) == 0;
          if (p.out_f32) {
            float* o = (float*)p.out[which] + off;
#pragma unroll
            for (int e = 0; e < 8; ++e) {
              const unsigned* src = e < 4 ? r0 + e * 8 : r1 + (e - 4) * 8;
              unsigned v[8];
#pragma unroll
              for (int q = 0; q < 8; ++q) v[q] = __float_as_uint(__uint_as_float(src[q]) + (p.accumulate ? o[e * 8 + q] : 0.f));
              store_32b(o + e * 8, v, wide);
            }
          } else {
            __nv_bfloat16* o = (__nv_bfloat16*)p.out[which] + off;
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              const unsigned* src = e < 2 ? r0 + e * 16 : r1 + (e - 2) * 16;
              float f[16];
#pragma unroll
              for (int q = 0; q < 16; ++q) f[q] = __uint_as_float(src[q]);
              if (p.accumulate) {
                const uint4 x = *reinterpret_cast<const uint4*>(o + e * 16), y = *reinterpret_cast<const uint4*>(o + e * 16 + 8);
                const unsigned ow[8] = {x.x, x.y, x.z, x.w, y.x, y.y, y.z, y.w};
#pragma unroll
                for (int q = 0; q < 8; ++q) {
                  f[2 * q] += __uint_as_float(ow[q] << 16);
                  f[2 * q + 1] += __uint_as_float(ow[q] & 0xffff0000u);
                }
              }
              unsigned v[8];
#pragma unroll
              for (int q = 0; q < 8; ++q) v[q] = pack2(__float_as_uint(f[2 * q]), __float_as_uint(f[2 * q + 1]));
              store_32b(o + e * 16, v, wide);
            }
          }
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&tempty[buf]);
    }
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  abort_linger(ab);
  if (warp == 1) tmem_dealloc(tmem_base, 512);
}

bool fast_token_gemm_tc_supported(const TokSeg* seg, int n, int K) {
  // worth a persistent tensor-core launch only when there are enough tiles; shapes: K a multiple of 64 (full
  // swizzled slabs), outputs a multiple of 128 columns
  if (K % 64 != 0 || K < 64) return false;
  for (int i = 0; i < n; ++i)
    if (seg[i].N % 128 != 0 || seg[i].N < 128) return false;
  return seg[0].rows >= 2048 && seg[0].rows <= 0x7FFFFF00ll;
}

template <int BN>
static nt_status launch_tg(TokGemmTcParams& p, const char* name, cudaStream_t st) {
  static bool attr_set[64] = {};
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev < 0 || dev >= 64) return NT_ERR_UNSUPPORTED;
  const size_t smem = (size_t)TG_STAGES * (TG_A_BYTES + BN * 128) + 1024;
  if (!attr_set[dev]) {
    if (cudaFuncSetAttribute(token_gemm_tc_kernel<BN>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess)
      return cuda_fail("token gemm tc smem attribute");
    attr_set[dev] = true;
  }
  const long long njobs = ((p.rows + 127) / 128) * p.ncol;
  const int sms = sm_count();
  {
    LaunchScope ls(name, st);
    launch_kernel(token_gemm_tc_kernel<BN>, (unsigned)(njobs < sms ? njobs : sms), TG_THREADS, smem, st, p);
  }
  return cuda_ok(name);
}

nt_status fast_token_gemm_tc(const TokSeg* seg, int n, int K, int out_f32, int accumulate, int* status, const char* name, cudaStream_t st) {
  if (!fast_token_gemm_tc_supported(seg, n, K)) return NT_ERR_UNSUPPORTED;
  const long long rows = seg[0].rows;
  TokGemmTcParams p;
  memset(&p, 0, sizeof(p));
  p.rows = rows;
  p.K = K;
  p.out_f32 = out_f32;
  p.accumulate = accumulate;
  p.status = status;
  int cols = 0;
  bool by256 = true;
  for (int i = 0; i < n; ++i) {
    p.out[i] = seg[i].out;
    p.N[i] = seg[i].N;
    cols += seg[i].N;
    by256 = by256 && seg[i].N % 256 == 0;
  }
  // tile width by wave quantisation: the width whose tile count leaves the shorter tail on this many SMs
  int BN = 128;
  if (by256) {
    const long long rb = (rows + 127) / 128, sms = sm_count();
    const long long j256 = rb * (cols / 256), j128 = rb * (cols / 128);
    if (((j256 + sms - 1) / sms) * 256 <= ((j128 + sms - 1) / sms) * 128) BN = 256;
  }
  p.BN = BN;
  p.ncol = cols / BN;
  {
    const unsigned long long dims[2] = {(unsigned long long)K, (unsigned long long)rows};
    const unsigned long long strides[1] = {(unsigned long long)K * 2};
    const unsigned box[2] = {64, 128};
    if (!make_tmap_bf16(&p.amap, seg[0].A, 2, dims, strides, box)) return cuda_fail("token gemm tc A map");
  }
  for (int i = 0; i < n; ++i) {
    p.ntile[i] = p.N[i] / BN;
    const unsigned long long dims[2] = {(unsigned long long)K, (unsigned long long)p.N[i]};
    const unsigned long long strides[1] = {(unsigned long long)K * 2};
    const unsigned box[2] = {64, (unsigned)BN};
    if (!make_tmap_bf16(&p.wmap[i], seg[i].W, 2, dims, strides, box)) return cuda_fail("token gemm tc W map");
  }
  return BN == 256 ? launch_tg<256>(p, name, st) : launch_tg<128>(p, name, st);
}

}  // namespace ntp
