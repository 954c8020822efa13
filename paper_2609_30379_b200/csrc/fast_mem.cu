// Memory-bound bf16 kernels on CUDA cores: the segmented mean/sum (pure streaming read), the token-axis
// GEMMs and the small row-wise helpers of the token-order calls.
#include "fast.cuh"

namespace ntp {

// ------------------------------------------------------------------------------------------
// segmented mean / sum over contiguous row groups, bf16 in, float accumulate, bf16 out.
// One block per group; VL = C / 8 lanes cover a row with 16-byte loads, 128 / VL rows in flight (small blocks: all
// groups of a typical batch are resident at once, so there is no second, partly filled wave).
// ------------------------------------------------------------------------------------------
constexpr int SR_THREADS = 128;
constexpr int SR_UNROLL = 4;
constexpr int SR_CHUNK = 128;     // channels per block

__global__ void __launch_bounds__(SR_THREADS) segment_reduce_fast_kernel(const __nv_bfloat16* v,
                                                                        __nv_bfloat16* out,
                                                                        const int64_t* splits, int C,
                                                                        int mean) {
  pdl_begin();
  extern __shared__ float part[];   // [RS][Cc]
  // a block reduces one group over a chunk of up to 128 channels (blockIdx.y): wide rows keep several row slots
  const int CV = C >> 3;                                  // 16-byte vectors per row
  const int cb = blockIdx.y * SR_CHUNK;                   // first channel of the chunk
  const int Cc = min(SR_CHUNK, C - cb);
  const int VL = Cc >> 3;
  const int RS = SR_THREADS / VL;
  const int t = threadIdx.x;
  const int slot = t / VL, vl = t - slot * VL;
  const long long g = blockIdx.x;
  const long long lo = splits[g], hi = splits[g + 1];
  float acc[8] = {};
  if (slot < RS) {
    const uint4* base = reinterpret_cast<const uint4*>(v) + (cb >> 3) + vl;
    long long r = lo + slot;
    for (; r + (long long)(SR_UNROLL - 1) * RS < hi; r += (long long)SR_UNROLL * RS) {
      uint4 d[SR_UNROLL];
#pragma unroll
      for (int uu = 0; uu < SR_UNROLL; ++uu) d[uu] = *(base + (r + (long long)uu * RS) * CV);
#pragma unroll
      for (int uu = 0; uu < SR_UNROLL; ++uu) {
        const unsigned w[4] = {d[uu].x, d[uu].y, d[uu].z, d[uu].w};
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          acc[2 * e] += __uint_as_float(w[e] << 16);
          acc[2 * e + 1] += __uint_as_float(w[e] & 0xffff0000u);
        }
      }
    }
    for (; r < hi; r += RS) {
      const uint4 d = *(base + r * CV);
      const unsigned w[4] = {d.x, d.y, d.z, d.w};
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        acc[2 * e] += __uint_as_float(w[e] << 16);
        acc[2 * e + 1] += __uint_as_float(w[e] & 0xffff0000u);
      }
    }
#pragma unroll
    for (int e = 0; e < 8; ++e) part[slot * Cc + vl * 8 + e] = acc[e];
  }
  __syncthreads();
  const long long n = hi - lo;
  const float sc = (mean && n > 0) ? 1.0f / (float)n : 1.0f;
  for (int c = t; c < Cc; c += SR_THREADS) {
    float tot = 0.f;
    for (int sl = 0; sl < RS; ++sl) tot += part[sl * Cc + c];
    if (NT_IN(cb + c, C, NT_SITE_FAST_SEGMENT)) out[g * C + cb + c] = __float2bfloat16_rn(tot * sc);
  }
}

bool fast_segment_reduce_supported(int C) { return C % 8 == 0 && C >= 8 && C <= 8 * SR_THREADS; }

nt_status fast_segment_reduce(const void* v, void* out, const int64_t* splits, long long G, int C, int mean,
                              cudaStream_t st) {
  if (G <= 0) return NT_OK;
  if (G > 0x7FFFFFFFll) return NT_ERR_UNSUPPORTED;
  const size_t smem = (size_t)SR_THREADS * 8 * sizeof(float);   // row slots x chunk channels never exceed threads x 8
  const dim3 grid((unsigned)G, (unsigned)((C + SR_CHUNK - 1) / SR_CHUNK));
  {
    LaunchScope ls("segment_reduce", st);
    launch_kernel(segment_reduce_fast_kernel, grid, SR_THREADS, smem, st, (const __nv_bfloat16*)v, (__nv_bfloat16*)out,
                                                                     splits, C, mean);
  }
  return cuda_ok();
}

}  // namespace ntp

namespace ntp {

// ------------------------------------------------------------------------------------------
// Token-side projection (a few thousand rows, so a fraction of a percent of a block's work):
//   out[r][n] (+)= sum_k A[r][k] W[n][k]   for up to four segments (rows, weight, output), one after the other in grid.y.
// 32 x 32 output tiles so that even T1 ~ 1.7k rows give several hundred CTAs; the A and W tiles are
// staged whole in shared memory (K <= 1024).
// ------------------------------------------------------------------------------------------
struct TokGemmArgs {
  const __nv_bfloat16* A[TOK_SEGS];
  long long rows[TOK_SEGS];
  int K;
  const __nv_bfloat16* W[TOK_SEGS];
  int N[TOK_SEGS];
  void* out[TOK_SEGS];
  int out_f32;       // outputs are float (store) instead of bf16
  int accumulate;    // bf16 outputs: out += result
};

__global__ void __launch_bounds__(256) token_gemm_kernel(TokGemmArgs a) {
  pdl_begin();
  extern __shared__ __align__(16) unsigned char tg_smem[];
  const int K = a.K, ldk = K + 8;
  __nv_bfloat16* As = reinterpret_cast<__nv_bfloat16*>(tg_smem);
  __nv_bfloat16* Ws = As + 32 * ldk;
  const long long r0 = (long long)blockIdx.x * 32;
  int n0 = blockIdx.y * 32, which = 0;
  while (n0 >= a.N[which]) n0 -= a.N[which++];
  const __nv_bfloat16 *A = a.A[which], *W = a.W[which];
  const long long rows = a.rows[which];
  if (r0 >= rows) return;
  const int N = a.N[which];
  const int t = threadIdx.x, kv = K / 8;
  for (int idx = t; idx < 32 * kv; idx += 256) {
    const int r = idx / kv, c = idx - r * kv;
    uint4 va = make_uint4(0, 0, 0, 0), vw = make_uint4(0, 0, 0, 0);
    if (r0 + r < rows) va = *reinterpret_cast<const uint4*>(A + (r0 + r) * K + c * 8);
    if (n0 + r < N) vw = *reinterpret_cast<const uint4*>(W + (long long)(n0 + r) * K + c * 8);
    *reinterpret_cast<uint4*>(As + r * ldk + c * 8) = va;
    *reinterpret_cast<uint4*>(Ws + r * ldk + c * 8) = vw;
  }
  __syncthreads();
  const int ty = t >> 4, tx = t & 15;
  float acc[2][2] = {};
  for (int k = 0; k < K; k += 8) {
    uint4 av[2], wv[2];
    av[0] = *reinterpret_cast<const uint4*>(As + ty * ldk + k);
    av[1] = *reinterpret_cast<const uint4*>(As + (ty + 16) * ldk + k);
    wv[0] = *reinterpret_cast<const uint4*>(Ws + tx * ldk + k);
    wv[1] = *reinterpret_cast<const uint4*>(Ws + (tx + 16) * ldk + k);
    const unsigned* ap0 = reinterpret_cast<const unsigned*>(&av[0]);
    const unsigned* ap1 = reinterpret_cast<const unsigned*>(&av[1]);
    const unsigned* wp0 = reinterpret_cast<const unsigned*>(&wv[0]);
    const unsigned* wp1 = reinterpret_cast<const unsigned*>(&wv[1]);
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const float a0l = __uint_as_float(ap0[e] << 16), a0h = __uint_as_float(ap0[e] & 0xffff0000u);
      const float a1l = __uint_as_float(ap1[e] << 16), a1h = __uint_as_float(ap1[e] & 0xffff0000u);
      const float w0l = __uint_as_float(wp0[e] << 16), w0h = __uint_as_float(wp0[e] & 0xffff0000u);
      const float w1l = __uint_as_float(wp1[e] << 16), w1h = __uint_as_float(wp1[e] & 0xffff0000u);
      acc[0][0] = fmaf(a0l, w0l, fmaf(a0h, w0h, acc[0][0]));
      acc[0][1] = fmaf(a0l, w1l, fmaf(a0h, w1h, acc[0][1]));
      acc[1][0] = fmaf(a1l, w0l, fmaf(a1h, w0h, acc[1][0]));
      acc[1][1] = fmaf(a1l, w1l, fmaf(a1h, w1h, acc[1][1]));
    }
  }
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const long long r = r0 + ty + 16 * i;
      const int n = n0 + tx + 16 * j;
      if (r >= rows || n >= N) continue;
      if (a.out_f32) {
        reinterpret_cast<float*>(a.out[which])[r * N + n] = acc[i][j];
      } else {
        __nv_bfloat16* o = reinterpret_cast<__nv_bfloat16*>(a.out[which]) + r * N + n;
        const float base = a.accumulate ? __bfloat162float(*o) : 0.f;
        *o = __float2bfloat16_rn(base + acc[i][j]);
      }
    }
}

// Tensor-core version (mma.sync m16n8k16, bf16 in, float accumulate) for 64 x 64 output tiles: the token-side GEMMs
// have only a few thousand rows, so one small CTA tile per SM and a whole-K shared-memory panel is all they need.
// Eight warps: warp w owns rows (w & 3) * 16 .. + 16 and columns (w >> 2) * 32 .. + 32 of the tile.
__device__ inline void tg_ldsm_x4(unsigned& r0, unsigned& r1, unsigned& r2, unsigned& r3, const void* p) {
  const unsigned a = (unsigned)__cvta_generic_to_shared(p);
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];\n" : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3) : "r"(a));
}
__device__ inline void tg_mma(float (&c)[4], const unsigned (&a)[4], unsigned b0, unsigned b1) {
  asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};\n"
               : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3]) : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

__global__ void __launch_bounds__(256) token_gemm_mma_kernel(TokGemmArgs a) {
  pdl_begin();
  extern __shared__ __align__(16) unsigned char tg_smem[];
  const int K = a.K, ldk = K + 8;                      // row pitch 16 bytes off a multiple of 128: conflict-free ldmatrix
  __nv_bfloat16* As = reinterpret_cast<__nv_bfloat16*>(tg_smem);
  __nv_bfloat16* Ws = As + 64 * ldk;
  const long long r0 = (long long)blockIdx.x * 64;
  int n0 = blockIdx.y * 64, which = 0;
  while (n0 >= a.N[which]) n0 -= a.N[which++];
  const __nv_bfloat16 *A = a.A[which], *W = a.W[which];
  const long long rows = a.rows[which];
  if (r0 >= rows) return;
  const int N = a.N[which];
  const int t = threadIdx.x, kv = K / 8;
  // both panels with asynchronous 16-byte copies: every load of the CTA is in flight at once
  for (int idx = t; idx < 64 * kv; idx += 256) {
    const int r = idx / kv, c = idx - r * kv;
    const bool ok = r0 + r < rows;
    const unsigned da = (unsigned)__cvta_generic_to_shared(As + r * ldk + c * 8), dw = (unsigned)__cvta_generic_to_shared(Ws + r * ldk + c * 8);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(da), "l"(A + (ok ? r0 + r : 0) * K + c * 8), "r"(ok ? 16 : 0));
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(dw), "l"(W + (long long)(n0 + r) * K + c * 8));
  }
  asm volatile("cp.async.wait_all;\n" ::: "memory");
  __syncthreads();
  const int warp = t >> 5, lane = t & 31;
  const int wr = (warp & 3) * 16, wc = (warp >> 2) * 32;
  float acc[4][4] = {};
  const __nv_bfloat16* ap = As + (wr + (lane & 7) + ((lane >> 3) & 1) * 8) * ldk + (lane >> 4) * 8;
  const __nv_bfloat16* wp = Ws + (wc + (lane & 7) + (lane >> 4) * 8) * ldk + ((lane >> 3) & 1) * 8;
  for (int k = 0; k < K; k += 16) {
    unsigned af[4], b[4], d[4];
    tg_ldsm_x4(af[0], af[1], af[2], af[3], ap + k);
    tg_ldsm_x4(b[0], b[1], b[2], b[3], wp + k);
    tg_ldsm_x4(d[0], d[1], d[2], d[3], wp + 16 * ldk + k);
    tg_mma(acc[0], af, b[0], b[1]);
    tg_mma(acc[1], af, b[2], b[3]);
    tg_mma(acc[2], af, d[0], d[1]);
    tg_mma(acc[3], af, d[2], d[3]);
  }
  const int g = lane >> 2, tq = lane & 3;
#pragma unroll
  for (int nt = 0; nt < 4; ++nt)
#pragma unroll
    for (int hh = 0; hh < 2; ++hh) {
      const long long r = r0 + wr + g + hh * 8;
      const int n = n0 + wc + nt * 8 + 2 * tq;
      if (r >= rows) continue;
      const float x0 = acc[nt][hh * 2], x1 = acc[nt][hh * 2 + 1];
      if (a.out_f32) {
        *reinterpret_cast<float2*>(reinterpret_cast<float*>(a.out[which]) + r * N + n) = make_float2(x0, x1);
      } else {
        __nv_bfloat162* o = reinterpret_cast<__nv_bfloat162*>(reinterpret_cast<__nv_bfloat16*>(a.out[which]) + r * N + n);
        float2 base = make_float2(0.f, 0.f);
        if (a.accumulate) base = __bfloat1622float2(*o);
        *o = __floats2bfloat162_rn(base.x + x0, base.y + x1);
      }
    }
}

bool fast_token_gemm_supported(int K, int N0, int N1) {
  return K % 8 == 0 && K >= 8 && K <= 1024 && N0 % 32 == 0 && N1 % 32 == 0;
}

nt_status fast_token_gemm(const TokSeg* seg, int n, int K, int out_f32, int accumulate, const char* name, cudaStream_t st) {
  TokGemmArgs a{};
  long long rows = 0;
  int cols = 0, m = 0;
  bool by64 = K % 16 == 0, shared = true;
  TokSeg used[TOK_SEGS];
  for (int i = 0; i < n; ++i) {
    if (!seg[i].W || seg[i].N == 0 || seg[i].rows <= 0) continue;
    if (m == TOK_SEGS) return NT_ERR_UNSUPPORTED;
    shared = shared && (m == 0 || (seg[i].A == used[0].A && seg[i].rows == used[0].rows));
    by64 = by64 && seg[i].N % 64 == 0;
    rows = rows > seg[i].rows ? rows : seg[i].rows;
    cols += seg[i].N;
    a.A[m] = (const __nv_bfloat16*)seg[i].A;
    a.rows[m] = seg[i].rows;
    a.W[m] = (const __nv_bfloat16*)seg[i].W;
    a.N[m] = seg[i].N;
    a.out[m] = seg[i].out;
    used[m++] = seg[i];
  }
  if (m == 0) return NT_OK;
  if (shared && fast_token_gemm_tc_supported(used, m, K))         // a token axis long enough for persistent tcgen05 tiles
    return fast_token_gemm_tc(used, m, K, out_f32, accumulate, nullptr, name, st);
  if (!shared) {                                                  // any segment that is long enough for them goes by itself
    bool lone = false;
    for (int i = 0; i < m; ++i) lone = lone || fast_token_gemm_tc_supported(used + i, 1, K);
    if (lone) {
      for (int i = 0; i < m; ++i) {
        nt_status r = fast_token_gemm(used + i, 1, K, out_f32, accumulate, name, st);
        if (r != NT_OK) return r;
      }
      return NT_OK;
    }
  }
  a.K = K;
  a.out_f32 = out_f32;
  a.accumulate = accumulate;
  if (by64) {
    const size_t smem64 = (size_t)2 * 64 * (K + 8) * 2;
    static bool attr64_dev[64] = {};
    int attr_dev = 0;
    cudaGetDevice(&attr_dev);
    bool& attr64 = attr64_dev[attr_dev & 63];
    if (!attr64) {
      if (cudaFuncSetAttribute(token_gemm_mma_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024) != cudaSuccess)
        return cuda_fail("token gemm smem attribute");
      attr64 = true;
    }
    if (smem64 <= 200 * 1024) {
      const long long bx64 = (rows + 63) / 64;
      if (bx64 > 0x7FFFFFFFll) return NT_ERR_UNSUPPORTED;
      dim3 grid64((unsigned)bx64, (unsigned)(cols / 64));
      {
        LaunchScope ls(name, st);
        launch_kernel(token_gemm_mma_kernel, grid64, 256, smem64, st, a);
      }
      return cuda_ok(name);
    }
  }
  const size_t smem = (size_t)2 * 32 * (K + 8) * 2;
  static size_t attr_by_dev[64] = {};
  int attr_dev2 = 0;
  cudaGetDevice(&attr_dev2);
  size_t& attr = attr_by_dev[attr_dev2 & 63];
  if (smem > 48 * 1024 && smem > attr) {
    if (cudaFuncSetAttribute(token_gemm_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 140 * 1024) != cudaSuccess)
      return cuda_fail("token gemm smem attribute");
    attr = 140 * 1024;
  }
  const long long bx = (rows + 31) / 32;
  if (bx > 0x7FFFFFFFll) return NT_ERR_UNSUPPORTED;
  dim3 grid((unsigned)bx, (unsigned)(cols / 32));
  {
    LaunchScope ls(name, st);
    launch_kernel(token_gemm_kernel, grid, 256, smem, st, a);
  }
  return cuda_ok(name);
}

}  // namespace ntp

// ------------------------------------------------------------------------------------------------------------------
// Pair-biased single attention: the CUDA-core pieces around the token GEMMs and the attention core.
// ------------------------------------------------------------------------------------------------------------------
namespace ntp {

// LayerNorm of token rows, bf16 in / bf16 out: one warp per row, 16-byte loads.
__global__ void __launch_bounds__(256) ln_rows_kernel(const __nv_bfloat16* x, const __nv_bfloat16* gamma,
                                                      const __nv_bfloat16* beta, float eps, int C, long long rows,
                                                      __nv_bfloat16* out) {
  pdl_begin();
  const long long r = (long long)blockIdx.x * 8 + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (r >= rows) return;
  const int nch = C / 8;
  uint4 v[8];
  float s = 0.f, q = 0.f;
#pragma unroll
  for (int u = 0; u < 8; ++u) {
    const int c8 = lane + u * 32;
    if (c8 < nch) {
      v[u] = *reinterpret_cast<const uint4*>(x + r * C + c8 * 8);
      const unsigned w[4] = {v[u].x, v[u].y, v[u].z, v[u].w};
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const float lo = __uint_as_float(w[e] << 16), hi = __uint_as_float(w[e] & 0xffff0000u);
        s += lo + hi;
        q = fmaf(lo, lo, q);
        q = fmaf(hi, hi, q);
      }
    }
  }
#pragma unroll
  for (int o = 16; o; o >>= 1) {
    s += __shfl_xor_sync(0xffffffffu, s, o);
    q += __shfl_xor_sync(0xffffffffu, q, o);
  }
  const float mean = s / (float)C;
  const float rstd = rsqrtf(fmaxf(q / (float)C - mean * mean, 0.f) + eps);
#pragma unroll
  for (int u = 0; u < 8; ++u) {
    const int c8 = lane + u * 32;
    if (c8 < nch) {
      const uint4 g4 = *reinterpret_cast<const uint4*>(gamma + c8 * 8), b4 = *reinterpret_cast<const uint4*>(beta + c8 * 8);
      const unsigned w[4] = {v[u].x, v[u].y, v[u].z, v[u].w}, gw[4] = {g4.x, g4.y, g4.z, g4.w}, bw[4] = {b4.x, b4.y, b4.z, b4.w};
      unsigned o4[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const float lo = (__uint_as_float(w[e] << 16) - mean) * rstd, hi = (__uint_as_float(w[e] & 0xffff0000u) - mean) * rstd;
        __nv_bfloat162 h = __floats2bfloat162_rn(fmaf(lo, __uint_as_float(gw[e] << 16), __uint_as_float(bw[e] << 16)),
                                                 fmaf(hi, __uint_as_float(gw[e] & 0xffff0000u), __uint_as_float(bw[e] & 0xffff0000u)));
        o4[e] = *reinterpret_cast<unsigned*>(&h);
      }
      *reinterpret_cast<uint4*>(out + r * C + c8 * 8) = make_uint4(o4[0], o4[1], o4[2], o4[3]);
    }
  }
}

// o <- sigmoid(g) * o, elementwise on bf16 (eight elements per thread)
__global__ void __launch_bounds__(256) gate_mul_kernel(const __nv_bfloat16* g, __nv_bfloat16* o, long long n8) {
  pdl_begin();
  const long long i = (long long)blockIdx.x * 256 + threadIdx.x;
  if (i >= n8) return;
  const uint4 gv = *reinterpret_cast<const uint4*>(g + i * 8);
  uint4 ov = *reinterpret_cast<const uint4*>(o + i * 8);
  const unsigned gw[4] = {gv.x, gv.y, gv.z, gv.w};
  unsigned ow[4] = {ov.x, ov.y, ov.z, ov.w};
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    const float g0 = __uint_as_float(gw[e] << 16), g1 = __uint_as_float(gw[e] & 0xffff0000u);
    const float o0 = __uint_as_float(ow[e] << 16), o1 = __uint_as_float(ow[e] & 0xffff0000u);
    __nv_bfloat162 h = __floats2bfloat162_rn(o0 / (1.0f + __expf(-g0)), o1 / (1.0f + __expf(-g1)));
    ow[e] = *reinterpret_cast<unsigned*>(&h);
  }
  *reinterpret_cast<uint4*>(o + i * 8) = make_uint4(ow[0], ow[1], ow[2], ow[3]);
}

// Bias planes of the pair-biased single attention: bias[s][h][i][j] = scale * (LN(z_ij) W_b^T)[h], head-major with the
// padded row stride of the channel-major buffers.  The pair state is read once; the H results per position are tiny.
// A warp takes 32 consecutive packed positions: sixteen lanes work on one position (16-byte loads, LayerNorm folded
// into the H weight rows kept in shared memory), the results are handed to the lane that owns the position, and the
// warp writes each head's 32 values as one run.
constexpr int SB_MAXH = 8;
template <int HT>      // heads the arithmetic runs over (H <= HT; rows H .. HT - 1 of the weight table are zeros)
__global__ void __launch_bounds__(256) single_bias_kernel(const __nv_bfloat16* z, const __nv_bfloat16* gamma,
                                                          const __nv_bfloat16* beta, const __nv_bfloat16* Wb,
                                                          float eps, int C, int H, float scale, BatchMeta m,
                                                          __nv_bfloat16* bias) {
  pdl_begin();
  extern __shared__ float sbw[];            // [HT][C] folded weights, then c0[HT], c1[HT]
  float* c0 = sbw + HT * C;
  float* c1 = c0 + SB_MAXH;
  for (int idx = threadIdx.x; idx < HT * C; idx += 256) {
    const int c = idx % C;
    sbw[idx] = idx < H * C ? __bfloat162float(Wb[idx]) * __bfloat162float(gamma[c]) : 0.f;
  }
  if (threadIdx.x < 2 * SB_MAXH) c0[threadIdx.x] = 0.f;
  __syncthreads();
  if ((threadIdx.x >> 5) < H) {            // warp h sums row h (H <= 8 = warps per block)
    const int h = threadIdx.x >> 5;
    float a0 = 0.f, a1 = 0.f;
    for (int c = threadIdx.x & 31; c < C; c += 32) {
      a0 = fmaf(__bfloat162float(Wb[h * C + c]), __bfloat162float(beta[c]), a0);
      a1 += sbw[h * C + c];
    }
#pragma unroll
    for (int o = 16; o; o >>= 1) {
      a0 += __shfl_xor_sync(0xffffffffu, a0, o);
      a1 += __shfl_xor_sync(0xffffffffu, a1, o);
    }
    if ((threadIdx.x & 31) == 0) {
      c0[h] = a0;
      c1[h] = a1;
    }
  }
  __syncthreads();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, hw = lane >> 4, l16 = lane & 15;
  const long long p0 = m.pair_off[0], p1 = m.pair_off[m.B];
  const long long nblk = (p1 - p0 + 31) / 32;
  const int nch = C / 8;
  for (long long blk = (long long)blockIdx.x * 8 + warp; blk < nblk; blk += (long long)gridDim.x * 8) {
    const long long base = p0 + blk * 32;
    float keep[HT];
#pragma unroll
    for (int h = 0; h < HT; ++h) keep[h] = 0.f;
    // four positions' loads are issued before the first is used (one 16-byte chunk per lane covers C <= 128;
    // wider rows take further chunks inside the step)
    for (int t0 = 0; t0 < 16; t0 += 4) {
      uint4 first[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const long long p = base + 2 * (t0 + u) + hw;
        first[u] = (p < p1 && l16 < nch) ? *reinterpret_cast<const uint4*>(z + p * C + l16 * 8) : make_uint4(0, 0, 0, 0);
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int t = t0 + u;
        const long long p = base + 2 * t + hw;
        float s = 0.f, q = 0.f, dot[HT];
#pragma unroll
        for (int h = 0; h < HT; ++h) dot[h] = 0.f;
        for (int c8 = l16; c8 < nch; c8 += 16) {
          uint4 v = first[u];
          if (c8 != l16) v = p < p1 ? *reinterpret_cast<const uint4*>(z + p * C + c8 * 8) : make_uint4(0, 0, 0, 0);
          const unsigned w[4] = {v.x, v.y, v.z, v.w};
          float f[8];
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            f[2 * e] = __uint_as_float(w[e] << 16);
            f[2 * e + 1] = __uint_as_float(w[e] & 0xffff0000u);
          }
#pragma unroll
          for (int e = 0; e < 8; ++e) {
            s += f[e];
            q = fmaf(f[e], f[e], q);
          }
#pragma unroll
          for (int h = 0; h < HT; ++h) {
              const float4 w0 = *reinterpret_cast<const float4*>(sbw + h * C + c8 * 8), w1 = *reinterpret_cast<const float4*>(sbw + h * C + c8 * 8 + 4);
              dot[h] = fmaf(f[0], w0.x, fmaf(f[1], w0.y, fmaf(f[2], w0.z, fmaf(f[3], w0.w, dot[h]))));
              dot[h] = fmaf(f[4], w1.x, fmaf(f[5], w1.y, fmaf(f[6], w1.z, fmaf(f[7], w1.w, dot[h]))));
            }
        }
#pragma unroll
        for (int o = 8; o; o >>= 1) {
          s += __shfl_xor_sync(0xffffffffu, s, o);
          q += __shfl_xor_sync(0xffffffffu, q, o);
#pragma unroll
          for (int h = 0; h < HT; ++h) dot[h] += __shfl_xor_sync(0xffffffffu, dot[h], o);
        }
        const float mean = s / (float)C;
        const float rstd = rsqrtf(fmaxf(q / (float)C - mean * mean, 0.f) + eps);
#pragma unroll
        for (int h = 0; h < HT; ++h) {
            const float r = (rstd * (dot[h] - mean * c1[h]) + c0[h]) * scale;
            const float got = __shfl_sync(0xffffffffu, r, (lane & 1) * 16);     // from the half-warp that holds position 2 t + (lane & 1)
            if ((lane >> 1) == t) keep[h] = got;
          }
      }
    }
    const long long p = base + lane;
    if (p < p1) {
      const int s_ = find_sample(m.pair_off, m.B, p);
      const int N = m.N[s_], ld = round_up8(N);
      const long long r = p - m.pair_off[s_];
      const int i = (int)(r / N), j = (int)(r - (long long)i * N);
      __nv_bfloat16* bp = bias + (long long)H * m.cm_off[s_] + (long long)i * ld + j;
#pragma unroll
      for (int h = 0; h < HT; ++h)
        if (h < H) bp[(long long)h * N * ld] = __float2bfloat16_rn(keep[h]);
    }
  }
}

// The same planes on the tensor cores (H <= 4, C = 16 NK): per 16 positions one m16n8k16 MMA per 16 channels against
// B = [W'_0 .. W'_3 | 1 | 0 ..] gives the H dot products and the row sum; a second MMA of the squared inputs against
// a ones column adds the sum of squares as column 5 of the same accumulator, so the LayerNorm statistics cost no
// shuffle reductions at all.  A fragments come straight from global memory; a dot product does not
// care which channel is which k as long as A and B agree, so a lane's eight contiguous channels (one 16-byte load) are
// the k positions it holds in two k steps: an eighth of the load instructions of the layout in order, and two whole
// sectors of a row per instruction; the next tile is requested before the epilogue of the current one.  Measured (c = 128): one
// sample of 977, 86 -> 58 us (HBM 38); eight of about 215, 38 -> 26.  W' = W_b gamma is rounded to bf16; c1 is the sum of the rounded values.
__device__ inline void mma_bf16_16816(float (&c)[4], const unsigned (&a)[4], unsigned b0, unsigned b1) {
  asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};\n"
               : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
               : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

template <int NK>
__global__ void __launch_bounds__(256) single_bias_mma_kernel(const __nv_bfloat16* z, const __nv_bfloat16* gamma,
                                                              const __nv_bfloat16* beta, const __nv_bfloat16* Wb,
                                                              float eps, int H, float scale, BatchMeta m,
                                                              __nv_bfloat16* bias) {
  pdl_begin();
  constexpr int C = 16 * NK;
  __shared__ __nv_bfloat16 sW[4][C];        // W' rounded to bf16 (rows H .. 3 zero)
  __shared__ float c0[4], c1[4];
  for (int idx = threadIdx.x; idx < 4 * C; idx += 256) {
    const int h = idx / C, c = idx - h * C;
    sW[h][c] = __float2bfloat16_rn(h < H ? __bfloat162float(Wb[h * C + c]) * __bfloat162float(gamma[c]) : 0.f);
  }
  __syncthreads();
  if ((threadIdx.x >> 5) < 4) {
    const int h = threadIdx.x >> 5;
    float a0 = 0.f, a1 = 0.f;
    for (int c = threadIdx.x & 31; c < C; c += 32) {
      if (h < H) a0 = fmaf(__bfloat162float(Wb[h * C + c]), __bfloat162float(beta[c]), a0);
      a1 += __bfloat162float(sW[h][c]);
    }
#pragma unroll
    for (int o = 16; o; o >>= 1) {
      a0 += __shfl_xor_sync(0xffffffffu, a0, o);
      a1 += __shfl_xor_sync(0xffffffffu, a1, o);
    }
    if ((threadIdx.x & 31) == 0) { c0[h] = a0; c1[h] = a1; }
  }
  __syncthreads();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  // B fragments: column n = g of the MMA is head g (g < 4), the ones column (g == 4) or zero
  unsigned bw[NK][2];
#pragma unroll
  for (int ks = 0; ks < NK; ++ks) {
    if (g < 4) {
      const int ch = (ks >> 1) * 32 + t * 8 + (ks & 1) * 4;
      bw[ks][0] = *reinterpret_cast<const unsigned*>(&sW[g][ch]);
      bw[ks][1] = *reinterpret_cast<const unsigned*>(&sW[g][ch + 2]);
    } else {
      bw[ks][0] = bw[ks][1] = g == 4 ? 0x3F803F80u : 0u;
    }
  }
  const unsigned bsq = g == 5 ? 0x3F803F80u : 0u;
  const float k0a = c0[(2 * t) & 3], k0b = c0[(2 * t + 1) & 3], k1a = c1[(2 * t) & 3], k1b = c1[(2 * t + 1) & 3];
  const long long p0 = m.pair_off[0], p1 = m.pair_off[m.B];
  const long long ntile = (p1 - p0 + 15) / 16;
  const long long step = (long long)gridDim.x * 8;
  uint4 va[NK / 2], vb[NK / 2];
  auto load = [&](long long tile) {
    const long long pa = p0 + tile * 16 + g, pb = pa + 8;
    const __nv_bfloat16* ra = z + (pa < p1 ? pa : p1 - 1) * C + 8 * t;
    const __nv_bfloat16* rb = z + (pb < p1 ? pb : p1 - 1) * C + 8 * t;
#pragma unroll
    for (int kb = 0; kb < NK / 2; ++kb) {
      va[kb] = *reinterpret_cast<const uint4*>(ra + kb * 32);
      vb[kb] = *reinterpret_cast<const uint4*>(rb + kb * 32);
    }
  };
  long long tile = (long long)blockIdx.x * 8 + warp;
  if (tile < ntile) load(tile);
  for (; tile < ntile; tile += step) {
    const long long pa = p0 + tile * 16 + g, pb = pa + 8;
    float acc[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int ks = 0; ks < NK; ++ks) {
      const uint4 x = va[ks >> 1], y = vb[ks >> 1];
      const unsigned a[4] = {ks & 1 ? x.z : x.x, ks & 1 ? y.z : y.x, ks & 1 ? x.w : x.y, ks & 1 ? y.w : y.y};
      mma_bf16_16816(acc, a, bw[ks][0], bw[ks][1]);
      unsigned sq[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const __nv_bfloat162 v = *reinterpret_cast<const __nv_bfloat162*>(&a[e]);
        const __nv_bfloat162 v2 = __hmul2(v, v);
        sq[e] = *reinterpret_cast<const unsigned*>(&v2);
      }
      mma_bf16_16816(acc, sq, bsq, bsq);
    }
    if (tile + step < ntile) load(tile + step);            // under the statistics and the stores of this tile
    // columns 4 / 5 (lanes with t == 2) hold the row sum and the sum of squares
    const int src = (lane & ~3) | 2;
    const float sa = __shfl_sync(0xffffffffu, acc[0], src), qa = __shfl_sync(0xffffffffu, acc[1], src);
    const float sb = __shfl_sync(0xffffffffu, acc[2], src), qb = __shfl_sync(0xffffffffu, acc[3], src);
    if (t < 2) {
      const float ma = sa / (float)C, mb = sb / (float)C;
      const float rsa = rsqrtf(fmaxf(qa / (float)C - ma * ma, 0.f) + eps), rsb = rsqrtf(fmaxf(qb / (float)C - mb * mb, 0.f) + eps);
      const float out[2][2] = {{(rsa * (acc[0] - ma * k1a) + k0a) * scale, (rsa * (acc[1] - ma * k1b) + k0b) * scale},
                               {(rsb * (acc[2] - mb * k1a) + k0a) * scale, (rsb * (acc[3] - mb * k1b) + k0b) * scale}};
#pragma unroll
      for (int rr = 0; rr < 2; ++rr) {
        const long long p = rr ? pb : pa;
        if (p < p1) {
          const int s_ = find_sample(m.pair_off, m.B, p);
          const int N = m.N[s_], ld = round_up8(N);
          const long long r = p - m.pair_off[s_];
          const int i = r >> 32 ? (int)(r / N) : (int)((unsigned)r / (unsigned)N), j = (int)(r - (long long)i * N);
          __nv_bfloat16* bp = bias + (long long)H * m.cm_off[s_] + (long long)i * ld + j;
          if (2 * t < H) bp[(long long)(2 * t) * N * ld] = __float2bfloat16_rn(out[rr][0]);
          if (2 * t + 1 < H) bp[(long long)(2 * t + 1) * N * ld] = __float2bfloat16_rn(out[rr][1]);
        }
      }
    }
  }
}

bool fast_single_attn_supported(int c_s, int c_z, int H, int d) {
  const int Hd = H * d;
  return c_s % 8 == 0 && c_s <= 2048 && c_z % 8 == 0 && c_z <= 1024 && H >= 1 && H <= SB_MAXH && fast_attn_fr_supported(H, d) &&
         fast_token_gemm_supported(c_s, Hd, Hd) && fast_token_gemm_supported(Hd, c_s, 0);
}

nt_status fast_ln_rows(const void* x, const void* g, const void* b, float eps, int C, long long rows, void* out, cudaStream_t st,
                       const char* name) {
  if (rows <= 0) return NT_OK;
  {
    LaunchScope ls(name, st);
    launch_kernel(ln_rows_kernel, (unsigned)((rows + 7) / 8), 256, 0, st, (const __nv_bfloat16*)x, (const __nv_bfloat16*)g, (const __nv_bfloat16*)b, eps, C,
                                                               rows, (__nv_bfloat16*)out);
  }
  return cuda_ok("single attention LayerNorm launch");
}

nt_status fast_gate_mul(const void* g, void* o, long long n, cudaStream_t st, const char* name) {
  if (n <= 0) return NT_OK;
  const long long n8 = n / 8;
  {
    LaunchScope ls(name, st);
    launch_kernel(gate_mul_kernel, (unsigned)((n8 + 255) / 256), 256, 0, st, (const __nv_bfloat16*)g, (__nv_bfloat16*)o, n8);
  }
  return cuda_ok("single attention gate launch");
}

nt_status fast_single_bias(const void* z, const void* g, const void* b, const void* Wb, float eps, int C, int H, float scale,
                           const BatchMeta& m, void* bias, cudaStream_t st) {
  const long long rows = m.pair_off[m.B] - m.pair_off[0];
  if (rows <= 0) return NT_OK;
  const long long nblk = (rows + 31) / 32;
  const long long want = (nblk + 7) / 8;
  const unsigned grid = (unsigned)(want < sm_count() * 3 ? want : sm_count() * 3);      // 3 blocks of 256 threads fit an SM at 79 registers
  if (H <= 4 && (C == 128 || C == 64)) {
    const long long ntile = (rows + 15) / 16, wantb = (ntile + 7) / 8;
    const unsigned gridm = (unsigned)(wantb < sm_count() * 3 ? wantb : sm_count() * 3);      // what is resident at 80 registers
    {
      LaunchScope ls("single_attn_bias", st);
      if (C == 128)
        launch_kernel(single_bias_mma_kernel<8>, gridm, 256, 0, st, (const __nv_bfloat16*)z, (const __nv_bfloat16*)g, (const __nv_bfloat16*)b,
                                                         (const __nv_bfloat16*)Wb, eps, H, scale, m, (__nv_bfloat16*)bias);
      else
        launch_kernel(single_bias_mma_kernel<4>, gridm, 256, 0, st, (const __nv_bfloat16*)z, (const __nv_bfloat16*)g, (const __nv_bfloat16*)b,
                                                         (const __nv_bfloat16*)Wb, eps, H, scale, m, (__nv_bfloat16*)bias);
    }
    return cuda_ok("single attention bias launch");
  }
  const int HT = H <= 4 ? 4 : SB_MAXH;
  const size_t smem = ((size_t)HT * C + 2 * SB_MAXH) * sizeof(float);
  {
    LaunchScope ls("single_attn_bias", st);
    if (HT == 4)
      launch_kernel(single_bias_kernel<4>, grid, 256, smem, st, (const __nv_bfloat16*)z, (const __nv_bfloat16*)g, (const __nv_bfloat16*)b,
                                                     (const __nv_bfloat16*)Wb, eps, C, H, scale, m, (__nv_bfloat16*)bias);
    else
      launch_kernel(single_bias_kernel<8>, grid, 256, smem, st, (const __nv_bfloat16*)z, (const __nv_bfloat16*)g, (const __nv_bfloat16*)b,
                                                     (const __nv_bfloat16*)Wb, eps, C, H, scale, m, (__nv_bfloat16*)bias);
  }
  return cuda_ok("single attention bias launch");
}

}  // namespace ntp
