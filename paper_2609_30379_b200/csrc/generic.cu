// Shape-generic CUDA-core kernels: tiled projection with LayerNorm / gate prologues and
// row-major or channel-major epilogues (several outputs of the same rows in one launch), the
// per-(sample, channel) triangle contraction, the gather + LayerNorm broadcast, an online-softmax
// attention core and the segmented reduction.
#include "generic.cuh"

namespace ntp {

// four consecutive elements as floats
__device__ inline float4 ld4(const float* p) { return *reinterpret_cast<const float4*>(p); }
__device__ inline float4 ld4(const __nv_bfloat16* p) {
  const uint2 w = *reinterpret_cast<const uint2*>(p);
  return make_float4(__uint_as_float(w.x << 16), __uint_as_float(w.x & 0xffff0000u), __uint_as_float(w.y << 16), __uint_as_float(w.y & 0xffff0000u));
}
__device__ inline void st4(float* p, float4 v) { *reinterpret_cast<float4*>(p) = v; }
__device__ inline void st4(__nv_bfloat16* p, float4 v) {
  __nv_bfloat162 lo = __floats2bfloat162_rn(v.x, v.y), hi = __floats2bfloat162_rn(v.z, v.w);
  *reinterpret_cast<uint2*>(p) = make_uint2(*reinterpret_cast<unsigned*>(&lo), *reinterpret_cast<unsigned*>(&hi));
}
// elements k .. k + 3 of a row of K (zero past the end); vec: rows are aligned for four elements at a time
template <typename T>
__device__ inline float4 ld4_row(const T* row, int k, int K, bool vec) {
  if (vec && k + 3 < K) return ld4(row + k);
  float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
  if (k < K) v.x = Cvt<T>::ld(row + k);
  if (k + 1 < K) v.y = Cvt<T>::ld(row + k + 1);
  if (k + 2 < K) v.z = Cvt<T>::ld(row + k + 2);
  if (k + 3 < K) v.w = Cvt<T>::ld(row + k + 3);
  return v;
}

// ------------------------------------------------------------------------------------------
// projection: 64 rows x 64 output columns at a time, K in panels of 32.  The column tiles of all outputs that share their
// rows are one launch; a block takes one of them where there are few rows (the smallest states are latency and nothing
// else) and more where the rows alone fill the GPU: the rows are then read and normalised less often.  Rows of up to 64
// elements are normalised in shared memory, the next panel is in registers while one is worked on, and results leave
// through shared memory in a rolled loop.  The loops are rolled on purpose: on a state of 531 rows a fully unrolled
// kernel spent its time fetching instructions (17 us a launch for 1500 to 2200 instructions per warp, two thirds of the
// stalls "no instruction").  VEC: rows of A and W can be read four elements at a time.
// ------------------------------------------------------------------------------------------
constexpr int PBM = 64, PBN = 64, PBK = 32, PTHREADS = 256, PPITCH = PBM + 4;
constexpr int PKA = 64;         // A tiles of up to this many columns stay in shared memory for all of a block's column tiles
constexpr int PSMALL = 8;       // outputs of up to this many columns: one column per thread instead of a 4 x 4 patch
constexpr int PTILE = 64 * PPITCH;
constexpr size_t PSMEM = (size_t)3 * PTILE * sizeof(float);    // A tile | W1 and W2 panels (results later) | gated values

__device__ inline float sigmoidf_acc(float x) { return 1.0f / (1.0f + expf(-x)); }

template <typename T, bool VEC>
__device__ inline float4 ld4_k(const T* row, int k, int K) {
  if (VEC) return k < K ? ld4(row + k) : make_float4(0.f, 0.f, 0.f, 0.f);
  return ld4_row(row, k, K, false);
}

template <typename T, bool VEC>
__global__ void __launch_bounds__(PTHREADS, 3) proj_kernel(const __grid_constant__ ProjArgs a, const __grid_constant__ BatchMeta m,
                                                           int tiles, int tiles_per_block) {
  pdl_begin();
  extern __shared__ __align__(16) float psmem[];
  float* As = psmem;                           // [k][row]
  float* Ws = psmem + PTILE;                   // W1 [32][column] | W2 [32][column]; afterwards the result tile
  float* Gs = psmem + 2 * PTILE;               // the second factor of a gated result
  __shared__ float mu[PBM], rstd[PBM];
  __shared__ long long cmbase[PBM], inpl[PBM], plane[PBM];

  const int t = threadIdx.x;
  const long long r0 = a.row0 + (long long)blockIdx.x * PBM;
  const int rows = (int)min((long long)PBM, a.row0 + a.rows - r0);
  int sg = 0, n0 = 0;
  const int tile0 = blockIdx.y * tiles_per_block, tile1 = min(tiles, tile0 + tiles_per_block);
  for (int skip = tile0; skip > 0; --skip) {
    n0 += PBN;
    if (n0 >= a.seg[sg].Nout) { n0 = 0; ++sg; }
  }
  const T* A = (const T*)a.A + (a.a_mode == A_ROWMAJOR ? r0 * a.K : 0);
  const T* gA = a.gateA ? (const T*)a.gateA + r0 * a.K : nullptr;
  const T* lng = (const T*)a.ln_g;
  const T* lnb = (const T*)a.ln_b;
  const int K = a.K;
  const bool rowmajor = a.a_mode == A_ROWMAJOR, has_ln = lng != nullptr, resident = K <= PKA;

  if (a.need_pos && t < rows) {                // where the block's positions lie in channel-major buffers
    const long long p = r0 + t;
    const int s = find_sample(m.pair_off, m.B, p);
    const int N = m.N[s], ld = round_up8(N);
    const unsigned long long r = (unsigned long long)(p - m.pair_off[s]);
    unsigned long long i;
    if (r >> 32) i = r / (unsigned)N;
    else i = (unsigned)r / (unsigned)N;
    cmbase[t] = m.cm_off[s];
    plane[t] = (long long)N * ld;
    inpl[t] = (long long)i * ld + (long long)(r - i * N);
  }
  if (!rowmajor) __syncthreads();

  if (has_ln && !resident) {                   // two-pass row statistics from memory
    float (*part)[PBM] = reinterpret_cast<float (*)[PBM]>(As);
    const int rl = rowmajor ? t >> 2 : t & 63, pt = rowmajor ? t & 3 : t >> 6;      // four threads per row
    const bool in = rl < rows;
    const T* Ar = rowmajor ? A + (in ? (long long)rl * K : 0) : A + (in ? (long long)K * cmbase[rl] + inpl[rl] : 0);
    const T* Gr = gA ? gA + (in ? (long long)rl * K : 0) : nullptr;
    const long long step = rowmajor ? 1 : in ? plane[rl] : 0;
    float s = 0.f, q = 0.f;
#pragma unroll 4
    for (int k = pt; k < K; k += 4) s += Cvt<T>::ld(Ar + k * step) * (Gr ? Cvt<T>::ld(Gr + k) : 1.f);
    part[pt][rl] = s;
    __syncthreads();
    const float mean = ((part[0][rl] + part[1][rl]) + (part[2][rl] + part[3][rl])) / (float)K;
#pragma unroll 4
    for (int k = pt; k < K; k += 4) {
      const float d = Cvt<T>::ld(Ar + k * step) * (Gr ? Cvt<T>::ld(Gr + k) : 1.f) - mean;
      q += d * d;
    }
    part[4 + pt][rl] = q;
    __syncthreads();
    if (pt == 0) {
      mu[rl] = mean;
      rstd[rl] = rsqrtf(((part[4][rl] + part[5][rl]) + (part[6][rl] + part[7][rl])) / (float)K + a.eps);
    }
    __syncthreads();
  }

  // panel loads: thread -> (row, 4 + 4 elements of K) of A (row-major) and W; channel-major A: (position, 8 channels)
  const int lr = t >> 2, lk = (t & 3) * 4;
  const int cr = t & 63, ck = (t >> 6) * 8;
  float4 ra[2], rw[2][2];
  const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
  auto load_a = [&](int k0) {
    if (rowmajor) {
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const int k = k0 + lk + 16 * u;
        ra[u] = lr < rows ? ld4_k<T, VEC>(A + (long long)lr * K, k, K) : zero;
        if (gA && lr < rows) {
          const float4 gv = ld4_k<T, VEC>(gA + (long long)lr * K, k, K);
          ra[u] = make_float4(ra[u].x * gv.x, ra[u].y * gv.y, ra[u].z * gv.z, ra[u].w * gv.w);
        }
      }
    } else {
      float v[8];
      const T* Ar = A + (cr < rows ? (long long)K * cmbase[cr] + inpl[cr] : 0);
      const long long pl = cr < rows ? plane[cr] : 0;
#pragma unroll
      for (int u = 0; u < 8; ++u) v[u] = cr < rows && k0 + ck + u < K ? Cvt<T>::ld(Ar + (k0 + ck + u) * pl) : 0.f;
      ra[0] = make_float4(v[0], v[1], v[2], v[3]);
      ra[1] = make_float4(v[4], v[5], v[6], v[7]);
    }
  };
  auto load_w = [&](int k0) {
    const int n = n0 + lr;
    const T* w1 = (const T*)a.seg[sg].W1 + (long long)n * K;
    const T* w2 = (const T*)a.seg[sg].W2 + (long long)n * K;
    const bool in = n < a.seg[sg].Nout, two = a.seg[sg].W2 != nullptr;
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      rw[0][u] = in ? ld4_k<T, VEC>(w1, k0 + lk + 16 * u, K) : zero;
      rw[1][u] = in && two ? ld4_k<T, VEC>(w2, k0 + lk + 16 * u, K) : zero;
    }
  };
  auto put_a = [&](int k0, int at, bool ln) {
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const float av[4] = {ra[u].x, ra[u].y, ra[u].z, ra[u].w};
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const int row = rowmajor ? lr : cr, kk = rowmajor ? lk + 16 * u + e : ck + 4 * u + e, k = k0 + kk;
        float v = av[e];
        if (ln && k < K) v = (v - mu[row]) * rstd[row] * Cvt<T>::ld(lng + k) + Cvt<T>::ld(lnb + k);
        As[(at + kk) * PPITCH + row] = v;
      }
    }
  };
  auto put_w = [&](bool two) {
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const float w1[4] = {rw[0][u].x, rw[0][u].y, rw[0][u].z, rw[0][u].w};
      const float w2[4] = {rw[1][u].x, rw[1][u].y, rw[1][u].z, rw[1][u].w};
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        Ws[(lk + 16 * u + e) * PPITCH + lr] = w1[e];
        if (two) Ws[(PBK + lk + 16 * u + e) * PPITCH + lr] = w2[e];
      }
    }
  };
  load_a(0);
  load_w(0);
  if (resident) {                              // the whole A tile; its LayerNorm in shared memory, four threads per row
    put_a(0, 0, false);
    if (K > PBK) {
      load_a(PBK);
      put_a(PBK, PBK, false);
    }
    __syncthreads();
    if (has_ln) {
      const int rl = t >> 2, pt = t & 3;
      float s = 0.f, q = 0.f;
#pragma unroll 4
      for (int k = pt; k < K; k += 4) s += As[k * PPITCH + rl];
      s += __shfl_xor_sync(0xffffffffu, s, 1);
      s += __shfl_xor_sync(0xffffffffu, s, 2);
      const float mean = s / (float)K;
#pragma unroll 4
      for (int k = pt; k < K; k += 4) {
        const float d = As[k * PPITCH + rl] - mean;
        q += d * d;
      }
      q += __shfl_xor_sync(0xffffffffu, q, 1);
      q += __shfl_xor_sync(0xffffffffu, q, 2);
      const float rs = rsqrtf(q / (float)K + a.eps);
#pragma unroll 4
      for (int k = pt; k < K; k += 4) As[k * PPITCH + rl] = (As[k * PPITCH + rl] - mean) * rs * Cvt<T>::ld(lng + k) + Cvt<T>::ld(lnb + k);
    }
  }
  const int ty = t >> 4, tx = t & 15;
  const T* gO = (const T*)a.gateO;
#pragma unroll 1
  for (int tile = tile0; tile < tile1; ++tile) {
    const ProjSeg g = a.seg[sg];
    const bool small = g.Nout <= PSMALL && resident, gated = g.W2 != nullptr;
    const int nt0 = n0;                      // first column of this tile (n0 moves on while the tile is worked on)
    float acc1[4][4] = {}, acc2[4][4] = {};
#pragma unroll 1
    for (int k0 = 0; k0 < K; k0 += PBK) {
      const bool last = k0 + PBK >= K;
      if (!resident) put_a(k0, 0, has_ln);
      put_w(gated);
      __syncthreads();
      if (last && tile + 1 < tile1) {        // the next tile's first panel
        n0 += PBN;
        if (n0 >= g.Nout) { n0 = 0; ++sg; }
        load_w(0);
        if (!resident) load_a(0);
      } else if (!last) {
        load_w(k0 + PBK);
        if (!resident) load_a(k0 + PBK);
      }
      const int kmax = (min(K - k0, PBK) + 3) & ~3;      // (the panels are zero beyond K)
      const float* Ak = As + (resident ? k0 : 0) * PPITCH;
      if (small) {                           // column t / 64 (and + 4) of row t % 64
        const float *ap = Ak + (t & 63), *wp = Ws + (t >> 6);
#pragma unroll 4
        for (int kk = 0; kk < kmax; ++kk, ap += PPITCH, wp += PPITCH) {
          acc1[0][0] = fmaf(*ap, wp[0], acc1[0][0]);
          acc1[0][1] = fmaf(*ap, wp[4], acc1[0][1]);
          if (gated) {
            acc2[0][0] = fmaf(*ap, wp[PBK * PPITCH], acc2[0][0]);
            acc2[0][1] = fmaf(*ap, wp[PBK * PPITCH + 4], acc2[0][1]);
          }
        }
      } else {
        const float *ap = Ak + ty * 4, *wp = Ws + tx * 4;
#pragma unroll 4
        for (int kk = 0; kk < kmax; ++kk, ap += PPITCH, wp += PPITCH) {
          const float4 av = *reinterpret_cast<const float4*>(ap);
          const float4 wv = *reinterpret_cast<const float4*>(wp);
          const float ar[4] = {av.x, av.y, av.z, av.w};
          const float wr[4] = {wv.x, wv.y, wv.z, wv.w};
#pragma unroll
          for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) acc1[i][j] = fmaf(ar[i], wr[j], acc1[i][j]);
          if (gated) {
            const float4 w2 = *reinterpret_cast<const float4*>(wp + PBK * PPITCH);
            const float w2r[4] = {w2.x, w2.y, w2.z, w2.w};
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
              for (int j = 0; j < 4; ++j) acc2[i][j] = fmaf(ar[i], w2r[j], acc2[i][j]);
          }
        }
      }
      __syncthreads();
    }
    // results to shared memory, the faster index of the output innermost, then out in order
    const bool cm = g.out_mode == O_CHANNEL_MAJOR;
    const int si = cm ? 1 : PPITCH, sj = cm ? PPITCH : 1;      // step of a row / of a column
    if (small) {
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        Ws[(t & 63) * si + ((t >> 6) + 4 * u) * sj] = acc1[0][u];
        if (gated) Gs[(t & 63) * si + ((t >> 6) + 4 * u) * sj] = acc2[0][u];
      }
    } else {
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          Ws[(ty * 4 + i) * si + (tx * 4 + j) * sj] = acc1[i][j];
          if (gated) Gs[(ty * 4 + i) * si + (tx * 4 + j) * sj] = acc2[i][j];
        }
    }
    __syncthreads();
    const int ncol = min(PBN, g.Nout - nt0);
    const int total = cm ? ncol * PBM : rows * PBN;
    const bool accum = g.out_mode == O_ACCUM;
    auto emit = [&](int idx, bool have, float old) {          // result idx; have: its old value has been fetched
      const int hi = idx >> 6, lo = idx & 63, rl = cm ? lo : hi, n = nt0 + (cm ? hi : lo);
      if (rl >= rows || n >= g.Nout) return;
      const long long p = r0 + rl;
      float v = Ws[hi * PPITCH + lo];
      if (gated) v = (g.act == ACT_SILU ? v * sigmoidf_acc(v) : sigmoidf_acc(v)) * Gs[hi * PPITCH + lo];
      else if (g.act == ACT_SIGMOID) v = sigmoidf_acc(v);
      if (cm) {
        const long long at = (long long)g.Nout * cmbase[rl] + (long long)n * plane[rl] + inpl[rl];
        if (NT_IN(at, (long long)g.Nout * m.cm_off[m.B], NT_SITE_PROJ_OUT)) Cvt<T>::st((T*)g.out + at, v);
        return;
      }
      if (!NT_IN(p, a.row0 + a.rows, NT_SITE_PROJ_OUT)) return;
      if (gO) v *= Cvt<T>::ld(gO + p * g.Nout + n);
      if (g.out_f32) {
        float* o = (float*)g.out + p * g.Nout + n;
        *o = accum ? (have ? old : *o) + v : v;
      } else {
        T* o = (T*)g.out + p * g.Nout + n;
        Cvt<T>::st(o, accum ? v + (have ? old : Cvt<T>::ld(o)) : v);
      }
    };
    // An output that is added to costs a trip to memory before each store; four are fetched at a time (402 float rows, 16 -> 32:
    // 10.6 -> 7.4 us, 8.4 with everything unrolled; bf16, 96 -> 100: 17.5 -> 15.3, 16.5 unrolled).  In a loop of its own: outputs that are
    // only stored lost 0.8 us to the longer code.
    if (accum && !g.out_f32) {
      float old[4] = {};
#pragma unroll 1
      for (int idx0 = t; idx0 < total; idx0 += 4 * PTHREADS) {
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int rl = (idx0 + u * PTHREADS) >> 6, n = nt0 + ((idx0 + u * PTHREADS) & 63);
          if (rl < rows && n < g.Nout) old[u] = Cvt<T>::ld((const T*)g.out + (r0 + rl) * g.Nout + n);
        }
#pragma unroll
        for (int u = 0; u < 4; ++u)
          if (idx0 + u * PTHREADS < total) emit(idx0 + u * PTHREADS, true, old[u]);
      }
    } else {
#pragma unroll 2
      for (int idx = t; idx < total; idx += PTHREADS) emit(idx, false, 0.f);
    }
    __syncthreads();
  }
}

template <typename T, bool VEC>
static nt_status run_proj(const ProjArgs& a, const BatchMeta& m, dim3 grid, int tiles, int tpb, cudaStream_t st) {
  static bool attr_set[64] = {};
  int dev = 0;
  cudaGetDevice(&dev);
  if (!attr_set[dev & 63]) {
    if (cudaFuncSetAttribute(proj_kernel<T, VEC>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)PSMEM) != cudaSuccess)
      return cuda_fail("projection smem attribute");
    attr_set[dev & 63] = true;
  }
  launch_kernel(proj_kernel<T, VEC>, grid, PTHREADS, PSMEM, st, a, m, tiles, tpb);
  return NT_OK;
}

template <typename T>
nt_status launch_proj(const ProjArgs& args, const BatchMeta& m, cudaStream_t st, const char* name) {
  ProjArgs a = args;
  long long tiles = 0;
  uintptr_t low = (uintptr_t)a.A | (uintptr_t)a.gateA;
  a.need_pos = a.a_mode != A_ROWMAJOR;
  for (int s = 0; s < a.nseg; ++s) {
    tiles += (a.seg[s].Nout + PBN - 1) / PBN;
    low |= (uintptr_t)a.seg[s].W1 | (uintptr_t)a.seg[s].W2;
    if (a.seg[s].out_mode == O_CHANNEL_MAJOR) a.need_pos = 1;
  }
  if (a.rows <= 0 || tiles <= 0) return NT_OK;
  long long bx = (a.rows + PBM - 1) / PBM;
  if (bx > 0x7FFFFFFFll || tiles > 65535) return NT_ERR_UNSUPPORTED;
  // Column tiles per block: the number for which the blocks' rounds take least.  A block costs its tiles (between the most and
  // the average, where they do not divide evenly) and a little for its rows and their LayerNorm; three blocks fit an SM, and
  // an SM with one or two left works at 0.6 or 0.9 of its rate, so a last round of up to one, two or three blocks per SM
  // takes 1.6, 2.3 or 3 block times.  Fitted to the times of every tile count (widths 40 to 256, 1 to 16 tiles, 256 to 160 k rows,
  // float and bf16; 984 launches): 1.5 % from the best choice on average, 15 % at worst.  (One tile per block up to two blocks per
  // SM and whole rounds beyond that: 6 %, 56 %, and 31 % slower than a block per tile for a hidden layer of 1024 on 14400 rows.)
  const long long sms = sm_count();
  int tpb = 1;
  double best = 1e300;
  for (int k = 1; k <= tiles; ++k) {
    const long long y = (tiles + k - 1) / k, n = bx * y, rounds = n / (3 * sms), rest = n - rounds * 3 * sms;
    const double last = rest == 0 ? 0.0 : rest <= sms ? 1.6 : rest <= 2 * sms ? 2.3 : 3.0;
    const double cost = (3.0 * (double)rounds + last) * (0.15 + 0.75 * (double)tiles / (double)y + 0.25 * k);
    if (cost < best) { best = cost; tpb = k; }
  }
  const dim3 grid((unsigned)bx, (unsigned)((tiles + tpb - 1) / tpb));
  const bool vec = (a.K & 3) == 0 && (low & 15) == 0;      // (not every entry point asks for aligned weights)
  nt_status r;
  {
    LaunchScope ls(name, st);
    r = vec ? run_proj<T, true>(a, m, grid, (int)tiles, tpb, st) : run_proj<T, false>(a, m, grid, (int)tiles, tpb, st);
  }
  return r != NT_OK ? r : cuda_ok();
}
template nt_status launch_proj<float>(const ProjArgs&, const BatchMeta&, cudaStream_t, const char*);
template nt_status launch_proj<__nv_bfloat16>(const ProjArgs&, const BatchMeta&, cudaStream_t, const char*);

// ------------------------------------------------------------------------------------------
// triangle contraction  t[c][i][j] = sum_k a[c][i][k] b[c][j][k]   (outgoing)
//                       t[c][i][j] = sum_k a[c][k][i] b[c][k][j]   (incoming)
// 64 x 64 tiles; the operands arrive four elements at a time (rows start on multiples of 8 elements) and the next panel is
// in registers while one is worked on.
// ------------------------------------------------------------------------------------------
constexpr int CT = 64, CK = 32;

template <typename T>
__global__ void __launch_bounds__(256) contract_kernel(const T* a, const T* b,
                                                      T* tout, int C, BatchMeta m, int incoming) {
  pdl_begin();
  __shared__ __align__(16) float As[CK][CT + 4];
  __shared__ __align__(16) float Bs[CK][CT + 4];
  long long w = blockIdx.x;
  int s = 0, nt = 0;
  for (; s < m.B; ++s) {   // tile -> sample
    nt = (m.N[s] + CT - 1) / CT;
    long long cnt = (long long)C * nt * nt;
    if (w < cnt) break;
    w -= cnt;
  }
  if (s >= m.B) return;
  const int N = m.N[s], ld = round_up8(N);
  const int c = (int)(w / (nt * nt));
  const int rem = (int)(w - (long long)c * nt * nt);
  const int i0 = (rem / nt) * CT, j0 = (rem % nt) * CT;
  const long long base = (long long)C * m.cm_off[s] + (long long)c * N * ld;
  const T* Ap = a + base;
  const T* Bp = b + base;
  const int t = threadIdx.x, ty = t >> 4, tx = t & 15;
  // outgoing: thread -> (row t / 4, 4 + 4 elements of k); incoming: (k t / 16 and + 16, 4 elements of the row)
  const int lr = t >> 2, lk = (t & 3) * 4, ik = t >> 4, ir = (t & 15) * 4;
  float4 ra[2], rb[2];
  const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
  auto clip = [](float4 v, int left) {      // elements from `left` on are padding
    if (left < 4) v.w = 0.f;
    if (left < 3) v.z = 0.f;
    if (left < 2) v.y = 0.f;
    if (left < 1) v.x = 0.f;
    return v;
  };
  auto load = [&](int k0) {
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      if (incoming) {
        const int k = k0 + ik + 16 * u;
        ra[u] = k < N && i0 + ir < N ? clip(ld4(Ap + (long long)k * ld + i0 + ir), N - i0 - ir) : zero;
        rb[u] = k < N && j0 + ir < N ? clip(ld4(Bp + (long long)k * ld + j0 + ir), N - j0 - ir) : zero;
      } else {
        const int k = k0 + lk + 16 * u;
        ra[u] = k < N && i0 + lr < N ? clip(ld4(Ap + (long long)(i0 + lr) * ld + k), N - k) : zero;
        rb[u] = k < N && j0 + lr < N ? clip(ld4(Bp + (long long)(j0 + lr) * ld + k), N - k) : zero;
      }
    }
  };
  float acc[4][4] = {};
  load(0);
  for (int k0 = 0; k0 < N; k0 += CK) {
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      if (incoming) {
        *reinterpret_cast<float4*>(&As[ik + 16 * u][ir]) = ra[u];
        *reinterpret_cast<float4*>(&Bs[ik + 16 * u][ir]) = rb[u];
      } else {
        const float av[4] = {ra[u].x, ra[u].y, ra[u].z, ra[u].w}, bv[4] = {rb[u].x, rb[u].y, rb[u].z, rb[u].w};
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          As[lk + 16 * u + e][lr] = av[e];
          Bs[lk + 16 * u + e][lr] = bv[e];
        }
      }
    }
    __syncthreads();
    if (k0 + CK < N) load(k0 + CK);
    const int kmax = N - k0 < CK ? N - k0 : CK;
#pragma unroll 8
    for (int kk = 0; kk < kmax; ++kk) {
      const float4 av = *reinterpret_cast<const float4*>(&As[kk][ty * 4]);
      const float4 bv = *reinterpret_cast<const float4*>(&Bs[kk][tx * 4]);
      const float ar[4] = {av.x, av.y, av.z, av.w};
      const float br[4] = {bv.x, bv.y, bv.z, bv.w};
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(ar[i], br[j], acc[i][j]);
    }
    __syncthreads();
  }
  T* Tp = tout + base;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int ii = i0 + ty * 4 + i, jj = j0 + tx * 4;
    // (jj < N and ld a multiple of 8: the four columns lie inside the row, padding included)
    if (ii < N && jj < N && NT_IN(base + (long long)ii * ld + jj, (long long)C * m.cm_off[m.B], NT_SITE_CONTRACT_OUT))
      st4(Tp + (long long)ii * ld + jj, make_float4(acc[i][0], acc[i][1], acc[i][2], acc[i][3]));
  }
}

template <typename T>
nt_status launch_contract(const T* a, const T* b, T* t, int C, const BatchMeta& m, cudaStream_t st, bool incoming) {
  long long tiles = 0;
  for (int s = 0; s < m.B; ++s) {
    long long nt = (m.N[s] + CT - 1) / CT;
    tiles += (long long)C * nt * nt;
  }
  if (tiles == 0) return NT_OK;
  if (tiles > 0x7FFFFFFFll) return NT_ERR_UNSUPPORTED;
  {
    LaunchScope ls(incoming ? "generic_tri_contract_in" : "generic_tri_contract", st);
    launch_kernel(contract_kernel<T>, (unsigned)tiles, 256, 0, st, a, b, t, C, m, incoming ? 1 : 0);
  }
  return cuda_ok();
}
template nt_status launch_contract<float>(const float*, const float*, float*, int, const BatchMeta&, cudaStream_t, bool);
template nt_status launch_contract<__nv_bfloat16>(const __nv_bfloat16*, const __nv_bfloat16*, __nv_bfloat16*, int,
                                                  const BatchMeta&, cudaStream_t, bool);

// ------------------------------------------------------------------------------------------
// broadcast + LayerNorm (generic widths).  L = 4 .. 32 lanes per packed position, four channels per lane (L = 0: a warp
// per position, one channel per lane and step, for widths that are not a multiple of 4 or beyond 128).
// ------------------------------------------------------------------------------------------
template <typename T, int L>
__global__ void __launch_bounds__(256) broadcast_ln_kernel(const float* u, const float* v,
                                                          const T* gamma, const T* beta,
                                                          float eps, int c_z, T* z, BatchMeta m, int accumulate) {
  pdl_begin();
  constexpr int W = L ? L : 32;
  const int lane = threadIdx.x % W;
  const long long p = m.pair_off[0] + (long long)blockIdx.x * (256 / W) + threadIdx.x / W;
  const bool live = p < m.pair_off[m.B];
  const int s = live ? find_sample(m.pair_off, m.B, p) : 0;
  const unsigned N = live ? (unsigned)m.N[s] : 1u;
  const long long r = live ? p - m.pair_off[s] : 0;
  const long long i = r / N, j = r - i * N;
  const float* ur = u + (live ? m.tok_off[s] + i : 0) * c_z;
  const float* vr = v + (live ? m.tok_off[s] + j : 0) * c_z;
  T* zr = z + p * c_z;
  const bool ok = live && NT_IN(m.tok_off[s] + i, m.tok_off[m.B], NT_SITE_BROADCAST_OUT) && NT_IN(m.tok_off[s] + j, m.tok_off[m.B], NT_SITE_BROADCAST_OUT);
  if (L) {
    const int c = lane * 4;
    const bool has = ok && c < c_z;
    float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
    if (has) {
      const float4 uu = ld4(ur + c), vv = ld4(vr + c);
      x = make_float4(uu.x + vv.x, uu.y + vv.y, uu.z + vv.z, uu.w + vv.w);
    }
    float sum = (x.x + x.y) + (x.z + x.w);
#pragma unroll
    for (int o = W / 2; o; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
    const float mean = sum / (float)c_z;
    const float4 d = make_float4(x.x - mean, x.y - mean, x.z - mean, x.w - mean);
    float q = has ? (d.x * d.x + d.y * d.y) + (d.z * d.z + d.w * d.w) : 0.f;
#pragma unroll
    for (int o = W / 2; o; o >>= 1) q += __shfl_xor_sync(0xffffffffu, q, o);
    if (!has) return;
    const float rs = rsqrtf(q / (float)c_z + eps);
    const float4 g = ld4(gamma + c), be = ld4(beta + c);
    float4 y = make_float4(d.x * rs * g.x + be.x, d.y * rs * g.y + be.y, d.z * rs * g.z + be.z, d.w * rs * g.w + be.w);
    if (accumulate) {
      const float4 b = ld4(zr + c);
      y = make_float4(y.x + b.x, y.y + b.y, y.z + b.z, y.w + b.w);
    }
    st4(zr + c, y);
    return;
  }
  if (!ok) return;      // (a whole warp)
  float sum = 0.f;
  for (int c = lane; c < c_z; c += 32) sum += ur[c] + vr[c];
#pragma unroll
  for (int o = 16; o; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
  const float mean = sum / (float)c_z;
  float q = 0.f;
  for (int c = lane; c < c_z; c += 32) {
    float dlt = ur[c] + vr[c] - mean;
    q += dlt * dlt;
  }
#pragma unroll
  for (int o = 16; o; o >>= 1) q += __shfl_xor_sync(0xffffffffu, q, o);
  const float rs = rsqrtf(q / (float)c_z + eps);
  for (int c = lane; c < c_z; c += 32)
    Cvt<T>::st(zr + c, (ur[c] + vr[c] - mean) * rs * Cvt<T>::ld(gamma + c) + Cvt<T>::ld(beta + c) + (accumulate ? Cvt<T>::ld(zr + c) : 0.f));
}

template <typename T, int L>
static void run_broadcast_ln(const float* u, const float* v, const T* gamma, const T* beta, float eps, int c_z, T* z,
                             const BatchMeta& m, cudaStream_t st, bool accumulate, long long npos) {
  const int per = 256 / (L ? L : 32);
  launch_kernel(broadcast_ln_kernel<T, L>, (unsigned)((npos + per - 1) / per), 256, 0, st, u, v, gamma, beta, eps, c_z, z, m, accumulate ? 1 : 0);
}

template <typename T>
nt_status launch_broadcast_ln(const float* u, const float* v, const T* gamma, const T* beta, float eps, int c_z,
                              T* z, const BatchMeta& m, cudaStream_t st, bool accumulate) {
  long long npos = m.pair_off[m.B] - m.pair_off[0];
  if (npos <= 0) return NT_OK;
  if (npos / 8 + 1 > 0x7FFFFFFFll) return NT_ERR_UNSUPPORTED;
  // four elements at a time need aligned gamma / beta (the entry points ask 16 bytes of the other arrays only)
  const bool vec = c_z % 4 == 0 && c_z <= 128 && (((uintptr_t)gamma | (uintptr_t)beta) & 15) == 0;
  {
    LaunchScope ls(accumulate ? "generic_broadcast_ln_add" : "generic_broadcast_ln", st);
    if (!vec) run_broadcast_ln<T, 0>(u, v, gamma, beta, eps, c_z, z, m, st, accumulate, npos);
    else if (c_z <= 16) run_broadcast_ln<T, 4>(u, v, gamma, beta, eps, c_z, z, m, st, accumulate, npos);
    else if (c_z <= 32) run_broadcast_ln<T, 8>(u, v, gamma, beta, eps, c_z, z, m, st, accumulate, npos);
    else if (c_z <= 64) run_broadcast_ln<T, 16>(u, v, gamma, beta, eps, c_z, z, m, st, accumulate, npos);
    else run_broadcast_ln<T, 32>(u, v, gamma, beta, eps, c_z, z, m, st, accumulate, npos);
  }
  return cuda_ok();
}
template nt_status launch_broadcast_ln<float>(const float*, const float*, const float*, const float*, float, int,
                                              float*, const BatchMeta&, cudaStream_t, bool);
template nt_status launch_broadcast_ln<__nv_bfloat16>(const float*, const float*, const __nv_bfloat16*,
                                                      const __nv_bfloat16*, float, int, __nv_bfloat16*,
                                                      const BatchMeta&, cudaStream_t, bool);

// ------------------------------------------------------------------------------------------
// attention core: a block per (attention row, head, block of queries), keys in chunks of 32 staged in shared memory and
// read by broadcast; LP lanes share a query (DC channels each, LP = 1 up to head dim 32) and keep its q, its accumulator
// and the running maximum and sum in registers; eight scores are taken between two looks at the maximum.  (One warp per
// query with the lanes over the keys read K with a stride of H d elements and V once per key and query: 1215 us for
// lengths 24-110 with 4 heads of 16 in float, 55 now.)
// pair_order: 0 = token segments, 1 = pair rows (queries and keys run along j of row i), 2 = pair columns (queries
// and keys run along the first index of column i; the bias of (query, key) is bias[key][query]).
// ------------------------------------------------------------------------------------------
constexpr int AT = 64;        // threads
constexpr int AKC = 32;       // keys per chunk
constexpr int AKS = 8;        // keys per softmax step
constexpr int AD_MAX = 128;   // head dim limit of the generic core

template <typename T, int DC, int LP>
__global__ void __launch_bounds__(AT) attn_core_kernel(const T* q, const T* k,
                                                       const T* v, const T* bias,
                                                       T* o, int H, int d, int pair_order,
                                                       BatchMeta m, float bias_scale) {
  pdl_begin();
  constexpr int DP = DC * LP, QB = AT / LP;
  __shared__ __align__(16) float Ks[AKC][DP], Vs[AKC][DP];
  long long w = blockIdx.x;
  int s = 0, N = 0, nqb = 0;
  for (; s < m.B; ++s) {
    N = m.N[s];
    nqb = (N + QB - 1) / QB;
    const long long cnt = (long long)(pair_order ? N : (N > 0 ? 1 : 0)) * H * nqb;
    if (w < cnt) break;
    w -= cnt;
  }
  if (s >= m.B) return;
  const int jb = (int)(w % nqb);
  const int h = (int)((w / nqb) % H);
  const long long i = w / ((long long)nqb * H);
  const long long base = pair_order == 1 ? m.pair_off[s] + i * N : pair_order == 2 ? m.pair_off[s] + i : m.tok_off[s];
  const long long step = pair_order == 2 ? N : 1;          // packed rows between consecutive queries / keys
  const int t = threadIdx.x, part = t % LP;
  const int j = jb * QB + t / LP;
  const bool active = j < N, vec = (d & 3) == 0;
  const bool warp_live = jb * QB + (t & ~31) / LP < N;
  const long long Hd = (long long)H * d;
  const int c0 = part * DC;                                // this lane's channels
  float2 qv[DC / 2], acc[DC / 2];                          // channel pairs: two products per instruction
#pragma unroll
  for (int e = 0; e < DC / 2; e += 2) {
    const float4 x = active ? ld4_row(q + (base + j * step) * Hd + h * d, c0 + 2 * e, d, vec) : make_float4(0.f, 0.f, 0.f, 0.f);
    qv[e] = make_float2(x.x, x.y);
    qv[e + 1] = make_float2(x.z, x.w);
    acc[e] = acc[e + 1] = make_float2(0.f, 0.f);
  }
  const int ld = round_up8(N);
  const T* plane = bias ? bias + (long long)H * m.cm_off[s] + (long long)h * N * ld : nullptr;
  const float scale = rsqrtf((float)d);
  float mrun = -INFINITY, lrun = 0.f;
  for (int k0 = 0; k0 < N; k0 += AKC) {
    if (k0) __syncthreads();
    for (int idx = t; idx < AKC * (DP / 4); idx += AT) {
      const int r = idx / (DP / 4), c = (idx - r * (DP / 4)) * 4;
      const bool in = k0 + r < N;
      const long long at = (base + (in ? k0 + r : 0) * step) * Hd + h * d;
      const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
      *reinterpret_cast<float4*>(&Ks[r][c]) = in ? ld4_row(k + at, c, d, vec) : zero;
      *reinterpret_cast<float4*>(&Vs[r][c]) = in ? ld4_row(v + at, c, d, vec) : zero;
    }
    __syncthreads();
    if (!warp_live) continue;
    const int lim = min(AKC, N - k0);
    for (int kk = 0; kk < lim; kk += AKS) {
      float sc[AKS], b[AKS];
#pragma unroll
      for (int x = 0; x < AKS; ++x) b[x] = 0.f;
      if (plane && active) {
        if (pair_order == 2) {
#pragma unroll
          for (int x = 0; x < AKS; ++x) b[x] = k0 + kk + x < N ? Cvt<T>::ld(plane + (long long)(k0 + kk + x) * ld + j) : 0.f;
        } else {      // (pad columns of a row are readable and masked below)
          const float4 b0 = ld4(plane + (long long)j * ld + k0 + kk), b1 = ld4(plane + (long long)j * ld + k0 + kk + 4);
          b[0] = b0.x; b[1] = b0.y; b[2] = b0.z; b[3] = b0.w; b[4] = b1.x; b[5] = b1.y; b[6] = b1.z; b[7] = b1.w;
        }
      }
      float mx = -INFINITY;
#pragma unroll
      for (int x = 0; x < AKS; ++x) {
        float2 d2[2] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
#pragma unroll
        for (int e = 0; e < DC / 2; e += 2) {
          const float4 kv = *reinterpret_cast<const float4*>(&Ks[kk + x][c0 + 2 * e]);
          d2[0] = __ffma2_rn(qv[e], make_float2(kv.x, kv.y), d2[0]);
          d2[1] = __ffma2_rn(qv[e + 1], make_float2(kv.z, kv.w), d2[1]);
        }
        float dot = (d2[0].x + d2[0].y) + (d2[1].x + d2[1].y);
#pragma unroll
        for (int of = 1; of < LP; of <<= 1) dot += __shfl_xor_sync(0xffffffffu, dot, of);
        sc[x] = kk + x < lim ? dot * scale + b[x] * bias_scale : -INFINITY;
        mx = fmaxf(mx, sc[x]);
      }
      const float mnew = fmaxf(mrun, mx);                 // (a step has at least one key: finite)
      const float corr = expf(mrun - mnew);               // first step: exp(-inf) = 0
      float sum = 0.f;
#pragma unroll
      for (int x = 0; x < AKS; ++x) {
        sc[x] = expf(sc[x] - mnew);
        sum += sc[x];
      }
      lrun = lrun * corr + sum;
      mrun = mnew;
      const float2 corr2 = make_float2(corr, corr);
#pragma unroll
      for (int e = 0; e < DC / 2; e += 2) {
        float2 y0 = __fmul2_rn(acc[e], corr2), y1 = __fmul2_rn(acc[e + 1], corr2);
#pragma unroll
        for (int x = 0; x < AKS; ++x) {
          const float4 vv = *reinterpret_cast<const float4*>(&Vs[kk + x][c0 + 2 * e]);
          const float2 p2 = make_float2(sc[x], sc[x]);
          y0 = __ffma2_rn(p2, make_float2(vv.x, vv.y), y0);
          y1 = __ffma2_rn(p2, make_float2(vv.z, vv.w), y1);
        }
        acc[e] = y0;
        acc[e + 1] = y1;
      }
    }
  }
  if (!active || !NT_IN(base + j * step, pair_order ? m.pair_off[m.B] : m.tok_off[m.B], NT_SITE_ATTN_OUT)) return;
  const float inv = 1.0f / lrun;
  T* orow = o + (base + j * step) * Hd + h * d;
#pragma unroll
  for (int e = 0; e < DC / 2; e += 2) {
    const int c = c0 + 2 * e;
    const float r[4] = {acc[e].x * inv, acc[e].y * inv, acc[e + 1].x * inv, acc[e + 1].y * inv};
    if (vec && c < d) {
      st4(orow + c, make_float4(r[0], r[1], r[2], r[3]));
    } else {
#pragma unroll
      for (int x = 0; x < 4; ++x)
        if (c + x < d) Cvt<T>::st(orow + c + x, r[x]);
    }
  }
}

template <typename T>
nt_status launch_attn_core(const T* q, const T* k, const T* v, const T* bias, T* o, int H, int d, int pair_order,
                           const BatchMeta& m, cudaStream_t st, float bias_scale) {
  if (d > AD_MAX) return NT_ERR_UNSUPPORTED;
  const int lp = d <= 32 ? 1 : d <= 64 ? 2 : 4, qb = AT / lp;
  long long blocks = 0;
  for (int s = 0; s < m.B; ++s) {
    const long long N = m.N[s], nqb = (N + qb - 1) / qb;
    blocks += (pair_order ? N : (N > 0 ? 1 : 0)) * H * nqb;
  }
  if (blocks == 0) return NT_OK;
  if (blocks > 0x7FFFFFFFll) return NT_ERR_UNSUPPORTED;
  {
    LaunchScope ls(pair_order == 2 ? "generic_attn_core_col" : "generic_attn_core", st);
    const unsigned g = (unsigned)blocks;
    if (d <= 8) launch_kernel(attn_core_kernel<T, 8, 1>, g, AT, 0, st, q, k, v, bias, o, H, d, pair_order, m, bias_scale);
    else if (d <= 16) launch_kernel(attn_core_kernel<T, 16, 1>, g, AT, 0, st, q, k, v, bias, o, H, d, pair_order, m, bias_scale);
    else if (d <= 32) launch_kernel(attn_core_kernel<T, 32, 1>, g, AT, 0, st, q, k, v, bias, o, H, d, pair_order, m, bias_scale);
    else if (d <= 64) launch_kernel(attn_core_kernel<T, 32, 2>, g, AT, 0, st, q, k, v, bias, o, H, d, pair_order, m, bias_scale);
    else launch_kernel(attn_core_kernel<T, 32, 4>, g, AT, 0, st, q, k, v, bias, o, H, d, pair_order, m, bias_scale);
  }
  return cuda_ok();
}
template nt_status launch_attn_core<float>(const float*, const float*, const float*, const float*, float*, int, int,
                                           int, const BatchMeta&, cudaStream_t, float);
template nt_status launch_attn_core<__nv_bfloat16>(const __nv_bfloat16*, const __nv_bfloat16*, const __nv_bfloat16*,
                                                   const __nv_bfloat16*, __nv_bfloat16*, int, int, int,
                                                   const BatchMeta&, cudaStream_t, float);

// ------------------------------------------------------------------------------------------
// segmented reduction (generic widths): one block per group
// ------------------------------------------------------------------------------------------
template <typename T>
__global__ void __launch_bounds__(256) segment_reduce_kernel(const T* v, T* out,
                                                            const int64_t* splits, int C, int mean) {
  pdl_begin();
  __shared__ float part[256];
  const long long g = blockIdx.x;
  const long long lo = splits[g], hi = splits[g + 1];
  const long long n = hi - lo;
  const float sc = (mean && n > 0) ? 1.0f / (float)n : 1.0f;
  const int t = threadIdx.x;
  if (C >= 256) {
    for (int c = t; c < C; c += 256) {
      // (eight loads in flight, one sum in order: a loop left to the compiler's unrolling kept one in flight, 210 us for twelve
      // groups of 512 rows of 768 floats, 35 so)
      const T* col = v + c;
      float acc = 0.f;
      long long r = lo;
      for (; r + 7 < hi; r += 8) {
        float x[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) x[u] = Cvt<T>::ld(col + (r + u) * C);
#pragma unroll
        for (int u = 0; u < 8; ++u) acc += x[u];
      }
      for (; r < hi; ++r) acc += Cvt<T>::ld(col + r * C);
      Cvt<T>::st(out + g * C + c, acc * sc);
    }
    return;
  }
  const int RS = 256 / C;
  const int ch = t % C, slot = t / C;
  float acc = 0.f;
  if (slot < RS) {
#pragma unroll 8
    for (long long r = lo + slot; r < hi; r += RS) acc += Cvt<T>::ld(v + r * C + ch);
  }
  part[t] = acc;
  __syncthreads();
  if (t < C) {
    float tot = 0.f;
    for (int sl = 0; sl < RS; ++sl) tot += part[sl * C + t];
    Cvt<T>::st(out + g * C + t, tot * sc);
  }
}

template <typename T>
nt_status launch_segment_reduce(const T* v, T* out, const int64_t* splits, long long G, int C, int mean,
                                cudaStream_t st) {
  if (G <= 0) return NT_OK;
  if (G > 0x7FFFFFFFll) return NT_ERR_UNSUPPORTED;
  {
    LaunchScope ls("generic_segment_reduce", st);
    launch_kernel(segment_reduce_kernel<T>, (unsigned)G, 256, 0, st, v, out, splits, C, mean);
  }
  return cuda_ok();
}
template nt_status launch_segment_reduce<float>(const float*, float*, const int64_t*, long long, int, int,
                                                cudaStream_t);
template nt_status launch_segment_reduce<__nv_bfloat16>(const __nv_bfloat16*, __nv_bfloat16*, const int64_t*,
                                                        long long, int, int, cudaStream_t);

}  // namespace ntp
