// Rectangular pairs (N_s, M_s): the second pair layout of the method (Eq. 2: pairs (N_i, M_i, C) pack as
// (sum N_i M_i, C)).  Two entry points:
//   nt_rect_offsets_build     prefix sums of N_s, M_s and N_s M_s, the level-2 row splits (one group of M_s cells per
//                             row: the groups the column reduction of Eq. 4 consumes) and the cell decode
//   nt_rect_pair_broadcast    z[(s, a, b), :] = LN(W_a x_{s,a} + W_b y_{s,b}) gamma + beta from distinct row and
//                             column tokens (App. A.1: the rectangular variant has distinct row and column inputs)
// Everything downstream of the broadcast is position-wise or a segmented reduction over the row splits and is served
// by the existing calls (nt_pair_transition, nt_segment_reduce with these splits: its mean divides by M_s,
// nt_token_update).  Integer work is bit-exact; the broadcast is a pure streaming write of the packed state.
#include "fast.cuh"
#include "generic.cuh"

namespace ntp {

constexpr int RS_THREADS = 1024;

__global__ void __launch_bounds__(RS_THREADS)
rect_scan_kernel(const int64_t* ln, const int64_t* lm, int B, long long T1n, long long T1m,
                 long long T2, int64_t* tokn_off, int64_t* tokm_off,
                 int64_t* pair_off, int32_t* status) {
  pdl_begin();
  __shared__ long long s1[RS_THREADS], s2[RS_THREADS], s3[RS_THREADS];
  const int t = threadIdx.x;
  const int per = (B + RS_THREADS - 1) / RS_THREADS;
  const int lo = min(B, t * per), hi = min(B, lo + per);
  long long a = 0, b = 0, c = 0;
  bool neg = false;
  for (int s = lo; s < hi; ++s) {
    const long long n = ln[s], m = lm[s];
    neg |= n < 0 || m < 0;
    a += n;
    b += m;
    c += n * m;
  }
  s1[t] = a;
  s2[t] = b;
  s3[t] = c;
  __syncthreads();
  for (int off = 1; off < RS_THREADS; off <<= 1) {   // inclusive Hillis-Steele scan
    long long va = 0, vb = 0, vc = 0;
    if (t >= off) { va = s1[t - off]; vb = s2[t - off]; vc = s3[t - off]; }
    __syncthreads();
    s1[t] += va;
    s2[t] += vb;
    s3[t] += vc;
    __syncthreads();
  }
  long long ea = s1[t] - a, eb = s2[t] - b, ec = s3[t] - c;
  for (int s = lo; s < hi; ++s) {
    const long long n = ln[s], m = lm[s];
    tokn_off[s] = ea;
    tokm_off[s] = eb;
    pair_off[s] = ec;
    ea += n;
    eb += m;
    ec += n * m;
  }
  if (t == RS_THREADS - 1) {
    tokn_off[B] = s1[t];
    tokm_off[B] = s2[t];
    pair_off[B] = s3[t];
    if ((s1[t] != T1n || s2[t] != T1m || s3[t] != T2) && status) atomicCAS(status, 0, (int)NT_ERR_INCONSISTENT);
  }
  if (neg && status) atomicCAS(status, 0, (int)NT_ERR_INCONSISTENT);
}

__device__ inline int rect_search(const int64_t* off, int B, long long p) {   // largest s with off[s] <= p
  int lo = 0, hi = B;
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (off[mid] <= p) lo = mid; else hi = mid;
  }
  return lo;
}

__global__ void rect_row_splits_kernel(const int64_t* lm, const int64_t* tokn_off,
                                       const int64_t* pair_off, int B, long long T1n, long long T2,
                                       int64_t* row_splits) {
  pdl_begin();
  if (tokn_off[B] != T1n || pair_off[B] != T2) return;   // inconsistent totals: flagged by the scan
  const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t > T1n) return;
  if (t == T1n) { row_splits[t] = T2; return; }
  const int s = rect_search(tokn_off, B, t);
  row_splits[t] = pair_off[s] + (t - tokn_off[s]) * lm[s];
}

__global__ void __launch_bounds__(256)
rect_decode_kernel(const int64_t* lm, const int64_t* pair_off, int B, long long T2,
                   int32_t* ps, int32_t* pi, int32_t* pj) {
  pdl_begin();
  if (pair_off[B] != T2) return;
  const long long p = (long long)blockIdx.x * 256 + threadIdx.x;
  if (p >= T2) return;
  const int s = rect_search(pair_off, B, p);
  const unsigned long long r = (unsigned long long)(p - pair_off[s]), m = (unsigned long long)lm[s];
  const unsigned long long a = r / m;
  ps[p] = s;
  pi[p] = (int32_t)a;
  pj[p] = (int32_t)(r - a * m);
}

// ---- broadcast + LayerNorm
struct RectMeta {
  int B;
  int N[MAXB], M[MAXB];
  long long tokn_off[MAXB + 1], tokm_off[MAXB + 1], pair_off[MAXB + 1];
};

// Shape-generic form: one warp per packed cell (any c_z, float or bf16).
template <typename T>
__global__ void __launch_bounds__(256) rect_broadcast_ln_kernel(const float* u, const float* v,
                                                               const T* gamma, const T* beta,
                                                               float eps, int c_z, T* z, RectMeta m) {
  pdl_begin();
  const int lane = threadIdx.x & 31;
  const long long p = m.pair_off[0] + (long long)blockIdx.x * 8 + (threadIdx.x >> 5);
  if (p >= m.pair_off[m.B]) return;
  const int s = find_sample(m.pair_off, m.B, p);
  const int M = m.M[s];
  const long long r = p - m.pair_off[s];
  const long long a = r / M, b = r - a * M;
  const float* ur = u + (m.tokn_off[s] + a) * c_z;
  const float* vr = v + (m.tokm_off[s] + b) * c_z;
  float sum = 0.f;
  for (int c = lane; c < c_z; c += 32) sum += ur[c] + vr[c];
#pragma unroll
  for (int o = 16; o; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
  const float mean = sum / (float)c_z;
  float q = 0.f;
  for (int c = lane; c < c_z; c += 32) {
    const float dlt = ur[c] + vr[c] - mean;
    q += dlt * dlt;
  }
#pragma unroll
  for (int o = 16; o; o >>= 1) q += __shfl_xor_sync(0xffffffffu, q, o);
  const float rs = rsqrtf(q / (float)c_z + eps);
  T* zr = z + p * c_z;
  for (int c = lane; c < c_z; c += 32)
    Cvt<T>::st(zr + c, (ur[c] + vr[c] - mean) * rs * Cvt<T>::ld(gamma + c) + Cvt<T>::ld(beta + c));
}

// bf16 with c_z = 64, 128 or 256 goes through the band kernel of the square broadcast with rows x cols = N x M and
// distinct row / column token offsets.

static bool rect_totals(const int64_t* ln, const int64_t* lm, int B, long long& t1n, long long& t1m, long long& t2) {
  t1n = t1m = t2 = 0;
  for (int s = 0; s < B; ++s) {
    if (ln[s] < 0 || lm[s] < 0 || ln[s] > 0x7FFFFFFFll || lm[s] > 0x7FFFFFFFll) return false;
    t1n += ln[s];
    t1m += lm[s];
    t2 += ln[s] * lm[s];
  }
  return true;
}

template <typename T>
static nt_status rect_broadcast_impl(nt_dtype dt, int B, const int64_t* ln, const int64_t* lm, int c_s, int c_z, const void* x,
                                     const void* y, const void* W_a, const void* W_b, const void* g, const void* b, float eps,
                                     void* z, void* ws, long long t1n, long long t1m, cudaStream_t st) {
  const BcastPrepared bp = fast_broadcast_carve(ws, t1n, t1m, c_z);
  float* u = bp.u;
  float* v = bp.v;
  const bool fast = dt == NT_BF16 && !g_force_generic && fast_broadcast_supported(c_z);
  nt_status r;
  BatchMeta dummy;
  fill_meta(dummy, nullptr, 0, 0, 0, 0, 0);
  if (fast && fast_token_gemm_supported(c_s, c_z, 0)) {
    const TokSeg seg[2] = {{x, t1n, W_a, c_z, u}, {y, t1m, W_b, c_z, v}};      // rows and columns in one launch
    if ((r = fast_token_gemm(seg, 2, c_s, 1, 0, "rect_tok_proj", st)) != NT_OK) return r;
  } else {
    ProjArgs pa{};
    pa.a_mode = A_ROWMAJOR; pa.row0 = 0; pa.K = c_s;
    pa.A = x; pa.rows = t1n;
    pa.add(W_a, nullptr, c_z, ACT_NONE, u, O_STORE, 1);
    if (t1n > 0 && (r = launch_proj<T>(pa, dummy, st, "rect_tok_proj_u")) != NT_OK) return r;
    pa.A = y; pa.rows = t1m; pa.nseg = 0;
    pa.add(W_b, nullptr, c_z, ACT_NONE, v, O_STORE, 1);
    if (t1m > 0 && (r = launch_proj<T>(pa, dummy, st, "rect_tok_proj_v")) != NT_OK) return r;
  }
  if (fast && (r = fast_broadcast_prep(bp, t1n, t1m, g, c_z, st, "rect_broadcast_prep")) != NT_OK) return r;
  long long tn = 0, tm = 0, po = 0;
  for (int s0 = 0; s0 < B; s0 += MAXB) {
    RectMeta m;
    m.B = B - s0 < MAXB ? B - s0 : MAXB;
    for (int l = 0; l <= MAXB; ++l) {
      m.tokn_off[l] = tn; m.tokm_off[l] = tm; m.pair_off[l] = po;
      if (l < m.B) {
        m.N[l] = (int)ln[s0 + l];
        m.M[l] = (int)lm[s0 + l];
        tn += m.N[l]; tm += m.M[l]; po += (long long)m.N[l] * m.M[l];
      } else if (l < MAXB) {
        m.N[l] = m.M[l] = 0;
      }
    }
    const long long cells = m.pair_off[m.B] - m.pair_off[0];
    if (cells == 0) continue;
    if (fast) {
      BcastGeom geo;
      geo.B = m.B;
      for (int l = 0; l < MAXB; ++l) {
        geo.rows[l] = m.N[l]; geo.cols[l] = m.M[l];
        geo.u_off[l] = m.tokn_off[l]; geo.v_off[l] = m.tokm_off[l]; geo.z_off[l] = m.pair_off[l];
      }
      const nt_status r = fast_broadcast_ln_geom(bp, g, b, eps, c_z, z, geo, st, false, "rect_broadcast_ln");
      if (r != NT_OK) return r;
    } else {
      const long long blocks = (cells + 7) / 8;
      if (blocks > 0x7FFFFFFFll) return NT_ERR_UNSUPPORTED;
      LaunchScope ls("generic_rect_broadcast_ln", st);
      launch_kernel(rect_broadcast_ln_kernel<T>, (unsigned)blocks, 256, 0, st, u, v, (const T*)g, (const T*)b, eps, c_z, (T*)z, m);
    }
    if (cudaPeekAtLastError() != cudaSuccess) return cuda_fail("rectangular broadcast launch");
  }
  return NT_OK;
}

}  // namespace ntp

using namespace ntp;

extern "C" {

nt_status nt_rect_offsets_build(const int64_t* lengths_n_d, const int64_t* lengths_m_d, int32_t B, int64_t T1n, int64_t T1m,
                                int64_t T2, int64_t* tokn_off_d, int64_t* tokm_off_d, int64_t* pair_off_d,
                                int64_t* row_splits_d, int32_t* pos_sample_d, int32_t* pos_i_d, int32_t* pos_j_d,
                                int32_t* status_d, nt_stream stream_) {
  cudaStream_t stream = (cudaStream_t)stream_;
  if (B < 0 || T1n < 0 || T1m < 0 || T2 < 0) return NT_ERR_INVALID_ARG;
  if (!tokn_off_d || !tokm_off_d || !pair_off_d) return NT_ERR_INVALID_ARG;
  if (B > 0 && (!lengths_n_d || !lengths_m_d)) return NT_ERR_INVALID_ARG;
  const bool want_pos = pos_sample_d || pos_i_d || pos_j_d;
  if (want_pos && !(pos_sample_d && pos_i_d && pos_j_d)) return NT_ERR_INVALID_ARG;
  {
    LaunchScope ls("rect_offsets_scan", stream);
    launch_kernel(rect_scan_kernel, 1, RS_THREADS, 0, stream, lengths_n_d, lengths_m_d, B, T1n, T1m, T2, tokn_off_d, tokm_off_d, pair_off_d,
                                                   status_d);
  }
  if (row_splits_d) {
    const long long n = T1n + 1;
    LaunchScope ls("rect_offsets_row_splits", stream);
    launch_kernel(rect_row_splits_kernel, (unsigned)((n + 255) / 256), 256, 0, stream, lengths_m_d, tokn_off_d, pair_off_d, B, T1n, T2,
                                                                           row_splits_d);
  }
  if (want_pos && T2 > 0) {
    const long long blocks = (T2 + 255) / 256;
    if (blocks > 0x7FFFFFFFll) return NT_ERR_UNSUPPORTED;
    LaunchScope ls("rect_offsets_decode", stream);
    launch_kernel(rect_decode_kernel, (unsigned)blocks, 256, 0, stream, lengths_m_d, pair_off_d, B, T2, pos_sample_d, pos_i_d, pos_j_d);
  }
  return cuda_ok();
}

size_t nt_rect_broadcast_workspace_bytes(const int64_t* lengths_n_h, const int64_t* lengths_m_h, int32_t B, int32_t c_z) {
  long long t1n, t1m, t2;
  if (B <= 0 || c_z <= 0 || !lengths_n_h || !lengths_m_h || !rect_totals(lengths_n_h, lengths_m_h, B, t1n, t1m, t2)) return 0;
  return fast_broadcast_scratch_bytes(t1n, t1m, c_z);
}

nt_status nt_rect_pair_broadcast(nt_dtype dt, int32_t B, const int64_t* lengths_n_h, const int64_t* lengths_m_h, int32_t c_s,
                                 int32_t c_z, const void* x, const void* y, const void* W_a, const void* W_b,
                                 const void* ln_gamma, const void* ln_beta, float ln_eps, void* z, void* workspace,
                                 size_t workspace_bytes, nt_stream stream) {
  if (dt != NT_F32 && dt != NT_BF16) return NT_ERR_UNSUPPORTED;
  if (B < 0 || c_s <= 0 || c_z <= 0) return NT_ERR_INVALID_ARG;
  if (B == 0) return NT_OK;
  long long t1n, t1m, t2;
  if (!lengths_n_h || !lengths_m_h || !rect_totals(lengths_n_h, lengths_m_h, B, t1n, t1m, t2)) return NT_ERR_INVALID_ARG;
  if (t2 == 0) return NT_OK;
  if (!x || !y || !W_a || !W_b || !ln_gamma || !ln_beta || !z || !workspace) return NT_ERR_INVALID_ARG;
  if (((uintptr_t)x | (uintptr_t)y | (uintptr_t)z | (uintptr_t)workspace | (uintptr_t)W_a | (uintptr_t)W_b) & 15) return NT_ERR_INVALID_ARG;
  if (workspace_bytes < nt_rect_broadcast_workspace_bytes(lengths_n_h, lengths_m_h, B, c_z)) return NT_ERR_WORKSPACE;
  cudaStream_t st = (cudaStream_t)stream;
  if (dt == NT_F32)
    return rect_broadcast_impl<float>(dt, B, lengths_n_h, lengths_m_h, c_s, c_z, x, y, W_a, W_b, ln_gamma, ln_beta, ln_eps, z,
                                      workspace, t1n, t1m, st);
  return rect_broadcast_impl<__nv_bfloat16>(dt, B, lengths_n_h, lengths_m_h, c_s, c_z, x, y, W_a, W_b, ln_gamma, ln_beta, ln_eps,
                                            z, workspace, t1n, t1m, st);
}

}  // extern "C"
