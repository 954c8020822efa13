// Weight preparation for the tensor-core projections: LayerNorm folded into the weights.
//   out[n][:] = fp16(W[n][:] * gamma),  c01[n] = (sum_k W[n][k] beta[k],  sum_k out[n][k])
// so that (LN(z) W^T)[n] = rstd * (z . out[n] - mean * c01[n].y) + c01[n].x.
// One launch prepares up to two jobs (different K / gamma / beta); a job concatenates up to six
// source matrices; a NULL source stands for zero rows (padding).  gamma == NULL copies W.
// The folded weights are fp16: 11 significant bits instead of bf16's 8, at the same MMA rate.
#include "fast.cuh"

namespace ntp {

struct PrepJob {
  const __nv_bfloat16* src[6];
  int rows[6];
  float scale[6];   // extra factor on the rows of a source (and on its c0, c1)
  int bf16out[6];   // rows of this source are written as bf16 (for an MMA whose activation operand stays bf16)
  int nsrc, K, total;
  const __nv_bfloat16* gamma;
  const __nv_bfloat16* beta;
  __half* out;
  float2* c01;      // nullable
  __half* aug;      // nullable: [2][total][8] fp16 augmentation columns (see below)
};
struct PrepArgs { PrepJob job[2]; int njobs; };

__global__ void __launch_bounds__(256) ln_fold_prep_kernel(PrepArgs a) {
  pdl_begin();
  int n = blockIdx.x * 8 + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  int j = 0;
  while (j < a.njobs && n >= a.job[j].total) { n -= a.job[j].total; ++j; }
  if (j >= a.njobs) return;
  const PrepJob& J = a.job[j];
  int src = 0, r = n;
  while (r >= J.rows[src]) { r -= J.rows[src]; ++src; }
  const __nv_bfloat16* w = J.src[src] ? J.src[src] + (long long)r * J.K : nullptr;
  float c0 = 0.f, c1 = 0.f;
  // eight elements per lane with 16-byte accesses: the weight, gamma and beta loads of a row are all in flight at
  // once (the kernel is pure latency: a few hundred rows of K <= 1024 elements)
  const bool vec = J.K % 8 == 0 && (reinterpret_cast<size_t>(w) & 15) == 0 && (reinterpret_cast<size_t>(J.gamma) & 15) == 0 &&
                   (reinterpret_cast<size_t>(J.beta) & 15) == 0 && (reinterpret_cast<size_t>(J.out) & 15) == 0;
  for (int k8 = lane; vec && k8 < J.K / 8; k8 += 32) {
    const uint4 z4 = make_uint4(0, 0, 0, 0);
    const uint4 wv = w ? *reinterpret_cast<const uint4*>(w + k8 * 8) : z4;
    const uint4 gv = J.gamma ? *reinterpret_cast<const uint4*>(J.gamma + k8 * 8) : z4;
    const uint4 bv = J.gamma ? *reinterpret_cast<const uint4*>(J.beta + k8 * 8) : z4;
    const unsigned ww[4] = {wv.x, wv.y, wv.z, wv.w}, gw[4] = {gv.x, gv.y, gv.z, gv.w}, bw[4] = {bv.x, bv.y, bv.z, bv.w};
    unsigned ow[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      float f[2];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const float wvf = __uint_as_float(h ? ww[e] & 0xffff0000u : ww[e] << 16) * J.scale[src];
        const float gf = __uint_as_float(h ? gw[e] & 0xffff0000u : gw[e] << 16);
        const float bf = __uint_as_float(h ? bw[e] & 0xffff0000u : bw[e] << 16);
        f[h] = J.gamma ? wvf * gf : wvf;
        if (J.gamma) c0 = fmaf(wvf, bf, c0);
      }
      if (J.bf16out[src]) {
        const __nv_bfloat162 ob = __floats2bfloat162_rn(f[0], f[1]);
        if (J.gamma) c1 += __bfloat162float(ob.x) + __bfloat162float(ob.y);
        ow[e] = *reinterpret_cast<const unsigned*>(&ob);
      } else {
        const __half2 o = __floats2half2_rn(f[0], f[1]);
        if (J.gamma) c1 += __half2float(o.x) + __half2float(o.y);
        ow[e] = *reinterpret_cast<const unsigned*>(&o);
      }
    }
    *reinterpret_cast<uint4*>(J.out + (long long)n * J.K + k8 * 8) = make_uint4(ow[0], ow[1], ow[2], ow[3]);
  }
  for (int k = lane; !vec && k < J.K; k += 32) {
    const float wv = w ? __bfloat162float(w[k]) * J.scale[src] : 0.f;
    const float folded = J.gamma ? wv * __bfloat162float(J.gamma[k]) : wv;
    if (J.gamma) c0 = fmaf(wv, __bfloat162float(J.beta[k]), c0);
    if (J.bf16out[src]) {
      const __nv_bfloat16 ob = __float2bfloat16_rn(folded);
      if (J.gamma) c1 += __bfloat162float(ob);
      reinterpret_cast<__nv_bfloat16*>(J.out)[(long long)n * J.K + k] = ob;
    } else {
      const __half o = __float2half_rn(folded);
      if (J.gamma) c1 += __half2float(o);
      J.out[(long long)n * J.K + k] = o;
    }
  }
#pragma unroll
  for (int o = 16; o; o >>= 1) {
    c0 += __shfl_xor_sync(0xffffffffu, c0, o);
    c1 += __shfl_xor_sync(0xffffffffu, c1, o);
  }
  if (lane == 0) {
    if (J.c01) J.c01[n] = make_float2(c0, c1);
    if (J.aug) {
      // Extra K columns that make the MMA itself apply the LayerNorm correction: against activation columns
      // (m_hi, m_lo, m_hi, 1, 1) with m = -mean * rstd they contribute m * c1 + c0 (hi/lo split keeps ~22 bits).  The
      // columns 5 and 6 serve a reader that has c0 times a factor split into three fp16 parts instead of c0 times 1.
      const __half c1h = __float2half_rn(c1), c1l = __float2half_rn(c1 - __half2float(c1h));
      const __half c0h = __float2half_rn(c0), c0l = __float2half_rn(c0 - __half2float(c0h));
      const __half z = __float2half_rn(0.f);
      __half* r0 = J.aug + (long long)n * 8;
      __half* r1 = J.aug + ((long long)J.total + n) * 8;
      r0[0] = c1h; r0[1] = c1h; r0[2] = c1l; r0[3] = c0h; r0[4] = c0l; r0[5] = c0h; r0[6] = __float2half_rn(__half2float(c0h) * (1.f / 4096.f)); r0[7] = z;
      for (int e = 0; e < 8; ++e) r1[e] = z;
    }
  }
}

static void add_job(PrepArgs& a, const void* const* srcs, const int* rows, int nsrc, int K, const void* gamma,
                    const void* beta, void* out, void* c01, const float* scale = nullptr, void* aug = nullptr,
                    const int* bf16out = nullptr) {
  PrepJob& J = a.job[a.njobs++];
  J.total = 0;
  for (int i = 0; i < nsrc; ++i) {
    J.src[i] = (const __nv_bfloat16*)srcs[i];
    J.rows[i] = rows[i];
    J.scale[i] = scale ? scale[i] : 1.0f;
    J.bf16out[i] = bf16out ? bf16out[i] : 0;
    J.total += rows[i];
  }
  J.nsrc = nsrc;
  J.K = K;
  J.gamma = (const __nv_bfloat16*)gamma;
  J.beta = (const __nv_bfloat16*)beta;
  J.out = (__half*)out;
  J.c01 = (float2*)c01;
  J.aug = (__half*)aug;
}

static nt_status run_prep(const PrepArgs& a, cudaStream_t st) {
  int total = 0;
  for (int j = 0; j < a.njobs; ++j) total += a.job[j].total;
  {
    LaunchScope ls("weight_prep", st);
    launch_kernel(ln_fold_prep_kernel, (total + 7) / 8, 256, 0, st, a);
  }
  return cuda_ok("weight_prep launch");
}

// Triangle update: job 0 = [W_ag; W_ap; W_bg; W_bp; W_g] folded with LN_in (K = c_z),
//                  job 1 = W_o folded with LN_out (K = c_h).
nt_status fast_tri_prep(const nt_trimul_weights* W, int c_z, int c_h, void* prep, TriPrep& out, cudaStream_t st, bool launch) {
  char* p = (char*)prep;
  const int rows1 = 4 * c_h + c_z;
  out.w1 = p;
  out.wg = p + (size_t)4 * c_h * c_z * 2;
  p += align_up((size_t)rows1 * c_z * 2, 256);
  out.c01_1 = p;
  out.c01g = p + (size_t)4 * c_h * sizeof(float2);
  p += align_up((size_t)rows1 * sizeof(float2), 256);
  out.wo = p;
  p += align_up((size_t)c_z * c_h * 2, 256);
  out.c01o = p;
  p += align_up((size_t)c_z * sizeof(float2), 256);
  out.aug1 = p;                         // [2][rows1][8] fp16
  out.aug1_rows = rows1;
  PrepArgs a{};
  // The input projection computes D^T = W' z^T with 128 weight rows per MMA and pairs the gate rows of an
  // accumulator with the value rows of the next one: c_h = 128 -> [ag, ap, bg, bp]; c_h = 64 -> [ag, bg, ap, bp].
  const void* s128[5] = {W->W_ag, W->W_ap, W->W_bg, W->W_bp, W->W_g};
  const void* s64[5] = {W->W_ag, W->W_bg, W->W_ap, W->W_bp, W->W_g};
  const int r0[5] = {c_h, c_h, c_h, c_h, c_z};
  // gate and value rows are folded times 1/2 (exact): sigmoid(g) v = (tanh(g / 2) + 1) (v / 2) costs one MUFU and one FMA
  const float sc[5] = {0.5f, 0.5f, 0.5f, 0.5f, 1.0f};
  // W_g meets the bf16 state itself in the output stage (no conversion pass there): its folded rows are bf16
  const int asbf16[5] = {0, 0, 0, 0, 1};
  add_job(a, c_h == 64 ? s64 : s128, r0, 5, c_z, W->ln_in_gamma, W->ln_in_beta, out.w1, out.c01_1, sc, out.aug1, asbf16);
  const void* s1[1] = {W->W_o};
  const int r1[1] = {c_z};
  add_job(a, s1, r1, 1, c_h, W->ln_out_gamma, W->ln_out_beta, out.wo, out.c01o);
  return launch ? run_prep(a, st) : NT_OK;
}

// Attention: [W_q; W_k; W_v; W_b (H rows); zero rows up to 16; W_g] folded with LN (K = c).
nt_status fast_attn_prep(const nt_attn_weights* W, int c, int H, int d, void* prep, AttnPrep& out, cudaStream_t st, bool launch) {
  const int Hd = H * d;
  const int rows = 3 * Hd + 16 + Hd;
  char* p = (char*)prep;
  out.w = p;
  out.wg = p + (size_t)(3 * Hd + 16) * c * 2;
  p += align_up((size_t)rows * c * 2, 256);
  out.c01 = p;
  out.c01g = p + (size_t)(3 * Hd + 16) * sizeof(float2);
  p += align_up((size_t)rows * sizeof(float2), 256);
  out.aug = p;                          // [2][rows][8] fp16
  out.aug_rows = rows;
  PrepArgs a{};
  const void* s0[6] = {W->W_q, W->W_k, W->W_v, W->W_b, nullptr, W->W_g};
  if (H > 16) return NT_ERR_UNSUPPORTED;   // 16 bias rows are reserved between the projections and the gate
  const int r0[6] = {Hd, Hd, Hd, W->W_b ? H : 0, W->W_b ? 16 - H : 16, W->W_g ? Hd : 0};
  const float sc[6] = {1.f, 1.f, 1.f, sqrtf((float)d), 1.f, 1.f};   // bias rows times sqrt(d)
  // W_g meets the bf16 state itself in the output stage (no conversion pass there): its folded rows are bf16
  const int asbf16[6] = {0, 0, 0, 0, 0, 1};
  add_job(a, s0, r0, 6, c, W->ln_gamma, W->ln_beta, out.w, out.c01, sc, out.aug, asbf16);
  return launch ? run_prep(a, st) : NT_OK;
}

// Transition: [W_a (times 1/2: the gate goes through tanh); W_b] folded with LN (K = c).
nt_status fast_transition_prep(const nt_transition_weights* W, int c, int hidden, void* prep, TransPrep& out, cudaStream_t st) {
  const int rows = 2 * hidden;
  char* p = (char*)prep;
  out.w1 = p;
  p += align_up((size_t)rows * c * 2, 256);
  out.aug = p;                          // [2][rows][8] fp16; the kernel needs no (c0, c1) beside it
  out.rows = rows;
  PrepArgs a{};
  const void* s0[2] = {W->W_a, W->W_b};
  const int r0[2] = {hidden, hidden};
  const float sc[2] = {0.5f, 1.0f};
  add_job(a, s0, r0, 2, c, W->ln_gamma, W->ln_beta, out.w1, nullptr, sc, out.aug);
  return run_prep(a, st);
}

}  // namespace ntp
