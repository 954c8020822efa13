// bf16 kernels tuned for sm_100a.  Memory-bound steps stay on CUDA cores with 16-byte vector
// access; dense contractions use tcgen05 tensor-core tiles with TMEM accumulators.
#pragma once
#include "common.cuh"

namespace ntp {

// Geometry of a broadcast z[s][i][j] = LN(u[s][i] + v[s][j]): rows x cols cells per sample, token-row offsets of
// the two operands and cell offset of the result.  Square pairs use the same tokens for both operands.
struct BcastGeom {
  int B;
  int rows[MAXB], cols[MAXB];
  long long u_off[MAXB], v_off[MAXB], z_off[MAXB];
};
// Prepared token rows of the pair broadcast: u centred, v centred and times gamma (float, in place of the token
// projections), the centred rows as high and low bf16 parts, squared norms of the centred rows.
struct BcastPrepared {
  float* u;
  float* v;
  __nv_bfloat16* ub;
  __nv_bfloat16* vb;
  __nv_bfloat16* ubl;
  __nv_bfloat16* vbl;
  float* nu;
  float* nv;
};
size_t fast_broadcast_scratch_bytes(long long rows_u, long long rows_v, int c_z);
BcastPrepared fast_broadcast_carve(void* ws, long long rows_u, long long rows_v, int c_z);
// p.u / p.v hold the token projections on entry; afterwards every field is as described above.
nt_status fast_broadcast_prep(const BcastPrepared& p, long long rows_u, long long rows_v, const void* gamma, int c_z,
                              cudaStream_t st, const char* scope);
nt_status fast_broadcast_ln_geom(const BcastPrepared& p, const void* gamma, const void* beta, float eps, int c_z,
                                 void* z, const BcastGeom& m, cudaStream_t st, bool accumulate, const char* scope);
bool fast_broadcast_supported(int c_z);
nt_status fast_broadcast_ln(const BcastPrepared& p, const void* gamma, const void* beta, float eps, int c_z, void* z,
                            const BatchMeta& m, cudaStream_t st, bool accumulate = false);

bool fast_segment_reduce_supported(int C);
nt_status fast_segment_reduce(const void* v, void* out, const int64_t* splits, long long G, int C, int mean,
                              cudaStream_t st);

// token-side projections: out[r][n] (+)= sum_k A[r][k] W[n][k] for up to four segments in one launch
constexpr int TOK_SEGS = 4;
struct TokSeg { const void* A; long long rows; const void* W; int N; void* out; };
bool fast_token_gemm_supported(int K, int N0, int N1);
nt_status fast_token_gemm(const TokSeg* seg, int n, int K, int out_f32, int accumulate, const char* name, cudaStream_t st);

// the same on tcgen05 (persistent 128 x 256 tiles), for token axes long enough to fill the GPU with tiles; the segments
// share A
bool fast_token_gemm_tc_supported(const TokSeg* seg, int n, int K);
nt_status fast_token_gemm_tc(const TokSeg* seg, int n, int K, int out_f32, int accumulate, int* status, const char* name, cudaStream_t st);

// pair-biased single attention: LayerNorm of the token rows (bf16 out), o <- sigmoid(g) * o, and the bias planes
// bias[s][h][i][j] = scale * (LN(z_ij) W_b^T)[h] in the head-major padded layout of the attention core
bool fast_single_attn_supported(int c_s, int c_z, int H, int d);
nt_status fast_ln_rows(const void* x, const void* g, const void* b, float eps, int C, long long rows, void* out, cudaStream_t st,
                       const char* name = "single_attn_ln");
nt_status fast_gate_mul(const void* g, void* o, long long n, cudaStream_t st, const char* name = "single_attn_gate");
nt_status fast_single_bias(const void* z, const void* g, const void* b, const void* Wb, float eps, int C, int H, float scale,
                           const BatchMeta& m, void* bias, cudaStream_t st);

// whole-row attention core on tcgen05 for the samples with 1 <= N <= n_max (pair order, d in {16, 32}, bias stored times sqrt(d));
// fast_attn_tc_max_n gives the largest N whose score row and bias tiles fit (0: not supported)
int fast_attn_tc_max_n(int d, bool has_bias);
nt_status fast_attn_core_tc(const void* q, const void* k, const void* v, const void* bias, void* o, int H, int d,
                            const BatchMeta& m, int n_max, int* status, cudaStream_t st, bool col = false);

// attention core with the softmax weights in register fragments (fast_attn_frag.cu): any sample length, d in {16, 32, 64},
// pair order (rows or columns; one bias plane per (sample, head), stored times sqrt(d), for columns stored transposed)
// or token order (rows = samples; the bias planes, if any, belong to the sample's own queries).  Samples with N <= n_min
// are left out (they belong to another kernel).
extern int g_fr_drop;
enum { FR_MODE_PAIR_ROW = 0, FR_MODE_TOKEN = 1, FR_MODE_PAIR_COL = 2 };
bool fast_attn_fr_supported(int H, int d);
nt_status fast_attn_core_fr(const void* q, const void* k, const void* v, const void* bias, void* o, int H, int d,
                            int mode, const BatchMeta& m, int* status, cudaStream_t st, int n_min = 0);

// triangle contraction on tcgen05: a, b, t are three equally spaced channel-major buffers
// (b = a + stride, t = a + 2 * stride); incoming = contraction over the first index (sum_k a[k][i] b[k][j])
nt_status fast_contract(const void* a, size_t buf_stride_bytes, int C, const BatchMeta& m, int* status,
                        cudaStream_t st, bool incoming = false);

// ---- tensor-core projections (tcgen05, LayerNorm folded into fp16 weights prepared once per call)
struct TriPrep { void *w1, *c01_1, *wg, *c01g, *wo, *c01o, *aug1; int aug1_rows; };
struct AttnPrep { void *w, *c01, *wg, *c01g, *aug; int aug_rows; };
// launch = false only lays the pointers of `out` over an already prepared buffer
nt_status fast_tri_prep(const nt_trimul_weights* W, int c_z, int c_h, void* prep, TriPrep& out, cudaStream_t st, bool launch = true);
// the bias rows are folded times sqrt(d): the attention cores keep scores in units of q.k
nt_status fast_attn_prep(const nt_attn_weights* W, int c, int H, int d, void* prep, AttnPrep& out, cudaStream_t st, bool launch = true);

// a = sig(LN(z) W_ag^T) * (LN(z) W_ap^T), b likewise: fp16, channel-major
bool fast_tri_in_supported(int c_z, int c_h);
nt_status fast_tri_in(const void* z, const TriPrep& tp, float eps, int c_z, int c_h, void* a, void* b,
                      const BatchMeta& m, int* status, cudaStream_t st, float2* zstats = nullptr);

// in place on z: z += sigmoid(LN_in(z) W_g^T) * (LN_out(t) W_o^T); t fp16 channel-major scaled by 1 / N
bool fast_tri_out_supported(int c_z, int c_h);
nt_status fast_tri_out(void* z, const void* t, const TriPrep& tp, float eps, int c_z, int c_h, const BatchMeta& m,
                       int* status, cudaStream_t st, const float2* zstats = nullptr);

// q, k, v row-major bf16, bias head-major bf16 (nullable)
bool fast_attn_in_supported(int c, int H, int d);
nt_status fast_attn_in(const void* z, const AttnPrep& ap, float eps, int c, int H, int d, void* q, void* k, void* v,
                       void* bias, const BatchMeta& m, int* status, cudaStream_t st, float2* zstats = nullptr,
                       int bias_tr_above = 0x7fffffff);   // samples longer than this: bias planes stored transposed

// in place on z: z += (sigmoid(LN(z) W_g^T) * o) W_o^T
bool fast_attn_out_supported(int c, int H, int d);
// Fused mean over j behind the attention output stage: column sums of 32-position groups land in `partial`
// (fast_attn_out_partial_bytes), fast_segment_partials adds them per pair row into out [T1, C] (bf16).
bool fast_attn_out_reduce_supported(const BatchMeta& m);
size_t fast_attn_out_partial_bytes(long long rows, int c);
nt_status fast_segment_partials(const float* partial, const BatchMeta& m, int C, int mean, void* out, cudaStream_t st);
nt_status fast_attn_out(void* z, const void* o, const void* W_o, const AttnPrep& ap, float eps, int c, int H, int d,
                        const BatchMeta& m, int* status, cudaStream_t st, float* partial = nullptr, const float2* zstats = nullptr);

// SwiGLU transition, fused on tcgen05: z += (silu(LN(z) W_a^T) * (LN(z) W_b^T)) W_2^T with the hidden activation
// kept on chip.  prep: at least 1 MiB of device scratch for the folded weights.
struct TransPrep { void *w1, *aug; int rows; };   // folded [W_a / 2; W_b] (2 hidden rows) and their augmentation columns
nt_status fast_transition_prep(const nt_transition_weights* W, int c, int hidden, void* prep, TransPrep& out, cudaStream_t st);
bool fast_transition_supported(int c, int hidden);
nt_status fast_transition(void* z, const nt_transition_weights* W, float eps, int c, int hidden, long long rows,
                          void* prep, int* status, cudaStream_t st);

}  // namespace ntp
