// C-ABI entry points of libnested_pair: argument validation, workspace carving and the launch
// sequence of every call.  Nothing here allocates or synchronises.
#include <cstdlib>
#include <cstring>
#include <mutex>
#include <string>
#include <vector>

#include "common.cuh"
#include "fast.cuh"
#include "generic.cuh"

namespace ntp {

#ifdef NT_DEBUG_BOUNDS
__device__ int g_nt_bounds[4] = {0, 0, 0, 0};
#endif

std::atomic<long long> g_launches{0};
int g_force_generic = 0;
int g_fr_drop = -1; // testing aid (nt_debug_attn_drop): key blocks a CTA of that core requests before it stops
int g_fr_all = 0;   // testing aid (nt_attn_core_mode): the register-fragment attention core for every sample length

// ---- per-kernel event timing (off unless nt_profile_begin was called) ----------------------
struct ProfRecord { const char* name; cudaEvent_t e0, e1; };
static std::mutex g_prof_mu;
static bool g_prof_on = false;
static std::vector<ProfRecord> g_prof;

LaunchScope::LaunchScope(const char* name, cudaStream_t s) : st(s), slot(-1) {
  g_launches.fetch_add(1, std::memory_order_relaxed);
  if (!g_prof_on) return;
  std::lock_guard<std::mutex> lk(g_prof_mu);
  ProfRecord r{name, nullptr, nullptr};
  if (cudaEventCreate(&r.e0) != cudaSuccess || cudaEventCreate(&r.e1) != cudaSuccess) return;
  cudaEventRecord(r.e0, st);
  slot = (int)g_prof.size();
  g_prof.push_back(r);
}

LaunchScope::~LaunchScope() {
  if (slot < 0) return;
  std::lock_guard<std::mutex> lk(g_prof_mu);
  cudaEventRecord(g_prof[slot].e1, st);
}

int sm_count() {
  static int cached[64] = {};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 148;
  if (cached[dev] == 0) {
    int n = 0;
    if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n <= 0) n = 148;
    cached[dev] = n;
  }
  return cached[dev];
}

nt_status cuda_fail(const char* where) {
  const cudaError_t e = cudaGetLastError();   // also clears a non-sticky error
  fprintf(stderr, "libnested_pair: CUDA failure at %s: %s\n", where, cudaGetErrorString(e));
  return NT_ERR_CUDA;
}

void fill_meta(BatchMeta& m, const int64_t* len, int s0, int s1, long long tok0, long long pair0, long long cm0) {
  m.B = s1 - s0;
  m.tok_off[0] = tok0;
  m.pair_off[0] = pair0;
  m.cm_off[0] = cm0;
  for (int s = s0; s < s1; ++s) {
    const int l = s - s0;
    const long long n = len[s];
    m.N[l] = (int)n;
    m.tok_off[l + 1] = m.tok_off[l] + n;
    m.pair_off[l + 1] = m.pair_off[l] + n * n;
    m.cm_off[l + 1] = m.cm_off[l] + n * round_up8((int)n);
  }
  for (int l = m.B; l < MAXB; ++l) {
    m.N[l] = 0;
    m.tok_off[l + 1] = m.tok_off[m.B];
    m.pair_off[l + 1] = m.pair_off[m.B];
    m.cm_off[l + 1] = m.cm_off[m.B];
  }
}

bool GroupIter::next(BatchMeta& m) {
  if (s0 >= B) return false;
  const int s1 = s0 + MAXB < B ? s0 + MAXB : B;
  fill_meta(m, len, s0, s1, tok, pair, cm);
  tok = m.tok_off[m.B];
  pair = m.pair_off[m.B];
  cm = m.cm_off[m.B];
  s0 = s1;
  return true;
}

static bool aligned16(const void* p) { return ((uintptr_t)p & 15) == 0; }
// every pointer of a weights structure, seen as an array of pointers (NULL entries are allowed where the call allows them)
template <typename W>
static bool weights_aligned16(const W* w) {
  const void* const* ptr = reinterpret_cast<const void* const*>(w);
  for (size_t i = 0; i < sizeof(W) / sizeof(void*); ++i)
    if (!aligned16(ptr[i])) return false;
  return true;
}

struct Totals { long long T1 = 0, T2 = 0, cm = 0; int nmax = 0; };

static nt_status totals_of(const int64_t* len, int B, Totals& t) {
  for (int s = 0; s < B; ++s) {
    const long long n = len[s];
    if (n < 0) return NT_ERR_INVALID_ARG;
    if (n > 0x3FFFFFFF) return NT_ERR_UNSUPPORTED;
    t.T1 += n;
    t.T2 += n * n;
    t.cm += n * round_up8((int)n);
    if (n > t.nmax) t.nmax = (int)n;
  }
  return NT_OK;
}

static nt_status check_layout(const nt_layout* L, Totals& t) {
  if (!L || L->B < 0) return NT_ERR_INVALID_ARG;
  if (L->B > 0 && !L->lengths_h) return NT_ERR_INVALID_ARG;
  nt_status st = totals_of(L->lengths_h, L->B, t);
  if (st != NT_OK) return st;
  if (t.T1 != L->T1 || t.T2 != L->T2) return NT_ERR_INCONSISTENT;
  return NT_OK;
}

static size_t esize(nt_dtype dt) { return dt == NT_F32 ? 4 : 2; }

struct Carver {   // hands out 256-byte aligned slices of the caller's workspace
  char* base;
  size_t off = 0;
  explicit Carver(void* p) : base((char*)p) {}
  void* take(size_t bytes) {
    void* r = base ? base + off : nullptr;
    off += align_up(bytes, 256);
    return r;
  }
};

struct TriWs { void *a, *b, *t, *g, *prep; size_t bytes; };
static TriWs carve_trimul(void* ws, nt_dtype dt, const Totals& t, int c_z, int c_h) {
  Carver c(ws);
  TriWs w;
  const size_t e = esize(dt);
  w.a = c.take((size_t)c_h * t.cm * e);
  w.b = c.take((size_t)c_h * t.cm * e);
  w.t = c.take((size_t)c_h * t.cm * e);
  w.g = c.take((size_t)t.T2 * c_z * e);
  w.prep = c.take(1 << 20);   // folded weights of the tensor-core projections
  w.bytes = c.off;
  return w;
}

struct AttnWs { void *q, *k, *v, *o, *g, *bias, *prep; size_t bytes; };
static AttnWs carve_attn(void* ws, nt_dtype dt, const Totals& t, nt_order order, int H, int d) {
  Carver c(ws);
  AttnWs w;
  const size_t e = esize(dt);
  const size_t rows = order == NT_ORDER_PAIR_IJC ? t.T2 : t.T1;
  const size_t Hd = (size_t)H * d;
  w.q = c.take(rows * Hd * e);
  w.k = c.take(rows * Hd * e);
  w.v = c.take(rows * Hd * e);
  w.o = c.take(rows * Hd * e);
  w.g = c.take(rows * Hd * e);
  w.bias = c.take(order == NT_ORDER_PAIR_IJC ? (size_t)H * t.cm * e : 0);
  w.prep = c.take(1 << 20);   // folded weights of the tensor-core projections
  w.bytes = c.off;
  return w;
}

struct SingleWs { void *q, *k, *v, *o, *g, *xh, *bias; size_t bytes; };
static SingleWs carve_single(void* ws, nt_dtype dt, const Totals& t, int c_s, int H, int d) {
  Carver c(ws);
  SingleWs w;
  const size_t e = esize(dt), Hd = (size_t)H * d;
  w.q = c.take(t.T1 * Hd * e);
  w.k = c.take(t.T1 * Hd * e);
  w.v = c.take(t.T1 * Hd * e);
  w.o = c.take(t.T1 * Hd * e);
  w.g = c.take(t.T1 * Hd * e);
  w.xh = c.take(t.T1 * (size_t)c_s * e);
  w.bias = c.take((size_t)H * t.cm * e);
  w.bytes = c.off;
  return w;
}

static size_t broadcast_ws_bytes(const Totals& t, int c_z) {
  // token projections u, v (float) + what the streaming kernel's preparation adds (bf16 copies, squared norms)
  return fast_broadcast_scratch_bytes(t.T1, t.T1, c_z);
}

// ------------------------------------------------------------------------------------------
template <typename T>
static nt_status pair_broadcast_impl(const nt_layout* L, const Totals& tot, int c_s, int c_z, const void* x,
                                     const void* W_a, const void* W_b, const void* g, const void* b, float eps,
                                     void* z, void* ws, cudaStream_t st, bool fast, bool accumulate = false) {
  const BcastPrepared bp = fast_broadcast_carve(ws, tot.T1, tot.T1, c_z);
  float* u = bp.u;
  float* v = bp.v;
  BatchMeta dummy;
  fill_meta(dummy, nullptr, 0, 0, 0, 0, 0);
  ProjArgs pa{};
  pa.A = x; pa.a_mode = A_ROWMAJOR; pa.row0 = 0; pa.rows = tot.T1; pa.K = c_s;
  pa.add(W_a, nullptr, c_z, ACT_NONE, u, O_STORE, 1);
  pa.add(W_b, nullptr, c_z, ACT_NONE, v, O_STORE, 1);
  nt_status r;
  if (fast && fast_token_gemm_supported(c_s, c_z, c_z)) {
    const TokSeg seg[2] = {{x, tot.T1, W_a, c_z, u}, {x, tot.T1, W_b, c_z, v}};
    r = fast_token_gemm(seg, 2, c_s, 1, 0, "tok_proj", st);
    if (r != NT_OK) return r;
  } else {
    r = launch_proj<T>(pa, dummy, st, "generic_tok_proj");
    if (r != NT_OK) return r;
  }
  if (fast && (r = fast_broadcast_prep(bp, tot.T1, tot.T1, g, c_z, st, "broadcast_prep")) != NT_OK) return r;
  GroupIter it(L->lengths_h, L->B);
  BatchMeta m;
  while (it.next(m)) {
    if (fast) r = fast_broadcast_ln(bp, g, b, eps, c_z, z, m, st, accumulate);
    else r = launch_broadcast_ln<T>(u, v, (const T*)g, (const T*)b, eps, c_z, (T*)z, m, st, accumulate);
    if (r != NT_OK) return r;
  }
  return NT_OK;
}

template <typename T>
static nt_status tri_mul_generic(const nt_layout* L, const Totals& tot, int c_z, int c_h, const nt_trimul_weights* W,
                                 float eps, void* z, void* ws, nt_dtype dt, cudaStream_t st, bool incoming) {
  TriWs w = carve_trimul(ws, dt, tot, c_z, c_h);
  // The tensor-core stages exchange a, b (fp16) and t (fp16, scaled by 1 / N): all three or none.
  // (the tensor-core kernels index positions inside a sample with 32 bits: N below 2^16)
  const bool tc = dt == NT_BF16 && !g_force_generic && tot.nmax < 60000 && fast_tri_in_supported(c_z, c_h) &&
                  fast_tri_out_supported(c_z, c_h);
  TriPrep tprep{};
  if (tc) {
    // folded weights: the caller's, prepared ahead of time, or built now into the workspace
    nt_status r0 = W->prepared ? fast_tri_prep(W, c_z, c_h, const_cast<void*>(W->prepared), tprep, st, false)
                               : fast_tri_prep(W, c_z, c_h, w.prep, tprep, st);
    if (r0 != NT_OK) return r0;
  }
  GroupIter it(L->lengths_h, L->B);
  BatchMeta m;
  while (it.next(m)) {
    const long long row0 = m.pair_off[0], rows = m.pair_off[m.B] - row0;
    if (rows == 0) continue;
    ProjArgs pa{};
    pa.A = z; pa.a_mode = A_ROWMAJOR; pa.row0 = row0; pa.rows = rows; pa.K = c_z;
    pa.ln_g = W->ln_in_gamma; pa.ln_b = W->ln_in_beta; pa.eps = eps;
    nt_status r;
    if (tc) {
      // the gate buffer is free on this path (the output stage recomputes the gate): it carries the z row statistics
      r = fast_tri_in(z, tprep, eps, c_z, c_h, w.a, w.b, m, L->status_d, st, (float2*)w.g);
      if (r != NT_OK) return r;
    } else {
      // a, b and the gate from the same normalised rows: one launch
      pa.add(W->W_ag, W->W_ap, c_h, ACT_SIGMOID, w.a, O_CHANNEL_MAJOR);
      pa.add(W->W_bg, W->W_bp, c_h, ACT_SIGMOID, w.b, O_CHANNEL_MAJOR);
      pa.add(W->W_g, nullptr, c_z, ACT_SIGMOID, w.g, O_STORE);
      r = launch_proj<T>(pa, m, st, "generic_tri_in");
      if (r != NT_OK) return r;
    }
    if (tc)
      r = fast_contract(w.a, (size_t)((char*)w.b - (char*)w.a), c_h, m, L->status_d, st, incoming);
    else
      r = launch_contract<T>((const T*)w.a, (const T*)w.b, (T*)w.t, c_h, m, st, incoming);
    if (r != NT_OK) return r;
    if (tc) {   // (recomputes the output gate from z)
      r = fast_tri_out(z, w.t, tprep, eps, c_z, c_h, m, L->status_d, st, (const float2*)w.g);
      if (r != NT_OK) return r;
      continue;
    }
    ProjArgs po{};
    po.A = w.t; po.a_mode = A_CHANNEL_MAJOR; po.row0 = row0; po.rows = rows; po.K = c_h;
    po.ln_g = W->ln_out_gamma; po.ln_b = W->ln_out_beta; po.eps = eps;
    po.gateO = w.g;
    po.add(W->W_o, nullptr, c_z, ACT_NONE, z, O_ACCUM);
    r = launch_proj<T>(po, m, st, "generic_tri_out");
    if (r != NT_OK) return r;
  }
  return NT_OK;
}

template <typename T>
static nt_status attn_generic(const nt_layout* L, const Totals& tot, nt_order order, int c, int H, int d,
                              const nt_attn_weights* W, float eps, void* zx, void* ws, nt_dtype dt,
                              cudaStream_t st, bool col, void* mean_out = nullptr, bool* mean_done = nullptr) {
  AttnWs w = carve_attn(ws, dt, tot, order, H, d);
  if (mean_done) *mean_done = mean_out != nullptr;
  const int Hd = H * d;
  const bool pair = order == NT_ORDER_PAIR_IJC;
  const bool tc = dt == NT_BF16 && !g_force_generic && pair && W->ln_gamma && tot.nmax < 60000;
  const bool tc_in = tc && fast_attn_in_supported(c, H, d) && fast_attn_fr_supported(H, d);   // bias goes out times sqrt(d)
  const bool tc_out = tc && W->W_g && fast_attn_out_supported(c, H, d);   // recomputes the gate from z
  const bool tok_fast = dt == NT_BF16 && !g_force_generic && !pair && !W->W_b && c % 8 == 0 && c <= Hd && c <= 2048 &&
                        fast_attn_fr_supported(H, d) && fast_token_gemm_supported(c, Hd, Hd) &&
                        fast_token_gemm_supported(Hd, c, 0);
  // the register-fragment core takes every sample length (pair order: the samples beyond the whole-row core's reach)
  // (a bias must come from the tensor-core projection, which writes it in the units the cores expect)
  const bool fr_pair = dt == NT_BF16 && !g_force_generic && pair && !col && tot.nmax < 60000 && (tc_in || !W->W_b) &&
                       fast_attn_fr_supported(H, d);
  AttnPrep aprep{};
  if (tc_in || tc_out) {
    nt_status r0 = W->prepared ? fast_attn_prep(W, c, H, d, const_cast<void*>(W->prepared), aprep, st, false)
                               : fast_attn_prep(W, c, H, d, w.prep, aprep, st);
    if (r0 != NT_OK) return r0;
  }
  GroupIter it(L->lengths_h, L->B);
  BatchMeta m;
  while (it.next(m)) {
    const long long row0 = pair ? m.pair_off[0] : m.tok_off[0];
    const long long rows = (pair ? m.pair_off[m.B] : m.tok_off[m.B]) - row0;
    if (rows == 0) continue;
    nt_status r;
    if (tok_fast) {
      // token order: the rows are T1 tokens, so the projections are small GEMMs on mma.sync tiles around the
      // segmented core: LayerNorm once into the (not yet written) o buffer, q | k | v | g in one launch that shares
      // the normalised rows, the core, the gate, the output GEMM accumulated into x
      const size_t e = 2, to = (size_t)row0 * Hd * e;
      char* xr = (char*)zx + (size_t)row0 * c * e;
      char* xh = xr;
      if (W->ln_gamma) {
        xh = (char*)w.o + to;
        if ((r = fast_ln_rows(xr, W->ln_gamma, W->ln_beta, eps, c, rows, xh, st, "tok_attn_ln")) != NT_OK) return r;
      }
      const TokSeg seg[4] = {{xh, rows, W->W_q, Hd, (char*)w.q + to}, {xh, rows, W->W_k, Hd, (char*)w.k + to}, {xh, rows, W->W_v, Hd, (char*)w.v + to},
                             {xh, rows, W->W_g, Hd, W->W_g ? (char*)w.g + to : nullptr}};
      if ((r = fast_token_gemm(seg, 4, c, 0, 0, "tok_attn_in", st)) != NT_OK) return r;
      if ((r = fast_attn_core_fr(w.q, w.k, w.v, nullptr, w.o, H, d, FR_MODE_TOKEN, m, L->status_d, st)) != NT_OK) return r;
      if (W->W_g && (r = fast_gate_mul((char*)w.g + to, (char*)w.o + to, rows * Hd, st, "tok_attn_gate")) != NT_OK) return r;
      const TokSeg so = {(char*)w.o + to, rows, W->W_o, c, xr};
      if ((r = fast_token_gemm(&so, 1, Hd, 0, 1, "tok_attn_out", st)) != NT_OK) return r;
      continue;
    }
    ProjArgs pa{};
    pa.A = zx; pa.a_mode = A_ROWMAJOR; pa.row0 = row0; pa.rows = rows; pa.K = c;
    pa.ln_g = W->ln_gamma; pa.ln_b = W->ln_beta; pa.eps = eps;
    // column-wise attention: the whole-row core gathers its (short) samples' bias tiles transposed itself; the
    // register-fragment core wants the planes of the longer samples stored transposed
    const bool fr_col = tc_in && col && fast_attn_fr_supported(H, d);
    const int n_tc_col = (fr_col && !g_fr_all) ? fast_attn_tc_max_n(d, W->W_b != nullptr) : 0;
    if (tc_in) {
      // the gate buffer is free when the output stage recomputes the gate: it carries the z row statistics to it
      r = fast_attn_in(zx, aprep, eps, c, H, d, w.q, w.k, w.v, W->W_b ? w.bias : nullptr, m, L->status_d, st,
                       tc_out ? (float2*)w.g : nullptr, fr_col ? n_tc_col : 0x7fffffff);
      if (r != NT_OK) return r;
    } else {
      pa.add(W->W_q, nullptr, Hd, ACT_NONE, w.q, O_STORE);
      pa.add(W->W_k, nullptr, Hd, ACT_NONE, w.k, O_STORE);
      pa.add(W->W_v, nullptr, Hd, ACT_NONE, w.v, O_STORE);
    }
    if (W->W_g && !tc_out) pa.add(W->W_g, nullptr, Hd, ACT_SIGMOID, w.g, O_STORE);
    if (W->W_b && !tc_in) pa.add(W->W_b, nullptr, H, ACT_NONE, w.bias, O_CHANNEL_MAJOR);
    if (pa.nseg && (r = launch_proj<T>(pa, m, st, "generic_attn_in")) != NT_OK) return r;
    if (col && fr_col) {
      bool any_short = false, any_long = false;
      for (int s = 0; s < m.B; ++s) {
        if (m.N[s] >= 1 && m.N[s] <= n_tc_col) any_short = true;
        else if (m.N[s] > n_tc_col) any_long = true;
      }
      r = NT_OK;
      if (any_short) r = fast_attn_core_tc(w.q, w.k, w.v, W->W_b ? w.bias : nullptr, w.o, H, d, m, n_tc_col, L->status_d, st, true);
      if (r == NT_OK && any_long)
        r = fast_attn_core_fr(w.q, w.k, w.v, W->W_b ? w.bias : nullptr, w.o, H, d, FR_MODE_PAIR_COL, m, L->status_d, st, n_tc_col);
    } else if (col) {
      // the shape-generic core (the bias is stored times sqrt(d) when the tensor-core projections wrote it)
      r = launch_attn_core<T>((const T*)w.q, (const T*)w.k, (const T*)w.v, W->W_b ? (const T*)w.bias : nullptr,
                              (T*)w.o, H, d, 2, m, st, tc_in ? rsqrtf((float)d) : 1.0f);
    } else if (fr_pair) {
      // a score row of up to n_tc keys fits the whole-row core's accumulator; longer samples take the register-fragment core
      int n_tc = g_fr_all ? 0 : fast_attn_tc_max_n(d, W->W_b != nullptr);
      bool any_short = false, any_long = false;
      for (int s = 0; s < m.B; ++s) {
        if (m.N[s] >= 1 && m.N[s] <= n_tc) any_short = true;
        else if (m.N[s] > n_tc) any_long = true;
      }
      r = NT_OK;
      if (any_short) r = fast_attn_core_tc(w.q, w.k, w.v, W->W_b ? w.bias : nullptr, w.o, H, d, m, n_tc, L->status_d, st);
      if (r == NT_OK && any_long)
        r = fast_attn_core_fr(w.q, w.k, w.v, W->W_b ? w.bias : nullptr, w.o, H, d, FR_MODE_PAIR_ROW, m, L->status_d, st, n_tc);
    }
    else
      r = launch_attn_core<T>((const T*)w.q, (const T*)w.k, (const T*)w.v, W->W_b ? (const T*)w.bias : nullptr,
                              (T*)w.o, H, d, pair ? 1 : 0, m, st);
    if (r != NT_OK) return r;
    if (tc_out) {
      // the mean over j of the updated state, taken while its tiles are still on chip; q is dead by now and lends
      // its memory to the partial sums
      float* partial = nullptr;
      if (mean_out && fast_attn_out_reduce_supported(m) &&
          fast_attn_out_partial_bytes(rows, c) <= (size_t)tot.T2 * Hd * sizeof(T))
        partial = (float*)w.q;
      r = fast_attn_out(zx, w.o, W->W_o, aprep, eps, c, H, d, m, L->status_d, st, partial,
                        tc_in ? (const float2*)w.g : nullptr);
      if (r != NT_OK) return r;
      if (partial) {
        if ((r = fast_segment_partials(partial, m, c, 1, mean_out, st)) != NT_OK) return r;
      } else if (mean_done) {
        *mean_done = false;
      }
      continue;
    }
    if (mean_done) *mean_done = false;
    ProjArgs po{};
    po.A = w.o; po.a_mode = A_ROWMAJOR; po.row0 = row0; po.rows = rows; po.K = Hd;
    po.gateA = W->W_g ? w.g : nullptr;
    po.add(W->W_o, nullptr, c, ACT_NONE, zx, O_ACCUM);
    if ((r = launch_proj<T>(po, m, st, "generic_attn_out")) != NT_OK) return r;
  }
  return NT_OK;
}

// Pair-biased single attention: token projections (T1 rows), the bias planes from the pair state (T2 rows, the
// only part that touches the pair state), the segmented attention core over the token axis, gate + output projection.
template <typename T>
static nt_status single_attn_impl(const nt_layout* L, const Totals& tot, int c_s, int c_z, int H, int d,
                                  const nt_single_attn_weights* W, float eps, void* x, const void* z, void* ws,
                                  nt_dtype dt, cudaStream_t st) {
  SingleWs w = carve_single(ws, dt, tot, c_s, H, d);
  const int Hd = H * d;
  const bool fast = dt == NT_BF16 && !g_force_generic && fast_single_attn_supported(c_s, c_z, H, d);
  GroupIter it(L->lengths_h, L->B);
  BatchMeta m;
  while (it.next(m)) {
    const long long trow0 = m.tok_off[0], trows = m.tok_off[m.B] - trow0;
    const long long prow0 = m.pair_off[0], prows = m.pair_off[m.B] - prow0;
    if (trows == 0) continue;
    nt_status r;
    if (fast) {
      // tensor-core path: LayerNorm once (bf16), token GEMMs on mma.sync, bias planes written times sqrt(d) as the
      // attention core wants them, the segmented core over the token axis, gate, output GEMM accumulated into x
      const size_t e = 2;
      char* xr = (char*)x + (size_t)trow0 * c_s * e;
      char* xh = (char*)w.xh + (size_t)trow0 * c_s * e;
      const size_t to = (size_t)trow0 * Hd * e;
      if ((r = fast_ln_rows(xr, W->ln_gamma, W->ln_beta, eps, c_s, trows, xh, st)) != NT_OK) return r;
      const TokSeg seg[4] = {{xh, trows, W->W_q, Hd, (char*)w.q + to}, {xh, trows, W->W_k, Hd, (char*)w.k + to},
                             {xh, trows, W->W_v, Hd, (char*)w.v + to}, {xh, trows, W->W_g, Hd, (char*)w.g + to}};
      if ((r = fast_token_gemm(seg, 4, c_s, 0, 0, "single_attn_in", st)) != NT_OK) return r;
      if ((r = fast_single_bias(z, W->ln_z_gamma, W->ln_z_beta, W->W_b, eps, c_z, H, sqrtf((float)d), m, w.bias, st)) != NT_OK) return r;
      if ((r = fast_attn_core_fr(w.q, w.k, w.v, w.bias, w.o, H, d, FR_MODE_TOKEN, m, L->status_d, st)) != NT_OK) return r;
      if ((r = fast_gate_mul((char*)w.g + to, (char*)w.o + to, trows * Hd, st)) != NT_OK) return r;
      const TokSeg so = {(char*)w.o + to, trows, W->W_o, c_s, xr};
      if ((r = fast_token_gemm(&so, 1, Hd, 0, 1, "single_attn_out", st)) != NT_OK) return r;
      continue;
    }
    ProjArgs pa{};
    pa.A = x; pa.a_mode = A_ROWMAJOR; pa.row0 = trow0; pa.rows = trows; pa.K = c_s;
    pa.ln_g = W->ln_gamma; pa.ln_b = W->ln_beta; pa.eps = eps;
    pa.add(W->W_q, nullptr, Hd, ACT_NONE, w.q, O_STORE);
    pa.add(W->W_k, nullptr, Hd, ACT_NONE, w.k, O_STORE);
    pa.add(W->W_v, nullptr, Hd, ACT_NONE, w.v, O_STORE);
    pa.add(W->W_g, nullptr, Hd, ACT_SIGMOID, w.g, O_STORE);
    if ((r = launch_proj<T>(pa, m, st, "generic_single_attn_in")) != NT_OK) return r;
    ProjArgs pb{};
    pb.A = z; pb.a_mode = A_ROWMAJOR; pb.row0 = prow0; pb.rows = prows; pb.K = c_z;
    pb.ln_g = W->ln_z_gamma; pb.ln_b = W->ln_z_beta; pb.eps = eps;
    pb.add(W->W_b, nullptr, H, ACT_NONE, w.bias, O_CHANNEL_MAJOR);
    if ((r = launch_proj<T>(pb, m, st, "single_attn_bias")) != NT_OK) return r;
    r = launch_attn_core<T>((const T*)w.q, (const T*)w.k, (const T*)w.v, (const T*)w.bias, (T*)w.o, H, d, 0, m, st);
    if (r != NT_OK) return r;
    ProjArgs po{};
    po.A = w.o; po.a_mode = A_ROWMAJOR; po.row0 = trow0; po.rows = trows; po.K = Hd;
    po.gateA = w.g;
    po.add(W->W_o, nullptr, c_s, ACT_NONE, x, O_ACCUM);
    if ((r = launch_proj<T>(po, m, st, "single_attn_out")) != NT_OK) return r;
  }
  return NT_OK;
}

}  // namespace ntp

using namespace ntp;

extern "C" {

nt_status nt_pair_broadcast(const nt_layout* L, nt_dtype dt, int32_t c_s, int32_t c_z, const void* x,
                            const void* W_a, const void* W_b, const void* ln_gamma, const void* ln_beta,
                            float ln_eps, void* z, void* workspace, size_t workspace_bytes, nt_stream stream) {
  Totals tot;
  nt_status r = check_layout(L, tot);
  if (r != NT_OK) return r;
  if (dt != NT_F32 && dt != NT_BF16) return NT_ERR_UNSUPPORTED;
  if (c_s <= 0 || c_z <= 0) return NT_ERR_INVALID_ARG;
  if (tot.T2 == 0) return NT_OK;
  if (!x || !W_a || !W_b || !ln_gamma || !ln_beta || !z || !workspace) return NT_ERR_INVALID_ARG;
  if (!aligned16(x) || !aligned16(z) || !aligned16(workspace) || !aligned16(W_a) || !aligned16(W_b))
    return NT_ERR_INVALID_ARG;
  if (workspace_bytes < broadcast_ws_bytes(tot, c_z)) return NT_ERR_WORKSPACE;
  cudaStream_t st = (cudaStream_t)stream;
  if (dt == NT_F32)
    return pair_broadcast_impl<float>(L, tot, c_s, c_z, x, W_a, W_b, ln_gamma, ln_beta, ln_eps, z, workspace, st, false);
  const bool fast = !g_force_generic && fast_broadcast_supported(c_z);
  return pair_broadcast_impl<__nv_bfloat16>(L, tot, c_s, c_z, x, W_a, W_b, ln_gamma, ln_beta, ln_eps, z, workspace, st,
                                            fast);
}

nt_status nt_pair_broadcast_add(const nt_layout* L, nt_dtype dt, int32_t c_s, int32_t c_z, const void* x,
                            const void* W_a, const void* W_b, const void* ln_gamma, const void* ln_beta,
                            float ln_eps, void* z, void* workspace, size_t workspace_bytes, nt_stream stream) {
  Totals tot;
  nt_status r = check_layout(L, tot);
  if (r != NT_OK) return r;
  if (dt != NT_F32 && dt != NT_BF16) return NT_ERR_UNSUPPORTED;
  if (c_s <= 0 || c_z <= 0) return NT_ERR_INVALID_ARG;
  if (tot.T2 == 0) return NT_OK;
  if (!x || !W_a || !W_b || !ln_gamma || !ln_beta || !z || !workspace) return NT_ERR_INVALID_ARG;
  if (!aligned16(x) || !aligned16(z) || !aligned16(workspace) || !aligned16(W_a) || !aligned16(W_b))
    return NT_ERR_INVALID_ARG;
  if (workspace_bytes < broadcast_ws_bytes(tot, c_z)) return NT_ERR_WORKSPACE;
  cudaStream_t st = (cudaStream_t)stream;
  if (dt == NT_F32)
    return pair_broadcast_impl<float>(L, tot, c_s, c_z, x, W_a, W_b, ln_gamma, ln_beta, ln_eps, z, workspace, st, false, true);
  const bool fast = !g_force_generic && fast_broadcast_supported(c_z);
  return pair_broadcast_impl<__nv_bfloat16>(L, tot, c_s, c_z, x, W_a, W_b, ln_gamma, ln_beta, ln_eps, z, workspace, st,
                                            fast, true);
}

static nt_status tri_mul_entry(const nt_layout* L, nt_dtype dt, int32_t c_z, int32_t c_h, const nt_trimul_weights* W,
                               float ln_eps, void* z, void* workspace, size_t workspace_bytes, nt_stream stream,
                               bool incoming) {
  Totals tot;
  nt_status r = check_layout(L, tot);
  if (r != NT_OK) return r;
  if (dt != NT_F32 && dt != NT_BF16) return NT_ERR_UNSUPPORTED;
  if (c_z <= 0 || c_h <= 0 || !W) return NT_ERR_INVALID_ARG;
  if (!W->ln_in_gamma || !W->ln_in_beta || !W->W_ap || !W->W_ag || !W->W_bp || !W->W_bg || !W->W_g ||
      !W->ln_out_gamma || !W->ln_out_beta || !W->W_o || !weights_aligned16(W) || ((uintptr_t)W->prepared & 255))
    return NT_ERR_INVALID_ARG;
  if (tot.T2 == 0) return NT_OK;
  if (!z || !workspace || !aligned16(z) || !aligned16(workspace)) return NT_ERR_INVALID_ARG;
  if (workspace_bytes < carve_trimul(nullptr, dt, tot, c_z, c_h).bytes) return NT_ERR_WORKSPACE;
  cudaStream_t st = (cudaStream_t)stream;
  if (dt == NT_F32) return tri_mul_generic<float>(L, tot, c_z, c_h, W, ln_eps, z, workspace, dt, st, incoming);
  return tri_mul_generic<__nv_bfloat16>(L, tot, c_z, c_h, W, ln_eps, z, workspace, dt, st, incoming);
}

nt_status nt_tri_mul_out(const nt_layout* L, nt_dtype dt, int32_t c_z, int32_t c_h, const nt_trimul_weights* W,
                         float ln_eps, void* z, void* workspace, size_t workspace_bytes, nt_stream stream) {
  return tri_mul_entry(L, dt, c_z, c_h, W, ln_eps, z, workspace, workspace_bytes, stream, false);
}

nt_status nt_tri_mul_in(const nt_layout* L, nt_dtype dt, int32_t c_z, int32_t c_h, const nt_trimul_weights* W,
                        float ln_eps, void* z, void* workspace, size_t workspace_bytes, nt_stream stream) {
  return tri_mul_entry(L, dt, c_z, c_h, W, ln_eps, z, workspace, workspace_bytes, stream, true);
}

nt_status nt_row_attn_pairbias(const nt_layout* L, nt_order order, nt_dtype dt, int32_t c, int32_t H, int32_t d,
                               const nt_attn_weights* W, float ln_eps, void* zx, void* workspace,
                               size_t workspace_bytes, nt_stream stream) {
  Totals tot;
  nt_status r = check_layout(L, tot);
  if (r != NT_OK) return r;
  if (dt != NT_F32 && dt != NT_BF16) return NT_ERR_UNSUPPORTED;
  if (order != NT_ORDER_PAIR_IJC && order != NT_ORDER_TOKEN_NC) return NT_ERR_UNSUPPORTED;
  if (c <= 0 || H <= 0 || d <= 0 || !W) return NT_ERR_INVALID_ARG;
  if (!W->W_q || !W->W_k || !W->W_v || !W->W_o || !weights_aligned16(W) || ((uintptr_t)W->prepared & 255)) return NT_ERR_INVALID_ARG;
  if ((W->ln_gamma == nullptr) != (W->ln_beta == nullptr)) return NT_ERR_INVALID_ARG;
  if (order == NT_ORDER_TOKEN_NC && W->W_b) return NT_ERR_INVALID_ARG;
  if (d > 128) return NT_ERR_UNSUPPORTED;
  const long long rows = order == NT_ORDER_PAIR_IJC ? tot.T2 : tot.T1;
  if (rows == 0) return NT_OK;
  if (!zx || !workspace || !aligned16(zx) || !aligned16(workspace)) return NT_ERR_INVALID_ARG;
  if (workspace_bytes < carve_attn(nullptr, dt, tot, order, H, d).bytes) return NT_ERR_WORKSPACE;
  cudaStream_t st = (cudaStream_t)stream;
  if (dt == NT_F32) return attn_generic<float>(L, tot, order, c, H, d, W, ln_eps, zx, workspace, dt, st, false);
  return attn_generic<__nv_bfloat16>(L, tot, order, c, H, d, W, ln_eps, zx, workspace, dt, st, false);
}

nt_status nt_row_attn_pairbias_mean(const nt_layout* L, nt_dtype dt, int32_t c, int32_t H, int32_t d,
                                    const nt_attn_weights* W, float ln_eps, void* z, void* m_out, void* workspace,
                                    size_t workspace_bytes, nt_stream stream) {
  Totals tot;
  nt_status r = check_layout(L, tot);
  if (r != NT_OK) return r;
  if (dt != NT_F32 && dt != NT_BF16) return NT_ERR_UNSUPPORTED;
  if (c <= 0 || H <= 0 || d <= 0 || !W) return NT_ERR_INVALID_ARG;
  if (!W->W_q || !W->W_k || !W->W_v || !W->W_o || !weights_aligned16(W) || ((uintptr_t)W->prepared & 255)) return NT_ERR_INVALID_ARG;
  if ((W->ln_gamma == nullptr) != (W->ln_beta == nullptr)) return NT_ERR_INVALID_ARG;
  if (d > 128) return NT_ERR_UNSUPPORTED;
  if (tot.T1 == 0) return NT_OK;
  if (!m_out || !aligned16(m_out) || !L->row_splits_d) return NT_ERR_INVALID_ARG;
  if (!z || !workspace || !aligned16(z) || !aligned16(workspace)) return NT_ERR_INVALID_ARG;
  if (workspace_bytes < carve_attn(nullptr, dt, tot, NT_ORDER_PAIR_IJC, H, d).bytes) return NT_ERR_WORKSPACE;
  cudaStream_t st = (cudaStream_t)stream;
  bool done = false;
  if (dt == NT_F32)
    r = attn_generic<float>(L, tot, NT_ORDER_PAIR_IJC, c, H, d, W, ln_eps, z, workspace, dt, st, false, m_out, &done);
  else
    r = attn_generic<__nv_bfloat16>(L, tot, NT_ORDER_PAIR_IJC, c, H, d, W, ln_eps, z, workspace, dt, st, false, m_out, &done);
  if (r != NT_OK || done) return r;
  // some part of the batch went through a path without the fused reduction: reduce the finished state as a whole
  return nt_segment_reduce(dt, NT_REDUCE_MEAN, c, tot.T1, tot.T2, L->row_splits_d, z, m_out, L->status_d, stream);
}

nt_status nt_col_attn_pairbias(const nt_layout* L, nt_dtype dt, int32_t c, int32_t H, int32_t d,
                               const nt_attn_weights* W, float ln_eps, void* z, void* workspace,
                               size_t workspace_bytes, nt_stream stream) {
  Totals tot;
  nt_status r = check_layout(L, tot);
  if (r != NT_OK) return r;
  if (dt != NT_F32 && dt != NT_BF16) return NT_ERR_UNSUPPORTED;
  if (c <= 0 || H <= 0 || d <= 0 || !W) return NT_ERR_INVALID_ARG;
  if (!W->W_q || !W->W_k || !W->W_v || !W->W_o || !weights_aligned16(W) || ((uintptr_t)W->prepared & 255)) return NT_ERR_INVALID_ARG;
  if ((W->ln_gamma == nullptr) != (W->ln_beta == nullptr)) return NT_ERR_INVALID_ARG;
  if (d > 128) return NT_ERR_UNSUPPORTED;
  if (tot.T2 == 0) return NT_OK;
  if (!z || !workspace || !aligned16(z) || !aligned16(workspace)) return NT_ERR_INVALID_ARG;
  if (workspace_bytes < carve_attn(nullptr, dt, tot, NT_ORDER_PAIR_IJC, H, d).bytes) return NT_ERR_WORKSPACE;
  cudaStream_t st = (cudaStream_t)stream;
  if (dt == NT_F32) return attn_generic<float>(L, tot, NT_ORDER_PAIR_IJC, c, H, d, W, ln_eps, z, workspace, dt, st, true);
  return attn_generic<__nv_bfloat16>(L, tot, NT_ORDER_PAIR_IJC, c, H, d, W, ln_eps, z, workspace, dt, st, true);
}

nt_status nt_single_attn_pairbias(const nt_layout* L, nt_dtype dt, int32_t c_s, int32_t c_z, int32_t H, int32_t d,
                                  const nt_single_attn_weights* W, float ln_eps, void* x, const void* z,
                                  void* workspace, size_t workspace_bytes, nt_stream stream) {
  Totals tot;
  nt_status r = check_layout(L, tot);
  if (r != NT_OK) return r;
  if (dt != NT_F32 && dt != NT_BF16) return NT_ERR_UNSUPPORTED;
  if (c_s <= 0 || c_z <= 0 || H <= 0 || d <= 0 || !W) return NT_ERR_INVALID_ARG;
  if (!W->ln_gamma || !W->ln_beta || !W->W_q || !W->W_k || !W->W_v || !W->W_g || !W->W_o || !W->ln_z_gamma ||
      !W->ln_z_beta || !W->W_b)
    return NT_ERR_INVALID_ARG;
  if (d > 128) return NT_ERR_UNSUPPORTED;
  if (tot.T1 == 0) return NT_OK;
  if (!x || !z || !workspace || !aligned16(x) || !aligned16(z) || !aligned16(workspace)) return NT_ERR_INVALID_ARG;
  if (workspace_bytes < carve_single(nullptr, dt, tot, c_s, H, d).bytes) return NT_ERR_WORKSPACE;
  cudaStream_t st = (cudaStream_t)stream;
  if (dt == NT_F32) return single_attn_impl<float>(L, tot, c_s, c_z, H, d, W, ln_eps, x, z, workspace, dt, st);
  return single_attn_impl<__nv_bfloat16>(L, tot, c_s, c_z, H, d, W, ln_eps, x, z, workspace, dt, st);
}

size_t nt_single_attn_workspace_bytes(nt_dtype dt, const int64_t* lengths_h, int32_t B, int32_t c_s, int32_t H, int32_t d) {
  if (B <= 0 || !lengths_h || c_s <= 0 || H <= 0 || d <= 0 || (dt != NT_F32 && dt != NT_BF16)) return 0;
  Totals tot;
  if (totals_of(lengths_h, B, tot) != NT_OK) return 0;
  return carve_single(nullptr, dt, tot, c_s, H, d).bytes;
}

nt_status nt_segment_reduce(nt_dtype dt, nt_reduce op, int32_t C, int64_t G, int64_t rows, const int64_t* splits_d,
                            const void* v, void* out, int32_t* status_d, nt_stream stream) {
  (void)status_d;
  if (dt != NT_F32 && dt != NT_BF16) return NT_ERR_UNSUPPORTED;
  if (op != NT_REDUCE_MEAN && op != NT_REDUCE_SUM) return NT_ERR_UNSUPPORTED;
  if (C <= 0 || G < 0 || rows < 0) return NT_ERR_INVALID_ARG;
  if (G == 0) return NT_OK;
  if (!splits_d || !out || (rows > 0 && !v)) return NT_ERR_INVALID_ARG;
  if (!aligned16(v) || !aligned16(out)) return NT_ERR_INVALID_ARG;
  cudaStream_t st = (cudaStream_t)stream;
  const int mean = op == NT_REDUCE_MEAN;
  if (dt == NT_F32) return launch_segment_reduce<float>((const float*)v, (float*)out, splits_d, G, C, mean, st);
  if (!g_force_generic && fast_segment_reduce_supported(C))
    return fast_segment_reduce(v, out, splits_d, G, C, mean, st);
  return launch_segment_reduce<__nv_bfloat16>((const __nv_bfloat16*)v, (__nv_bfloat16*)out, splits_d, G, C, mean, st);
}

nt_status nt_token_update(nt_dtype dt, int32_t c_s, int32_t c_z, int64_t T1, const void* mvals, const void* W_r,
                          void* x, nt_stream stream) {
  if (dt != NT_F32 && dt != NT_BF16) return NT_ERR_UNSUPPORTED;
  if (c_s <= 0 || c_z <= 0 || T1 < 0) return NT_ERR_INVALID_ARG;
  if (T1 == 0) return NT_OK;
  if (!mvals || !W_r || !x) return NT_ERR_INVALID_ARG;
  BatchMeta dummy;
  fill_meta(dummy, nullptr, 0, 0, 0, 0, 0);
  ProjArgs pa{};
  pa.A = mvals; pa.a_mode = A_ROWMAJOR; pa.row0 = 0; pa.rows = T1; pa.K = c_z;
  pa.add(W_r, nullptr, c_s, ACT_NONE, x, O_ACCUM);
  cudaStream_t st = (cudaStream_t)stream;
  if (dt == NT_F32) return launch_proj<float>(pa, dummy, st, "token_update");
  if (!g_force_generic && fast_token_gemm_supported(c_z, c_s, 0)) {
    const TokSeg seg = {mvals, T1, W_r, c_s, x};
    return fast_token_gemm(&seg, 1, c_z, 0, 1, "token_update", st);
  }
  return launch_proj<__nv_bfloat16>(pa, dummy, st, "token_update");
}

// rows of the hidden activation the generic transition keeps in the workspace at a time
static const long long TRANSITION_BLOCK_ROWS = 1 << 16;

size_t nt_transition_workspace_bytes(nt_dtype dt, int32_t c, int32_t hidden, int64_t rows) {
  if (c <= 0 || hidden <= 0 || rows <= 0) return 0;
  const size_t e = dt == NT_F32 ? 4 : 2;
  const long long blk = rows < TRANSITION_BLOCK_ROWS ? rows : TRANSITION_BLOCK_ROWS;
  return align_up((size_t)blk * hidden * e, 256) + (1 << 20);
}

nt_status nt_pair_transition(nt_dtype dt, int32_t c, int32_t hidden, int64_t rows, const nt_transition_weights* W,
                             float ln_eps, void* z, void* workspace, size_t workspace_bytes, int32_t* status_d,
                             nt_stream stream) {
  if (dt != NT_F32 && dt != NT_BF16) return NT_ERR_UNSUPPORTED;
  if (c <= 0 || hidden <= 0 || rows < 0 || !W) return NT_ERR_INVALID_ARG;
  if (rows == 0) return NT_OK;
  if (!W->ln_gamma || !W->ln_beta || !W->W_a || !W->W_b || !W->W_2 || !z) return NT_ERR_INVALID_ARG;
  if (!aligned16(z) || !aligned16(workspace) || !weights_aligned16(W)) return NT_ERR_INVALID_ARG;
  if (!workspace || workspace_bytes < nt_transition_workspace_bytes(dt, c, hidden, rows)) return NT_ERR_WORKSPACE;
  cudaStream_t st = (cudaStream_t)stream;
  const size_t e = dt == NT_F32 ? 4 : 2;
  const long long blk = rows < TRANSITION_BLOCK_ROWS ? rows : TRANSITION_BLOCK_ROWS;
  char* hbuf = (char*)workspace;
  char* prep = hbuf + align_up((size_t)blk * hidden * e, 256);
  if (dt == NT_BF16 && !g_force_generic && fast_transition_supported(c, hidden))
    return fast_transition(z, W, ln_eps, c, hidden, rows, prep, status_d, st);
  BatchMeta dummy;
  fill_meta(dummy, nullptr, 0, 0, 0, 0, 0);
  for (long long r0 = 0; r0 < rows; r0 += blk) {
    const long long n = rows - r0 < blk ? rows - r0 : blk;
    char* zr = (char*)z + (size_t)r0 * c * e;
    ProjArgs pa{};
    pa.A = zr; pa.a_mode = A_ROWMAJOR; pa.row0 = 0; pa.rows = n; pa.K = c;
    pa.ln_g = W->ln_gamma; pa.ln_b = W->ln_beta; pa.eps = ln_eps;
    pa.add(W->W_a, W->W_b, hidden, ACT_SILU, hbuf, O_STORE);
    ProjArgs po{};
    po.A = hbuf; po.a_mode = A_ROWMAJOR; po.row0 = 0; po.rows = n; po.K = hidden;
    po.add(W->W_2, nullptr, c, ACT_NONE, zr, O_ACCUM);
    nt_status r = dt == NT_F32 ? launch_proj<float>(pa, dummy, st, "generic_transition_in")
                               : launch_proj<__nv_bfloat16>(pa, dummy, st, "generic_transition_in");
    if (r != NT_OK) return r;
    r = dt == NT_F32 ? launch_proj<float>(po, dummy, st, "generic_transition_out")
                     : launch_proj<__nv_bfloat16>(po, dummy, st, "generic_transition_out");
    if (r != NT_OK) return r;
  }
  return NT_OK;
}

size_t nt_workspace_bytes(nt_op op, nt_dtype dt, nt_order order, const int64_t* lengths_h, int32_t B,
                          const int32_t* dims) {
  if (B <= 0 || !lengths_h || !dims) return 0;
  Totals tot;
  if (totals_of(lengths_h, B, tot) != NT_OK) return 0;
  const int c_z = dims[1], c_h = dims[2], H = dims[3], d = dims[4];
  size_t bb = broadcast_ws_bytes(tot, c_z);
  size_t tb = carve_trimul(nullptr, dt, tot, c_z, c_h).bytes;
  size_t ab = carve_attn(nullptr, dt, tot, order, H, d).bytes;
  switch (op) {
    case NT_OP_PAIR_BROADCAST: return bb;
    case NT_OP_TRI_MUL_OUT: return tb;
    case NT_OP_ROW_ATTN: return ab;
    case NT_OP_BLOCK: { size_t mx = bb > tb ? bb : tb; return mx > ab ? mx : ab; }
  }
  return 0;
}

const char* nt_status_string(nt_status st) {
  switch (st) {
    case NT_OK: return "ok";
    case NT_ERR_INVALID_ARG: return "invalid argument";
    case NT_ERR_UNSUPPORTED: return "unsupported dtype, width or order";
    case NT_ERR_WORKSPACE: return "workspace too small";
    case NT_ERR_CUDA: return "CUDA call failed";
    case NT_ERR_TIMEOUT: return "device wait timed out";
    case NT_ERR_INCONSISTENT: return "totals disagree with lengths";
  }
  return "unknown status";
}

int64_t nt_launch_count(void) { return g_launches.load(); }

int32_t nt_profile_begin(void) {
  std::lock_guard<std::mutex> lk(g_prof_mu);
  for (auto& r : g_prof) { cudaEventDestroy(r.e0); cudaEventDestroy(r.e1); }
  g_prof.clear();
  g_prof_on = true;
  return 0;
}

int32_t nt_profile_end(char* names, size_t names_bytes, float* total_ms, int64_t* launches, int32_t max_entries) {
  std::lock_guard<std::mutex> lk(g_prof_mu);
  g_prof_on = false;
  std::vector<std::string> nm;
  std::vector<float> ms;
  std::vector<long long> cnt;
  for (auto& r : g_prof) {
    float t = 0.f;
    cudaEventSynchronize(r.e1);
    cudaEventElapsedTime(&t, r.e0, r.e1);
    size_t k = 0;
    for (; k < nm.size(); ++k) if (nm[k] == r.name) break;
    if (k == nm.size()) { nm.push_back(r.name); ms.push_back(0.f); cnt.push_back(0); }
    ms[k] += t;
    cnt[k] += 1;
    cudaEventDestroy(r.e0);
    cudaEventDestroy(r.e1);
  }
  g_prof.clear();
  std::string joined;
  int32_t n = 0;
  for (size_t k = 0; k < nm.size() && n < max_entries; ++k) {
    if (joined.size() + nm[k].size() + 2 > names_bytes) break;
    joined += nm[k];
    joined += '\n';
    if (total_ms) total_ms[n] = ms[k];
    if (launches) launches[n] = cnt[k];
    ++n;
  }
  if (names && names_bytes) {
    std::memcpy(names, joined.c_str(), joined.size() + 1);
  }
  return n;
}

nt_status nt_debug_expire_wait(int32_t* status_d, int64_t limit_clocks, int32_t* observed_d, nt_stream stream) {
  if (!status_d || limit_clocks < 1 || limit_clocks > (1ll << 24)) return NT_ERR_INVALID_ARG;
  return launch_expire_wait(status_d, limit_clocks, observed_d, (cudaStream_t)stream);
}

nt_status nt_prepare_trimul_weights(nt_dtype dt, int32_t c_z, int32_t c_h, const nt_trimul_weights* W, void* prepared_out,
                                    size_t prepared_bytes, nt_stream stream) {
  if (!W || !prepared_out || ((size_t)prepared_out & 255) || prepared_bytes < NT_PREPARED_WEIGHTS_BYTES) return NT_ERR_INVALID_ARG;
  if (!W->ln_in_gamma || !W->ln_in_beta || !W->W_ap || !W->W_ag || !W->W_bp || !W->W_bg || !W->W_g || !W->ln_out_gamma ||
      !W->ln_out_beta || !W->W_o)
    return NT_ERR_INVALID_ARG;
  if (dt != NT_BF16 || !fast_tri_in_supported(c_z, c_h) || !fast_tri_out_supported(c_z, c_h))
    return NT_ERR_UNSUPPORTED;
  TriPrep tp{};
  return fast_tri_prep(W, c_z, c_h, prepared_out, tp, (cudaStream_t)stream);
}

nt_status nt_prepare_attn_weights(nt_dtype dt, int32_t c, int32_t H, int32_t d, const nt_attn_weights* W, void* prepared_out,
                                  size_t prepared_bytes, nt_stream stream) {
  if (!W || !prepared_out || ((size_t)prepared_out & 255) || prepared_bytes < NT_PREPARED_WEIGHTS_BYTES) return NT_ERR_INVALID_ARG;
  if (!W->ln_gamma || !W->ln_beta || !W->W_q || !W->W_k || !W->W_v || !W->W_o) return NT_ERR_INVALID_ARG;
  if (dt != NT_BF16 || !(fast_attn_in_supported(c, H, d) || (W->W_g && fast_attn_out_supported(c, H, d)))) return NT_ERR_UNSUPPORTED;
  AttnPrep ap{};
  return fast_attn_prep(W, c, H, d, prepared_out, ap, (cudaStream_t)stream);
}

nt_status nt_bench_exp_rate(int32_t variant, int32_t iters, int32_t blocks, float* sink_d, int64_t* clocks_d,
                            nt_stream stream) {
  if (!sink_d || !clocks_d || iters < 1 || blocks < 1 || blocks > 4096) return NT_ERR_INVALID_ARG;
  return launch_exp_rate(variant, iters, blocks, sink_d, (long long*)clocks_d, (cudaStream_t)stream);
}

nt_status nt_debug_bounds_report(int32_t* out_h, int32_t reset) {
#ifdef NT_DEBUG_BOUNDS
  if (!out_h) return NT_ERR_INVALID_ARG;
  int v[4] = {0, 0, 0, 0};
  if (cudaMemcpyFromSymbol(v, g_nt_bounds, sizeof(v)) != cudaSuccess) return cuda_fail("bounds report");
  for (int i = 0; i < 4; ++i) out_h[i] = v[i];
  if (reset) {
    const int z[4] = {0, 0, 0, 0};
    if (cudaMemcpyToSymbol(g_nt_bounds, z, sizeof(z)) != cudaSuccess) return cuda_fail("bounds reset");
  }
  return NT_OK;
#else
  (void)out_h;
  (void)reset;
  return NT_ERR_UNSUPPORTED;
#endif
}

int32_t nt_debug_attn_drop(int32_t blocks) {
  int32_t prev = g_fr_drop;
  g_fr_drop = blocks;
  return prev;
}

int32_t nt_attn_core_mode(int32_t mode) {
  int32_t prev = g_fr_all;
  g_fr_all = mode != 0;
  return prev;
}

int32_t nt_force_generic(int32_t on) {
  int32_t prev = g_force_generic;
  g_force_generic = on;
  return prev;
}

}  // extern "C"
