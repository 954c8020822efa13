/*
 * libnested_pair -- forward pass of a Pairformer-style block on a packed multi-ragged pair state.
 *
 * The pair state of a batch of B samples with lengths N_s is stored as T2 = sum_s N_s^2 packed
 * positions (never as a padded B x N_max^2 envelope).  Storage follows the paper's packed
 * representation (Sec. 3.1, Eq. 2): ragged axes first, static feature axis last, row-major,
 * samples concatenated; sample offsets o_0 = 0, o_{s+1} - o_s = N_s^2, o_B = T2 (App. A).
 * The packed row of logical coordinate (s, i, j) is  p = pair_off[s] + i * N_s + j  (Eq. 3).
 *
 * Common conventions for every call
 *   - All value / weight pointers are DEVICE pointers unless the name ends in _h (host).
 *   - Buffers are contiguous, channel-last; weights are [out, in] row-major (V' = V W^T, Sec. 3.3);
 *     there are no linear bias vectors anywhere.
 *   - dtype NT_F32: float storage, float arithmetic.  NT_BF16: bf16 storage of values and weights, float
 *     accumulation, float LayerNorm / softmax statistics.  Intermediates that never leave the workspace are bf16
 *     (q, k, v, o, bias) or, on the tensor-core path, fp16 where three more significant bits pay: the
 *     LayerNorm-folded weights, the triangle update's a, b (gated projections of a normalised row) and t / N_s.
 *     fp16 ends at 65504: the folded weights and the offsets W beta of the input projections and of the transition have
 *     to lie below; a, b and t / N_s are clamped to its finite range when they are written, so a state with
 *     absurdly large projections saturates instead of producing infinities.
 *   - A process may drive several devices: per-kernel launch attributes are kept per device.
 *   - The caller owns every buffer.  No call allocates, frees or synchronises; all work is
 *     enqueued on `stream` (a cudaStream_t passed as an opaque pointer; NULL = default stream).
 *   - Pointers must be 16-byte aligned.
 *   - Host-checkable errors are returned with nothing launched.  Device-detected conditions
 *     (offset totals that disagree with T1/T2, a bounded wait that expired) are written to
 *     *status_d (sticky; first error wins) and the kernel exits normally.
 *   - B = 0 or T2 = 0 is a valid no-op.  Zero-length samples are legal (coincident offsets) and
 *     contribute nothing.
 *   - Canonical sizes stay on the host with device mirrors (App. A): the layout carries both.
 */
#ifndef NESTED_PAIR_H
#define NESTED_PAIR_H

#include <stddef.h>
#include <stdint.h>

#ifdef __cplusplus
extern "C" {
#endif

typedef enum {
  NT_OK = 0,
  NT_ERR_INVALID_ARG = 1,   /* null pointer, negative size, misaligned pointer            */
  NT_ERR_UNSUPPORTED = 2,   /* dtype / width / order not implemented                       */
  NT_ERR_WORKSPACE = 3,     /* workspace smaller than nt_workspace_bytes()                 */
  NT_ERR_CUDA = 4,          /* a CUDA runtime / driver call failed                         */
  NT_ERR_TIMEOUT = 5,       /* device: a bounded wait expired                              */
  NT_ERR_INCONSISTENT = 6   /* T1 / T2 disagree with the lengths                           */
} nt_status;

typedef enum { NT_F32 = 0, NT_BF16 = 1 } nt_dtype;

/* logical dimension order of a packed buffer (ragged axes first, then the static feature axis) */
typedef enum {
  NT_ORDER_TOKEN_NC = 0,    /* [sum N, C]                                                  */
  NT_ORDER_PAIR_IJC = 1     /* [sum N^2, C], i major, j minor                              */
} nt_order;

typedef enum { NT_REDUCE_MEAN = 0, NT_REDUCE_SUM = 1 } nt_reduce;

typedef enum {
  NT_OP_PAIR_BROADCAST = 0, NT_OP_TRI_MUL_OUT = 1, NT_OP_ROW_ATTN = 2, NT_OP_BLOCK = 3 /* max of the three */
} nt_op;

typedef void *nt_stream;    /* cudaStream_t */

/* The partitions of one batch (Sec. 3.1 "Structural metadata"). */
typedef struct {
  int32_t B;                    /* samples                                                  */
  int64_t T1, T2;               /* sum N_s and sum N_s^2, computed by the caller            */
  const int64_t *lengths_h;     /* host   [B]    canonical sizes                            */
  const int64_t *lengths_d;     /* device [B]                                               */
  const int64_t *tok_off_d;     /* device [B+1]  exclusive prefix of N_s                    */
  const int64_t *pair_off_d;    /* device [B+1]  exclusive prefix of N_s^2                  */
  const int64_t *row_splits_d;  /* device [T1+1] level-2 splits: start of every pair row    */
  int32_t *status_d;            /* device [1], nullable                                     */
} nt_layout;

typedef struct {                /* triangle multiplicative update; all device, dtype = dt   */
  const void *ln_in_gamma, *ln_in_beta;     /* [c_z]                                        */
  const void *W_ap, *W_ag, *W_bp, *W_bg;    /* [c_h, c_z]                                   */
  const void *W_g;                          /* [c_z, c_z]                                   */
  const void *ln_out_gamma, *ln_out_beta;   /* [c_h]                                        */
  const void *W_o;                          /* [c_z, c_h]                                   */
  const void *prepared;                     /* NULL, or what nt_prepare_trimul_weights wrote for THESE weights */
} nt_trimul_weights;

typedef struct {                /* row-wise attention; all device, dtype = dt               */
  const void *ln_gamma, *ln_beta;           /* [c]      both NULL -> no LayerNorm           */
  const void *W_q, *W_k, *W_v;              /* [H*d, c]                                     */
  const void *W_b;                          /* [H, c]   NULL -> zero bias                   */
  const void *W_g;                          /* [H*d, c] NULL -> no gate                     */
  const void *W_o;                          /* [c, H*d]                                     */
  const void *prepared;                     /* NULL, or what nt_prepare_attn_weights wrote for THESE weights   */
} nt_attn_weights;

typedef struct {                /* pair-biased single attention; all device, dtype = dt     */
  const void *ln_gamma, *ln_beta;           /* [c_s]    LayerNorm of the tokens             */
  const void *W_q, *W_k, *W_v;              /* [H*d, c_s]                                   */
  const void *W_g;                          /* [H*d, c_s]                                   */
  const void *W_o;                          /* [c_s, H*d]                                   */
  const void *ln_z_gamma, *ln_z_beta;       /* [c_z]    LayerNorm of the pair state         */
  const void *W_b;                          /* [H, c_z]                                     */
} nt_single_attn_weights;

/*
 * nt_offsets_build -- prefix sums and position decode (Sec. 3.1 offsets o; Fig. 2 two-level row
 * splits; Eq. 3 coordinate map; the rows/columns gather indices of the program figure).
 *   tok_off[s]  = sum_{s'<s} N_s',  pair_off[s] = sum_{s'<s} N_s'^2            (each [B+1])
 *   row_splits[tok_off[s]+i] = pair_off[s] + i N_s,  row_splits[T1] = T2        ([T1+1], nullable)
 *   for p = pair_off[s] + i N_s + j: pos_sample[p]=s, pos_i[p]=i, pos_j[p]=j    (int32 [T2], nullable as a group)
 *                                    gather_rows[p]=tok_off[s]+i, gather_cols[p]=tok_off[s]+j (int64 [T2], nullable as a group)
 * Integer work, bit-exact.  If the scanned totals differ from T1 / T2, NT_ERR_INCONSISTENT is
 * written to *status_d and only the two offset arrays are produced.
 */
nt_status nt_offsets_build(const int64_t *lengths_d, int32_t B, int64_t T1, int64_t T2,
                           int64_t *tok_off_d, int64_t *pair_off_d, int64_t *row_splits_d,
                           int32_t *pos_sample_d, int32_t *pos_i_d, int32_t *pos_j_d,
                           int64_t *gather_rows_d, int64_t *gather_cols_d,
                           int32_t *status_d, nt_stream stream);

/*
 * nt_pair_broadcast -- ragged outer broadcast that creates the N_s x N_s axes from packed token
 * features, fused with LayerNorm (Eq. 1 line 1; Sec. 3.2 "Creating axes through broadcasting";
 * no activation at construction, App. A.1):
 *   u = x W_a^T, v = x W_b^T ([T1, c_z]);  z[p,:] = LN_{c_z}(u[tok_off[s]+i] + v[tok_off[s]+j]) * gamma + beta.
 *   x [T1, c_s] in;  z [T2, c_z] out (exactly T2 * c_z elements).
 */
nt_status nt_pair_broadcast(const nt_layout *L, nt_dtype dt, int32_t c_s, int32_t c_z,
                            const void *x, const void *W_a, const void *W_b,
                            const void *ln_gamma, const void *ln_beta, float ln_eps,
                            void *z, void *workspace, size_t workspace_bytes, nt_stream stream);

/*
 * nt_pair_broadcast_add -- the same broadcast accumulated onto the state: z[p,:] += LN(u_i + v_j) * gamma + beta.
 * For a pair state that persists across blocks (the Pairformer's pair stream) instead of being rebuilt from the
 * tokens by every block (Eq. 1).  z [T2, c_z] in/out; everything else as nt_pair_broadcast.
 */
nt_status nt_pair_broadcast_add(const nt_layout *L, nt_dtype dt, int32_t c_s, int32_t c_z,
                            const void *x, const void *W_a, const void *W_b,
                            const void *ln_gamma, const void *ln_beta, float ln_eps,
                            void *z, void *workspace, size_t workspace_bytes, nt_stream stream);

/*
 * nt_tri_mul_out -- outgoing triangle multiplicative update (the Pairformer block's triangle
 * multiplication, Sec. 4.3), a per-sample grouped contraction over channels:
 *   zh = LN_in(z); a = sig(zh W_ag^T) * (zh W_ap^T); b = sig(zh W_bg^T) * (zh W_bp^T); g = sig(zh W_g^T)
 *   t_s[i,j,c] = sum_k a_s[i,k,c] b_s[j,k,c];   z += g * (LN_out(t) W_o^T)      (in place)
 *   z [T2, c_z] in/out.  No weight pointer may be NULL.
 */
nt_status nt_tri_mul_out(const nt_layout *L, nt_dtype dt, int32_t c_z, int32_t c_h,
                         const nt_trimul_weights *W, float ln_eps, void *z,
                         void *workspace, size_t workspace_bytes, nt_stream stream);

/*
 * nt_tri_mul_in -- incoming triangle multiplicative update: the second direction of the block's triangle
 * multiplication (Sec. 4.3).  Same projections, gate, output normalisation, residual, weights, workspace and
 * error behaviour as nt_tri_mul_out; only the contraction runs over the FIRST pair index:
 *   t_s[i,j,c] = sum_k a_s[k,i,c] b_s[k,j,c];   z += g * (LN_out(t) W_o^T)      (in place)
 *   z [T2, c_z] in/out.  Workspace size: nt_workspace_bytes (the same as for nt_tri_mul_out).
 */
nt_status nt_tri_mul_in(const nt_layout *L, nt_dtype dt, int32_t c_z, int32_t c_h,
                         const nt_trimul_weights *W, float ln_eps, void *z,
                         void *workspace, size_t workspace_bytes, nt_stream stream);

/*
 * nt_row_attn_pairbias -- row-wise pair-biased softmax attention over ragged N_s (Sec. 3.3
 * "Attention through packed blocks": segments from the offsets, output adopts the query
 * structure; Sec. 4.3 triangle attention, starting node).
 *   order = NT_ORDER_PAIR_IJC: zx = z [T2, c]; attention rows are the pair rows (s, i); for each
 *     row and head h: S[j,k] = <q_ij, k_ik>/sqrt(d) + bias[j,k,h] with bias = LN(z) W_b^T shared by
 *     all rows of the sample; P = softmax_k S; o_ij = sum_k P[j,k] v_ik; z += (g * o) W_o^T.
 *   order = NT_ORDER_TOKEN_NC: zx = x [T1, c]; one attention row per sample (variable-length
 *     self-attention over the token segments); W_b must be NULL.
 *   zx in/out (in place).  H * d need not equal c.
 *   Range of the logits (bf16 path): the softmax is taken against a reference that need not be the
 *     row maximum.  Samples of up to 224 tokens use the bound max_k(q.k)/sqrt(d) + max_k(bias) of the
 *     query (the first maximum also runs over the up to 15 keys of the next pair row that pad the
 *     last group of 16); a row whose true maximum lies more than about 80 nats below that bound
 *     loses its weights to underflow (its output row is then not finite).  Longer samples, token order and d = 64 have no
 *     such limit: their reference is guessed from the query's previous row, and a row whose log-sum lies more than 42 nats
 *     below or 97 above that row's is computed a second time with a running maximum (a call in which nearly every row does
 *     so takes two to three times as long).  Activations that have passed a LayerNorm and projections of O(1) norm stay far inside
 *     either range.
 */
nt_status nt_row_attn_pairbias(const nt_layout *L, nt_order order, nt_dtype dt,
                               int32_t c, int32_t H, int32_t d,
                               const nt_attn_weights *W, float ln_eps, void *zx,
                               void *workspace, size_t workspace_bytes, nt_stream stream);

/*
 * nt_row_attn_pairbias_mean -- nt_row_attn_pairbias in pair order followed by the mean over j of the updated state
 * (Eq. 1 line 3, Eq. 4), in one call: where the tensor-core output stage runs, the column sums are taken from its
 * tiles while they are still on chip and the state is not read back for the reduction.
 *   z [T2, c] in/out as nt_row_attn_pairbias; m_out [T1, c] out (dtype dt): m_out[tok_off[s]+i,:] = mean_j z[(s,i,j),:]
 *   of the UPDATED state, accumulated in float, i.e. what nt_segment_reduce(NT_REDUCE_MEAN, row_splits) returns on it
 *   (the order of the float additions differs, so the two may differ by rounding).
 *   L->row_splits_d must be present (used when a part of the batch takes a path without the fused reduction:
 *   float data, a sample shorter than 32, shapes outside the tensor-core stage).
 *   Workspace and errors as nt_row_attn_pairbias.
 */
nt_status nt_row_attn_pairbias_mean(const nt_layout *L, nt_dtype dt, int32_t c, int32_t H, int32_t d,
                                    const nt_attn_weights *W, float ln_eps, void *z, void *m_out,
                                    void *workspace, size_t workspace_bytes, nt_stream stream);

/*
 * nt_col_attn_pairbias -- column-wise pair-biased softmax attention over ragged N_s: the second triangle
 * attention of the block (Sec. 4.3, "ending node"), the mirror image of nt_row_attn_pairbias in pair order.
 *   Attention rows are the pair COLUMNS (s, j); for each column and head h:
 *     S[i,k] = <q_ij, k_kj>/sqrt(d) + bias[k,i,h] with bias = LN(z) W_b^T shared by all columns of the sample;
 *     P = softmax_k S; o_ij = sum_k P[i,k] v_kj; z += (g * o) W_o^T.
 *   z [T2, c] in/out (in place).  Same weights structure, workspace size (nt_workspace_bytes) and error behaviour
 *   as nt_row_attn_pairbias with order = NT_ORDER_PAIR_IJC.  Keys of a column are N_s packed rows apart; nothing
 *   is transposed in memory.
 */
nt_status nt_col_attn_pairbias(const nt_layout *L, nt_dtype dt, int32_t c, int32_t H, int32_t d,
                               const nt_attn_weights *W, float ln_eps, void *z,
                               void *workspace, size_t workspace_bytes, nt_stream stream);

/*
 * nt_single_attn_pairbias -- pair-biased single attention (Sec. 4.3): the tokens of a sample attend the tokens of
 * the same sample, the logits biased by a projection of the sample's pair state; one segmented call for the
 * whole batch (Sec. 3.3 "Attention through packed blocks": segments from the offsets).
 *   xh = LN(x); q,k,v = xh W_{q,k,v}^T; g = sig(xh W_g^T); bias[j,k,h] = (LN_z(z_jk) W_b^T)[h]
 *   S[h,j,k] = <q_jh, k_kh>/sqrt(d) + bias[j,k,h]; P = softmax_k S; o_jh = sum_k P[h,j,k] v_kh; x += (g * o) W_o^T
 *   x [T1, c_s] in/out (in place); z [T2, c_z] in (not modified).  No weight pointer may be NULL.  d <= 128.
 *   Workspace: nt_single_attn_workspace_bytes (0 when the batch is empty or an argument is invalid).
 */
nt_status nt_single_attn_pairbias(const nt_layout *L, nt_dtype dt, int32_t c_s, int32_t c_z, int32_t H, int32_t d,
                                  const nt_single_attn_weights *W, float ln_eps, void *x, const void *z,
                                  void *workspace, size_t workspace_bytes, nt_stream stream);
size_t nt_single_attn_workspace_bytes(nt_dtype dt, const int64_t *lengths_h, int32_t B, int32_t c_s, int32_t H, int32_t d);

/*
 * Rectangular pairs (N_s, M_s): the method's second pair layout (Eq. 2: pairs (N_i, M_i, C) pack as (sum N_i M_i, C);
 * cell (s, a, b) lives at packed row pair_off[s] + a M_s + b).
 *
 * nt_rect_offsets_build -- prefix sums and cell decode of a batch of rectangular pairs.
 *   tokn_off[s] = sum_{s'<s} N_s', tokm_off[s] = sum_{s'<s} M_s', pair_off[s] = sum_{s'<s} N_s' M_s'   (each [B+1])
 *   row_splits[tokn_off[s]+a] = pair_off[s] + a M_s, row_splits[T1n] = T2  ([T1n+1], nullable): one group of M_s cells
 *     per row, the groups the column reduction of Eq. 4 consumes (nt_segment_reduce over them; its mean divides by M_s)
 *   pos_sample / pos_i / pos_j [T2] (int32, nullable as a group): the decode of every cell
 *   lengths_n_d, lengths_m_d [B] device int64.  Integer work, bit-exact; inconsistent totals or a negative length
 *   write NT_ERR_INCONSISTENT to *status_d.
 *
 * nt_rect_pair_broadcast -- z[(s,a,b),:] = LN(W_a x_{s,a} + W_b y_{s,b}) * gamma + beta from distinct row tokens
 *   x [T1n, c_s] and column tokens y [T1m, c_s] (App. A.1); z [T2, c_z] out (exactly T2 * c_z elements).
 *   lengths_n_h, lengths_m_h [B] HOST int64 (read during the call).  Workspace: nt_rect_broadcast_workspace_bytes.
 *   Errors as nt_pair_broadcast.
 */
nt_status nt_rect_offsets_build(const int64_t *lengths_n_d, const int64_t *lengths_m_d, int32_t B,
                                int64_t T1n, int64_t T1m, int64_t T2,
                                int64_t *tokn_off_d, int64_t *tokm_off_d, int64_t *pair_off_d, int64_t *row_splits_d,
                                int32_t *pos_sample_d, int32_t *pos_i_d, int32_t *pos_j_d,
                                int32_t *status_d, nt_stream stream);
nt_status nt_rect_pair_broadcast(nt_dtype dt, int32_t B, const int64_t *lengths_n_h, const int64_t *lengths_m_h,
                                 int32_t c_s, int32_t c_z, const void *x, const void *y,
                                 const void *W_a, const void *W_b, const void *ln_gamma, const void *ln_beta,
                                 float ln_eps, void *z, void *workspace, size_t workspace_bytes, nt_stream stream);
size_t nt_rect_broadcast_workspace_bytes(const int64_t *lengths_n_h, const int64_t *lengths_m_h, int32_t B, int32_t c_z);

/*
 * nt_segment_reduce -- segmented sum or mean of contiguous row groups (Eq. 4 pair reduction; the
 * mean over j of Eq. 1 line 3 divides by the group's count; App. A batch-axis convention).
 *   out[g,:] = (1/len_g or 1) * sum_{r = splits[g]}^{splits[g+1]-1} v[r,:],  empty group -> 0.
 *   splits [G+1] device, nondecreasing, splits[0] = 0, splits[G] = rows.  v [rows, C]; out [G, C].
 *   With splits = row_splits this is the mean over j back to the token axis; with
 *   splits = tok_off it pools a token buffer per sample.  Accumulation is in float.
 */
nt_status nt_segment_reduce(nt_dtype dt, nt_reduce op, int32_t C, int64_t G, int64_t rows,
                            const int64_t *splits_d, const void *v, void *out,
                            int32_t *status_d, nt_stream stream);

/*
 * nt_pair_broadcast_static -- nt_pair_broadcast without a caller workspace.  (The paper has no
 * counterpart: this entry point exists for integration, not for the method.)
 *
 * Same arguments, result and error behaviour as nt_pair_broadcast, minus `workspace`: the scratch
 * for the projected token features lives in a fixed array inside the library's device module.  It is
 * meant for callers that cannot allocate device memory themselves: an embedding application whose
 * interface passes only input and output pointers, or a serving loop that must never call
 * cudaMalloc (a device-wide synchronising call that can fail when memory is fragmented).
 *   - Limit: the batch must need at most NT_PAIR_BROADCAST_STATIC_BYTES of scratch, i.e. what
 *     nt_workspace_bytes(NT_OP_PAIR_BROADCAST, ...) returns: the two projected token arrays in float,
 *     each as two bf16 arrays as well (high and low parts) and their squared norms, 2 *
 *     (round_up(T1 * c_z * 4, 256) + 2 * round_up(T1 * c_z * 2, 256) + round_up(T1 * 4, 256)) bytes
 *     (about T1 * c_z <= 520,000); larger batches are refused with NT_ERR_WORKSPACE and a message on
 *     stderr, with nothing launched.
 *   - Every GPU that loads the library holds the array (NT_PAIR_BROADCAST_STATIC_BYTES) until the
 *     process exits.
 *   - The first call on each device looks up the array's device address (no allocation, no
 *     synchronisation); make that first call before any stream capture begins.
 *   - All calls share the one array and it keeps whatever the last call left in it.  Nothing in it
 *     needs clearing (every call overwrites what it reads), but two calls that overlap on the GPU --
 *     different streams, or different host threads -- race on it: serialise them.
 *   - The call itself performs no cudaMalloc / cudaFree and uses no allocating library routine.
 */
#define NT_PAIR_BROADCAST_STATIC_BYTES (8u << 20)
nt_status nt_pair_broadcast_static(const nt_layout *L, nt_dtype dt, int32_t c_s, int32_t c_z,
                                   const void *x, const void *W_a, const void *W_b,
                                   const void *ln_gamma, const void *ln_beta, float ln_eps,
                                   void *z, nt_stream stream);

/*
 * nt_pair_transition -- the SwiGLU feature update of the pair state (Eq. 1 line 2: P~ = P + h(LN(P)), h the
 * SwiGLU update named there; expansion four in the paper's settings, App. A.1), position-wise on packed values:
 *   zh = LN(z);  z += (silu(zh W_a^T) * (zh W_b^T)) W_2^T.
 *   z [rows, c] in/out (in place), row-major, dtype dt; rows = T2 for the pair state (any packed [rows, c]
 *   buffer works: no sample structure enters).  W_a, W_b [hidden, c], W_2 [c, hidden], ln_gamma, ln_beta [c]:
 *   device pointers of dtype dt, none may be NULL.  workspace: device scratch of at least
 *   nt_transition_workspace_bytes(...) bytes (hidden activations of a block of rows on the generic path, folded
 *   weights on the tensor-core path); the call allocates nothing and keeps no state.
 *   Errors: NT_ERR_INVALID_ARG (NULL pointer, non-positive width, rows < 0), NT_ERR_UNSUPPORTED (dtype),
 *   NT_ERR_WORKSPACE, NT_ERR_CUDA; a device-side wait that runs out reports NT_ERR_TIMEOUT in *status_d (nullable).
 */
typedef struct { const void *ln_gamma, *ln_beta, *W_a, *W_b, *W_2; } nt_transition_weights;
nt_status nt_pair_transition(nt_dtype dt, int32_t c, int32_t hidden, int64_t rows,
                             const nt_transition_weights *W, float ln_eps, void *z,
                             void *workspace, size_t workspace_bytes, int32_t *status_d, nt_stream stream);
size_t nt_transition_workspace_bytes(nt_dtype dt, int32_t c, int32_t hidden, int64_t rows);

/* ------------------------------- auxiliaries (not among the five) ------------------------------- */

/* x[T1, c_s] += m[T1, c_z] W_r^T  -- the projection g of Eq. 1 line 3 applied to the reduced
 * features and added to the tokens.  W_r is [c_s, c_z]. */
nt_status nt_token_update(nt_dtype dt, int32_t c_s, int32_t c_z, int64_t T1,
                          const void *m, const void *W_r, void *x, nt_stream stream);

/* Bytes of workspace a call needs for this batch.  dims = {c_s, c_z, c_h, H, d}; entries an op
 * does not use are ignored.  Host only.  Returns 0 for an empty batch. */
size_t nt_workspace_bytes(nt_op op, nt_dtype dt, nt_order order, const int64_t *lengths_h, int32_t B,
                          const int32_t *dims);

const char *nt_status_string(nt_status st);

/* Number of kernels the library has launched in this process since load (all calls). */
int64_t nt_launch_count(void);

/* Per-kernel timing for benchmarks.  Between nt_profile_begin() and nt_profile_end() every kernel the
 * library launches is bracketed by a pair of CUDA events on its stream.  nt_profile_end() waits for
 * those events and aggregates by kernel name: names are written to `names` separated by '\n', with
 * total milliseconds and launch counts in the parallel arrays; it returns the number of entries.
 * Host-side only; off by default; not thread-safe against concurrent library calls. */
int32_t nt_profile_begin(void);
int32_t nt_profile_end(char *names, size_t names_bytes, float *total_ms, int64_t *launches, int32_t max_entries);

/*
 * nt_prepare_trimul_weights / nt_prepare_attn_weights -- fold the LayerNorm parameters into the projection weights
 * once, ahead of the calls that use them.  The bf16 tensor-core stages of nt_tri_mul_out / nt_tri_mul_in and of the
 * pair-order nt_row_attn_pairbias / nt_row_attn_pairbias_mean / nt_col_attn_pairbias multiply the raw state tile by
 * LayerNorm-folded weights (W diag(gamma) in fp16, with the per-row constants W beta and the row sums) and would
 * otherwise rebuild those from the weights structure in a small launch of their own on every call.  Weights are
 * constant across calls in inference and across the micro-steps of a training step, so a caller may do it once:
 *   prepared_out   device, NT_PREPARED_WEIGHTS_BYTES bytes, 256-byte aligned, owned by the caller; it must stay
 *                  valid and unchanged while a weights structure points at it (field `prepared`).
 * The call is asynchronous on `stream`; a later call that finds `prepared` non-NULL uses it as it is and launches no
 * preparation (stream order is the caller's business).  The library keeps no state: `prepared` is just another
 * input.  With NT_F32, with shapes outside the tensor-core stages, or under nt_force_generic the field is ignored.
 * Returns NT_ERR_INVALID_ARG for null / misaligned pointers or a short buffer, NT_ERR_UNSUPPORTED for shapes the
 * tensor-core stages do not take (nothing is launched in either case).  The paper has no counterpart: its operators
 * take module weights as they are (Sec. 3.3 "feature-wise operators act directly on V").
 */
#define NT_PREPARED_WEIGHTS_BYTES ((size_t)1 << 20)
nt_status nt_prepare_trimul_weights(nt_dtype dt, int32_t c_z, int32_t c_h, const nt_trimul_weights *W,
                                    void *prepared_out, size_t prepared_bytes, nt_stream stream);
nt_status nt_prepare_attn_weights(nt_dtype dt, int32_t c, int32_t H, int32_t d, const nt_attn_weights *W,
                                  void *prepared_out, size_t prepared_bytes, nt_stream stream);

/* Measurement aid: the exponential rate of an SM, the third ceiling of the attention core's roofline.  Launches
 * `blocks` CTAs of 512 threads; every thread runs `iters` rounds of eight independent exponentials and the CTA
 * writes the SM clocks the loop took to clocks_d[block].  variant 0: ex2.approx.f32 (special-function unit);
 * 1: ex2.approx.bf16x2 (two results per instruction); 2: a polynomial on the FMA pipe only; 3..6: (variant - 2) of
 * every eight exponentials on the FMA pipe, the rest on the special-function unit; 7 / 8: variant 0 with the
 * results packed to bf16 pairs by cvt.rn.bf16x2.f32 / by integer add and prmt; 9: the softmax inner loop of the
 * attention cores on registers (16 exponentials per round); 10: the same with CTAs of 256 threads.  sink_d: device float
 * [blocks * 512] (keeps the work alive); clocks_d: device int64 [blocks].  Results per clock and SM =
 * 512 * 8 * iters (* 2 for variants 1 and 9) / clocks.  Asynchronous on `stream`; NT_ERR_INVALID_ARG for null pointers,
 * an unknown variant or counts out of range (nothing launched). */
nt_status nt_bench_exp_rate(int32_t variant, int32_t iters, int32_t blocks, float *sink_d, int64_t *clocks_d,
                            nt_stream stream);

/* Debugging aid of the CHECKED build (compiled with -DNT_DEBUG_BOUNDS -rdc=true; see build.py, variant "checked").
 * In that build every kernel tests the global indices it derives from the offsets against the extents its buffers
 * were given at the boundary; a stray index is counted, the first one is recorded and the access is skipped (the
 * checked build never faults, it reports).  out_h: host int32[4] = {violations, site of the first (a small code
 * naming the kernel and the buffer), its index low word, high word}.  reset != 0 clears the record.  Synchronises
 * the device (it reads a device variable): a debugging call, not part of any hot path.  In the normal build the
 * checks are compiled out and this returns NT_ERR_UNSUPPORTED. */
nt_status nt_debug_bounds_report(int32_t *out_h, int32_t reset);

/* Testing aid for the failure path of device-side waits.  Every wait inside the tensor-core kernels is bounded: when
 * its limit runs out the kernel writes NT_ERR_TIMEOUT to the layout's status word (first error wins), raises a flag
 * that makes the CTA's later waits give up quickly, and still ends normally, so the context stays usable.  This call
 * launches one tiny kernel (one CTA) whose only wait is on a barrier nobody arrives at, with a limit of
 * limit_clocks SM clocks (1 .. 2^24, i.e. at most a few milliseconds), so that a test can watch that path without any
 * fault, trap or unbounded loop.  status_d: device int32, receives NT_ERR_TIMEOUT if it held NT_OK; observed_d:
 * device int32, nullable, receives bit 0 = the wait gave up, bit 1 = the abort flag was raised.  Asynchronous on
 * `stream`.  Returns NT_ERR_INVALID_ARG (nothing launched) for a null status_d or a limit out of range. */
nt_status nt_debug_expire_wait(int32_t *status_d, int64_t limit_clocks, int32_t *observed_d, nt_stream stream);

/* Testing aid for the failure path of the register-fragment attention core: from now on each of its CTAs requests only
 * `blocks` blocks of 64 keys and then stops, so that the waits for the next one run out (about a second), the status word
 * receives NT_ERR_TIMEOUT and the kernel ends (the call's output is then undefined).  Negative (the default): all blocks.
 *  Returns the previous value. */
int32_t nt_debug_attn_drop(int32_t blocks);

/* Testing aid: the bf16 pair-order attention uses two tensor-core kernels, one that holds a whole score row
 * on chip (samples of up to 224 tokens) and one that walks the keys in blocks (longer samples).  mode 1 sends every
 * sample to the second kernel, mode 0 restores the split by length.  Returns the previous mode. */
int32_t nt_attn_core_mode(int32_t mode);

/* Testing aid: non-zero forces the shape-generic CUDA-core kernels even where a tensor-core
 * kernel exists for the shape.  Returns the previous value.  Both settings run on the GPU. */
int32_t nt_force_generic(int32_t on);

#ifdef __cplusplus
}
#endif
#endif /* NESTED_PAIR_H */
