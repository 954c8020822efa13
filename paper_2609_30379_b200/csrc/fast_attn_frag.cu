// Segmented pair-biased softmax attention for any sample length: scores on tcgen05, softmax weights in the
// register fragments of the second product.
//
// Work item: 128 queries of NT attention rows that see the same bias tile (pair order: rows i .. i + NT - 1 of one
// (sample, head, query block); token order without bias: NT heads of one (sample, query block); token order with
// bias: one row).  Each row is a "tile" with its own Q, K, V; keys come in blocks of 64.
// Per tile and block:
//   S = Q K^T       tcgen05, M = 128 queries, N = 64 keys, K = d, into one of the tile's two TMEM buffers;
//   softmax         four warps per tile, 32 queries each, 32 keys (a chunk) at a time.  S is read with
//                   tcgen05.ld.16x256b, whose register layout is the accumulator fragment of mma.m16n8k16: the weights
//                   exp2(S log2(e) / sqrt(d) + bias - ref), packed to bf16, ARE the A operand of the second product,
//                   and the bias comes in the same layout straight from its shared-memory tile by ldmatrix;
//   O += P V        mma.sync m16n8k16 from those registers (V by ldmatrix.trans), O stays in registers.
// Why this split: the exponentials bound the work (16 per clock and SM) and everything else has to hide behind them.
// With P handed over through shared memory the tile's P store, the MMA's re-read of it and the hand-over between warps
// cost more than the exponentials: 128 x 128 scores moved 150 KB through shared memory (1190 clocks at 128 B per clock,
// against 1024 for the exponentials) and every block was a chain of four barrier hops.  Here P and O never leave the
// registers and shared memory carries 96 KB per 128 x 128 scores.  mma.sync is the slower tensor path (8.4 clocks per
// m16n8k16 and quarter of an SM, measured), but the product needs only half (d = 32) or a quarter (d = 16) of the
// clocks the exponentials take.
// Tiles per CTA: three for d <= 32 (12 softmax warps of 152 registers: a warp alone reaches 14.4 clocks per 32
// exponentials and quarter of an SM, two 9.5, three 9.0 at d = 16; the unit's rate is 8), two for d = 64.
// Measured (B200, against the kernel with P in shared memory): lengths 384-2048, d = 16: 28.9 -> 20.0 ms per launch;
// one sample of 977, d = 32: 2457 -> 1589 us; token order, 7.4 k tokens, 12 x 64: 48.6 -> 34.9 us.  Counters: 10.4
// (d = 16) and 12.3 (d = 32) clocks per 32 exponentials in the loop, plus 660 and 970 per row.
#include <cstring>

#include "fast.cuh"
#include "tc_common.cuh"

namespace ntp {

constexpr int FR_KEYS = 64;                    // keys per block
constexpr int FR_MAXSTAGE = 8;
constexpr int FR_ITEM_COST = 2;                // per-item work, in chunks of 32 keys
constexpr int FR_BIAS_BYTES = 128 * 128;       // 128 queries x 64 keys, bf16, 128-byte swizzle
constexpr float FR_LOG2E = 1.4426950408889634f;
// The reference of a row is not its maximum but a guess from the query's previous row, FR_MARGIN binades above that
// row's log-sum, which any softmax may take as long as nothing overflows or vanishes: the weights have the whole
// exponent range of float and bf16, so the guess may be off by 60 binades downwards and 140 upwards.  A row whose sum
// leaves [FR_LOW, FR_HIGH] is computed again with a running maximum, by the warp alone (fr_exact_row).
constexpr float FR_MARGIN = 40.f;
constexpr float FR_HIGH = 1.2676506e30f;       // 2^100
constexpr float FR_LOW = 7.8886091e-31f;       // 2^-100

struct AttnFrParams {
  CUtensorMap qmap, kmap, vmap;   // flat {H d, rows}, box {d, 64}
  CUtensorMap cmap[MAXB];         // column mode, per sample: {H d, first pair index (stride N H d), column, which of q / k / v}, box {d, 64, 1, 1}
  CUtensorMap bmap[MAXB];         // per sample: bias planes {N keys, N queries, H}, box {64, 128, 1}, 128-byte swizzle
  BatchMeta m;
  long long item_off[MAXB + 1];   // prefix of the item counts
  long long cost_off[MAXB + 1];   // prefix of item count x (chunks + FR_ITEM_COST)
  const __nv_bfloat16 *q, *k, *v, *bias;   // as given (exact rows); bias nullable
  __nv_bfloat16* o;
  long long row0;                 // first row the flat maps cover
  long long rows;                 // rows the flat maps (and the output) cover from row0 on
  int H, mode, nstage, single_tile;
  float sc2;                      // log2(e) / sqrt(d)
  int drop;                       // testing aid: a CTA requests only this many key blocks (< 0: all)
  int* status;
};

// What the softmax warps need to know about an item; the producer leaves it beside the item's first stage.
struct FrInfo {
  int N, q0, tiles, step;         // row length, first query of the block, tiles with a row, packed rows between queries
  int orow, head, tile_row, tile_head;   // output row of the block's first query and head of tile 0; what tile t adds per t
  long long bias_plane;           // element offset of the (sample, head of tile 0) bias plane
  int ld, pad;
};

// Position in the item order.  Only the first item of a CTA is found by division; the rest follow by counting.
template <int NT>
struct FrItem {
  int s, N, njb, groups;          // groups: row groups of the sample (token order: head groups)
  int h, jb, g;                   // head, query block, row group
  __device__ inline void load_sample(const AttnFrParams& p) {
    N = p.m.N[s];
    njb = (N + 127) >> 7;
    groups = p.mode == FR_MODE_TOKEN ? (p.single_tile ? p.H : (p.H + NT - 1) / NT) : (N + NT - 1) / NT;
  }
  __device__ inline void seek(const AttnFrParams& p, long long item) {
    s = 0;
    while (s + 1 < p.m.B && item >= p.item_off[s + 1]) ++s;
    load_sample(p);
    const unsigned local = (unsigned)(item - p.item_off[s]);
    if (p.mode == FR_MODE_TOKEN) {       // (head group, query block)
      g = (int)(local / (unsigned)njb);
      jb = (int)(local - (unsigned)g * njb);
      h = 0;
    } else {                             // (head, query block, row group)
      const unsigned t = local / (unsigned)groups;
      g = (int)(local - t * groups);
      h = (int)(t / (unsigned)njb);
      jb = (int)(t - (unsigned)h * njb);
    }
  }
  __device__ inline void next(const AttnFrParams& p) {
    if (p.mode == FR_MODE_TOKEN) {
      if (++jb < njb) return;
      jb = 0;
      if (++g < groups) return;
      g = 0;
    } else {
      if (++g < groups) return;
      g = 0;
      if (++jb < njb) return;
      jb = 0;
      if (++h < p.H) return;
      h = 0;
    }
    do ++s; while (s < p.m.B && p.item_off[s + 1] == p.item_off[s]);
    if (s < p.m.B) load_sample(p);
  }
  __device__ inline int tiles(const AttnFrParams& p) const {     // tiles of the item that have a row
    if (p.single_tile) return 1;
    const int left = (p.mode == FR_MODE_TOKEN ? p.H : N) - g * NT;
    return left < NT ? left : NT;
  }
  __device__ inline int head(const AttnFrParams& p, int t) const {
    return p.mode == FR_MODE_TOKEN ? (p.single_tile ? g : g * NT + t) : h;
  }
  // flat row (relative to row0) of key 0 of tile t (row mode and token order)
  __device__ inline int kvrow(const AttnFrParams& p, int t) const {
    return p.mode == FR_MODE_TOKEN ? (int)(p.m.tok_off[s] - p.row0) : (int)(p.m.pair_off[s] - p.row0) + (g * NT + t) * N;
  }
};

// number of items that start before cost position x (0 <= x <= total cost)
__device__ inline long long fr_ordinal_at(const AttnFrParams& p, long long x) {
  const int B = p.m.B;
  if (x >= p.cost_off[B]) return p.item_off[B];
  int s = 0;
  while (s + 1 < B && x >= p.cost_off[s + 1]) ++s;
  const long long c = (p.m.N[s] + 31) / 32 + FR_ITEM_COST;
  return p.item_off[s] + (x - p.cost_off[s] + c - 1) / c;
}

__device__ inline float fr_exp2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;\n" : "=f"(y) : "f"(x));
  return y;
}
__device__ inline unsigned fr_pack(float lo, float hi) {
  unsigned y;
  asm("cvt.rn.bf16x2.f32 %0, %1, %2;\n" : "=r"(y) : "f"(hi), "f"(lo));
  return y;
}
// v += the two bf16 halves of b: the mixed-precision add widens the half exactly, which saves the unpacking
// (10.96 -> 10.34 clocks per 32 exponentials and quarter of an SM at d = 32)
__device__ inline float2 fr_bias_add(float2 v, unsigned b) {
  asm("{\n\t.reg .b16 l, h;\n\tmov.b32 {l, h}, %2;\n\tadd.rn.f32.bf16 %0, l, %0;\n\tadd.rn.f32.bf16 %1, h, %1;\n\t}\n"
      : "+f"(v.x), "+f"(v.y) : "r"(b));
  return v;
}
__device__ inline void fr_mma(float (&c)[4], const unsigned (&a)[4], unsigned b0, unsigned b1) {
  asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3},{%4,%5,%6,%7},{%8,%9},{%0,%1,%2,%3};\n"
               : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
               : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ inline void fr_ldsm(unsigned addr, unsigned (&r)[4]) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];\n"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr));
}
__device__ inline void fr_ldsm_t(unsigned addr, unsigned (&r)[4]) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];\n"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr));
}
// 16 lanes (queries) x 32 columns (keys): register 4 j + e of lane l is query l / 4 + 8 (e / 2), key 8 j + 2 (l % 4) + e % 2
__device__ inline void fr_tmem_ld(unsigned taddr, unsigned (&r)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.16x256b.x4.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];\n"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr) : "memory");
}
// the scores of a chunk: 32 queries x 32 keys
__device__ inline void fr_request_scores(unsigned s_addr, unsigned (&s)[2][16]) {
  fr_tmem_ld(s_addr, s[0]);
  fr_tmem_ld(s_addr + (16u << 16), s[1]);
}
// keys nv .. 31 of a chunk's scores become -inf
__device__ inline void fr_mask(unsigned (&s)[2][16], int nv, int lane) {
#pragma unroll
  for (int e = 0; e < 16; ++e) {
    const bool none = (e >> 2) * 8 + 2 * (lane & 3) + (e & 1) >= nv;
    s[0][e] = none ? 0xff800000u : s[0][e];
    s[1][e] = none ? 0xff800000u : s[1][e];
  }
}
// one arrival per warp, predicated instead of branched around
__device__ inline void fr_arrive(unsigned bar, int lane) {
  asm volatile("{\n\t.reg .pred p;\n\tsetp.eq.s32 p, %1, 0;\n\t@p mbarrier.arrive.shared::cta.b64 _, [%0];\n\t}\n"
               ::"r"(bar), "r"(lane) : "memory");
}
// whether the barrier's phase is complete, without waiting (try_wait would suspend the warp)
__device__ inline bool fr_ready(void* bar, unsigned parity) {
  unsigned ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.b32 %0, 1, 0, p;\n\t}\n"
      : "=r"(ok) : "r"(smem_u32(bar)), "r"(parity) : "memory");
  return ok != 0;
}
// The auxiliary warps' wait: they have a block's time in hand, and a warp that probes a barrier all the time takes issue
// slots from the exponentials (a parked try_wait came back so often that the four warps took a tenth of the slots).
// False: the wait ran out (as with mbar_wait).  A warp of this kernel then works through no further item, because what it
// waited for may not be there, and because its later waits mean nothing: a barrier that has stopped satisfies every other
// parity wait at once.
__device__ inline bool fr_wait_idle(void* bar, unsigned parity, const AbortCtx& ab) {
  if (fr_ready(bar, parity)) return true;
  const long long t0 = clock64();
  for (unsigned it = 0; it < WAIT_PROBES; ++it) {
    __nanosleep(200);
    if (fr_ready(bar, parity)) return true;
    if ((it & 15u) == 15u && (clock64() - t0 > (*ab.flag ? WAIT_CLOCKS_ABORTED : WAIT_CLOCKS) || *ab.flag)) break;
  }
  if (!*ab.flag) {
    *ab.flag = 1;
    if (ab.status) atomicCAS(ab.status, 0, (int)NT_ERR_TIMEOUT);
  }
  return false;
}
// swizzled operand descriptor for a K-major tile whose rows are `span` = 32, 64 or 128 bytes
__device__ inline unsigned long long fr_desc(unsigned saddr, int span) {
  unsigned long long d = 0;
  d |= (unsigned long long)((saddr & 0x3FFFFu) >> 4);
  d |= (unsigned long long)(((unsigned)(8 * span) >> 4) & 0x3FFF) << 16;
  d |= (unsigned long long)(((unsigned)(8 * span) >> 4) & 0x3FFF) << 32;
  d |= (unsigned long long)1 << 46;
  d |= (unsigned long long)(span == 128 ? 2 : span == 64 ? 4 : 6) << 61;
  return d;
}

// Weights of a 32-key chunk from its scores s (-inf: no key): pk[mt][kt] is the A fragment of queries 16 mt .. and keys
// 16 kt .. of the warp; l[r] sums this lane's weights of query row r = 2 mt + half (query 16 mt + 8 half + lane / 4).
// The product of the PREVIOUS chunk (its weights prev, its V at v_prev) is issued in between, so that the tensor pipe
// works in the shadow of the exponentials (one after the other, a 64-key block took 1330 clocks of weights plus 500 of
// products at d = 32, measured).  Straight-line code: scores requested before it may land while it runs.
template <int D, bool HAS_BIAS>
__device__ inline void fr_weights(const unsigned (&s)[2][16], unsigned bias_addr, int odd, float sc2, const float (&nref)[4],
                                  float2 (&l)[4], unsigned (&pk)[2][2][4], float (&o)[2][D / 8][4],
                                  const unsigned (&prev)[2][2][4], unsigned v_prev) {
  const float2 sc22 = make_float2(sc2, sc2);
#pragma unroll
  for (int kt = 0; kt < 2; ++kt) {
    unsigned v[D / 16][4];
#pragma unroll
    for (int g = 0; g < D / 16; ++g) fr_ldsm_t((v_prev + kt * 16 * 2 * D) ^ (g << 5), v[g]);
#pragma unroll
    for (int mt = 0; mt < 2; ++mt) {
      unsigned b[4] = {0u, 0u, 0u, 0u};
      if (HAS_BIAS) fr_ldsm((bias_addr + mt * 16 * 128) ^ ((odd * 4 + kt * 2) << 4), b);
#pragma unroll
      for (int q = 0; q < 4; ++q) {      // q & 1: query half; q >> 1: key octet
        const int e = (2 * kt + (q >> 1)) * 4 + (q & 1) * 2, r = 2 * mt + (q & 1);
        float2 x = make_float2(__uint_as_float(s[mt][e]), __uint_as_float(s[mt][e + 1]));
        if (HAS_BIAS) x = fr_bias_add(x, b[q]);
        x = __ffma2_rn(x, sc22, make_float2(nref[r], nref[r]));
        const float2 w = make_float2(fr_exp2(x.x), fr_exp2(x.y));
        l[r] = __fadd2_rn(l[r], w);
        pk[mt][kt][q] = fr_pack(w.x, w.y);
#pragma unroll
        for (int k = q * (D / 8) / 4; k < (q + 1) * (D / 8) / 4; ++k)
          fr_mma(o[mt][k], prev[mt][kt], v[k >> 1][(k & 1) * 2], v[k >> 1][(k & 1) * 2 + 1]);
      }
    }
  }
}

// O += P V for a 32-key chunk
template <int D>
__device__ inline void fr_pv(float (&o)[2][D / 8][4], const unsigned (&pk)[2][2][4], unsigned v_addr) {
#pragma unroll
  for (int kt = 0; kt < 2; ++kt) {
    unsigned v[D / 16][4];
#pragma unroll
    for (int g = 0; g < D / 16; ++g) fr_ldsm_t((v_addr + kt * 16 * 2 * D) ^ (g << 5), v[g]);
#pragma unroll
    for (int mt = 0; mt < 2; ++mt)
#pragma unroll
      for (int k = 0; k < D / 8; ++k) fr_mma(o[mt][k], pk[mt][kt], v[k >> 1][(k & 1) * 2], v[k >> 1][(k & 1) * 2 + 1]);
  }
}

// The reference of a query that has none yet (the first row a warp meets): the maximum over the first chunk.
template <bool HAS_BIAS>
__device__ inline void fr_first_reference(const unsigned (&s)[2][16], unsigned bias_addr, float sc2, float (&nref)[4]) {
#pragma unroll
  for (int mt = 0; mt < 2; ++mt) {
    float mx[2] = {-INFINITY, -INFINITY};
#pragma unroll
    for (int kt = 0; kt < 2; ++kt) {
      unsigned b[4] = {0u, 0u, 0u, 0u};
      if (HAS_BIAS) fr_ldsm((bias_addr + mt * 16 * 128) ^ ((kt * 2) << 4), b);
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int e = (2 * kt + (q >> 1)) * 4 + (q & 1) * 2;
        float2 x = make_float2(__uint_as_float(s[mt][e]), __uint_as_float(s[mt][e + 1]));
        if (HAS_BIAS) x = fr_bias_add(x, b[q]);
        mx[q & 1] = fmaxf(mx[q & 1], fmaxf(x.x, x.y));
      }
    }
#pragma unroll
    for (int hf = 0; hf < 2; ++hf) {
      mx[hf] = fmaxf(mx[hf], __shfl_xor_sync(0xffffffffu, mx[hf], 1));
      mx[hf] = fmaxf(mx[hf], __shfl_xor_sync(0xffffffffu, mx[hf], 2));
      // (a first chunk without a finite score says nothing; references stay finite, or every later row would be computed twice)
      nref[2 * mt + hf] = -((fabsf(mx[hf]) < 1e30f ? mx[hf] * sc2 : 0.f) + FR_MARGIN);
    }
  }
}

// The warp's 32 queries of a row again, from memory, with a running maximum and mma.sync for both products: rows whose sum
// left the window (scores that differ by tens of nats from those of the query's previous row).  It stores the output
// itself and returns the log2-sums of the lane's four query rows, from which the next row's references follow.
// Fragments straight from memory, 16 keys a step: some 30 loads and 200 other instructions per 512 scores, and nothing in
// flight between steps.  Rows come here one by one and their references follow.  Measured where nearly every row comes here
// (rows a hundred nats apart, whole row attention call): one sample of 400, 4 heads of 16, 0.50 ms against 0.23 for ordinary
// rows; of 977, 5.3 against 1.6, and 3.7 against 1.2 with 2 heads of 32.  With a query per lane and scalar loads the
// sample of 400 took 114 ms.
template <int D, bool HAS_BIAS>
static __device__ __noinline__ float4 fr_exact_row(const AttnFrParams& p, const FrInfo& inf, int t, int quarter, int lane) {
  const int N = inf.N, q0 = inf.q0 + quarter * 32, gr = lane >> 2, c2 = 2 * (lane & 3);
  const long long pitch = (long long)p.H * D * inf.step;                        // elements between consecutive queries / keys
  const long long key0 = (p.row0 + inf.orow + (long long)t * inf.tile_row - (long long)inf.q0 * inf.step) * p.H * D +
                         (inf.head + t * inf.tile_head) * D;                    // the row's key 0
  const __nv_bfloat16* bias = HAS_BIAS ? p.bias + inf.bias_plane : nullptr;
  auto ld2 = [](const __nv_bfloat16* a) { return *reinterpret_cast<const unsigned*>(a); };
  unsigned qa[2][D / 16][4];
#pragma unroll
  for (int mt = 0; mt < 2; ++mt)
#pragma unroll
    for (int hf = 0; hf < 2; ++hf) {
      const __nv_bfloat16* qp = p.q + key0 + min(q0 + mt * 16 + hf * 8 + gr, N - 1) * pitch + c2;
#pragma unroll
      for (int ks = 0; ks < D / 16; ++ks) {
        qa[mt][ks][hf] = ld2(qp + ks * 16);
        qa[mt][ks][hf + 2] = ld2(qp + ks * 16 + 8);
      }
    }
  float o[2][D / 8][4], l[4], mx[4];
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    l[r] = 0.f;
    mx[r] = -INFINITY;
  }
#pragma unroll
  for (int mt = 0; mt < 2; ++mt)
#pragma unroll
    for (int k = 0; k < D / 8; ++k)
#pragma unroll
      for (int e = 0; e < 4; ++e) o[mt][k][e] = 0.f;
#pragma unroll 1
  for (int k0 = 0; k0 < N; k0 += 16) {
    float s[2][2][4] = {};                       // [query half of the warp][key octet]
#pragma unroll
    for (int nt = 0; nt < 2; ++nt) {
      const __nv_bfloat16* kp = p.k + key0 + min(k0 + nt * 8 + gr, N - 1) * pitch + c2;
#pragma unroll
      for (int ks = 0; ks < D / 16; ++ks) {
        const unsigned b0 = ld2(kp + ks * 16), b1 = ld2(kp + ks * 16 + 8);
        fr_mma(s[0][nt], qa[0][ks], b0, b1);
        fr_mma(s[1][nt], qa[1][ks], b0, b1);
      }
    }
    unsigned pk[2][4];
#pragma unroll
    for (int r = 0; r < 4; ++r) {                // query row 16 (r / 2) + 8 (r % 2) + lane / 4
      float x[4], top = -INFINITY;
#pragma unroll
      for (int nt = 0; nt < 2; ++nt) {
        const int key = k0 + nt * 8 + c2;
        float2 v = make_float2(s[r >> 1][nt][(r & 1) * 2], s[r >> 1][nt][(r & 1) * 2 + 1]);
        if (HAS_BIAS && key < N)                 // (a plane's rows are padded to eight keys)
          v = fr_bias_add(v, ld2(bias + (long long)min(q0 + (r >> 1) * 16 + (r & 1) * 8 + gr, N - 1) * inf.ld + key));
        x[2 * nt] = key < N ? v.x * p.sc2 : -INFINITY;
        x[2 * nt + 1] = key + 1 < N ? v.y * p.sc2 : -INFINITY;
        top = fmaxf(top, fmaxf(x[2 * nt], x[2 * nt + 1]));
      }
      top = fmaxf(top, __shfl_xor_sync(0xffffffffu, top, 1));
      top = fmaxf(top, __shfl_xor_sync(0xffffffffu, top, 2));
      top = fmaxf(top, mx[r]);
      const float ref = top == -INFINITY ? 0.f : top, scale = fr_exp2(mx[r] - ref);
      mx[r] = top;
      l[r] *= scale;
#pragma unroll
      for (int k = 0; k < D / 8; ++k) {
        o[r >> 1][k][(r & 1) * 2] *= scale;
        o[r >> 1][k][(r & 1) * 2 + 1] *= scale;
      }
#pragma unroll
      for (int nt = 0; nt < 2; ++nt) {
        const float w0 = fr_exp2(x[2 * nt] - ref), w1 = fr_exp2(x[2 * nt + 1] - ref);
        l[r] += w0 + w1;
        pk[r >> 1][(r & 1) + 2 * nt] = fr_pack(w0, w1);
      }
    }
    const unsigned short* vp = reinterpret_cast<const unsigned short*>(p.v) + key0 + gr;
#pragma unroll
    for (int k = 0; k < D / 8; ++k) {
      unsigned b[2];
#pragma unroll
      for (int nt = 0; nt < 2; ++nt) {
        const int key = k0 + nt * 8 + c2;
        const unsigned lo = key < N ? vp[key * pitch + k * 8] : 0u, hi = key + 1 < N ? vp[(key + 1) * pitch + k * 8] : 0u;
        b[nt] = lo | hi << 16;
      }
      fr_mma(o[0][k], pk[0], b[0], b[1]);
      fr_mma(o[1][k], pk[1], b[0], b[1]);
    }
  }
  float lse[4];
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    l[r] += __shfl_xor_sync(0xffffffffu, l[r], 1);
    l[r] += __shfl_xor_sync(0xffffffffu, l[r], 2);
    const float inv = 1.0f / l[r];
    const int q = q0 + (r >> 1) * 16 + (r & 1) * 8 + gr;
    lse[r] = mx[r] + log2f(l[r]);
    if (q < N && NT_IN(inf.orow + (long long)t * inf.tile_row + (long long)(q - inf.q0) * inf.step, p.rows, NT_SITE_FRAG_ATTN_OUT)) {
#pragma unroll
      for (int k = 0; k < D / 8; ++k)
        *reinterpret_cast<unsigned*>(p.o + key0 + q * pitch + k * 8 + c2) =
            fr_pack(o[r >> 1][k][(r & 1) * 2] * inv, o[r >> 1][k][(r & 1) * 2 + 1] * inv);
    }
  }
  return make_float4(lse[0], lse[1], lse[2], lse[3]);
}

// 4 x 4 transpose inside a quad: lane q ends with word q of lanes 0 .. 3
__device__ inline uint4 fr_quad_transpose(unsigned w0, unsigned w1, unsigned w2, unsigned w3, int lane) {
  const bool h1 = lane & 1, h2 = lane & 2;
  const unsigned x0 = __shfl_xor_sync(0xffffffffu, h1 ? w0 : w1, 1), x1 = __shfl_xor_sync(0xffffffffu, h1 ? w2 : w3, 1);
  const unsigned a0 = h1 ? x0 : w0, a1 = h1 ? w1 : x0;      // words (lane & 1) of the pair's even and odd lane
  const unsigned b0 = h1 ? x1 : w2, b1 = h1 ? w3 : x1;      // words 2 + (lane & 1)
  const unsigned y0 = __shfl_xor_sync(0xffffffffu, h2 ? a0 : b0, 2), y1 = __shfl_xor_sync(0xffffffffu, h2 ? a1 : b1, 2);
  return h2 ? make_uint4(y0, y1, b0, b1) : make_uint4(a0, a1, y0, y1);
}

template <int D, bool HAS_BIAS, int NT>
__global__ void __launch_bounds__(128 + 128 * NT, 1) attn_fr_kernel(const __grid_constant__ AttnFrParams p) {
  constexpr int SPAN = 2 * D;                        // bytes per Q / K / V tile row = swizzle span
  constexpr int Q_BYTES = 128 * SPAN, KV_BYTES = FR_KEYS * SPAN;
  constexpr int BIAS_BYTES = HAS_BIAS ? FR_BIAS_BYTES : 0;
  constexpr int STAGE_BYTES = BIAS_BYTES + NT * 2 * KV_BYTES;
  extern __shared__ unsigned char smem_raw[];
  __shared__ __align__(8) unsigned long long bars[4 + 2 * FR_MAXSTAGE + 4 * NT];
  __shared__ unsigned tmem_base_s;
  __shared__ int abort_flag;
  // (at least as long as the ring of stages: an entry is written again only after its item's last stage has come back)
  __shared__ __align__(16) FrInfo info[FR_MAXSTAGE];
  unsigned char* smem = smem_raw + ((1024 - (smem_u32(smem_raw) & 1023)) & 1023);
  unsigned char* sQ = smem;                          // [2][NT tiles]
  unsigned char* sStage = sQ + 2 * NT * Q_BYTES;     // [nstage][bias | K0 V0 | K1 V1 | ...]
  unsigned long long* qfull = bars;                  // [2]
  unsigned long long* qempty = bars + 2;             // [2] count NT: every tile's last score MMAs of the item are done
  unsigned long long* full = bars + 4;               // [nstage]
  unsigned long long* empty = full + FR_MAXSTAGE;    // [nstage] count 4 NT: every softmax warp is done with the stage
  unsigned long long* sfull = empty + FR_MAXSTAGE;   // [NT][2] scores are in the buffer
  unsigned long long* sempty = sfull + 2 * NT;       // [NT][2] count 4: the scores have been read

  // (the shuffles here and below tell the compiler that a value is the same in the whole warp: addresses and branches
  // that hang on it then cost uniform instructions only)
  const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    abort_flag = 0;
    for (int b = 0; b < 2; ++b) {
      mbar_init(&qfull[b], 1);
      mbar_init(&qempty[b], NT);
    }
    for (int s = 0; s < FR_MAXSTAGE; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 4 * NT);
    }
    for (int b = 0; b < 2 * NT; ++b) {
      mbar_init(&sfull[b], 1);
      mbar_init(&sempty[b], 4);
    }
    mbar_fence_init();
  }
  if (warp == 1) tmem_alloc(&tmem_base_s, 512);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  pdl_begin();
  const unsigned tmem_base = __shfl_sync(0xffffffffu, tmem_base_s, 0);
  AbortCtx ab{p.status, &abort_flag};
  const unsigned nstage = (unsigned)p.nstage;

  const long long total_cost = p.cost_off[p.m.B];
  const long long g0 = fr_ordinal_at(p, total_cost * blockIdx.x / gridDim.x);
  const long long g1 = fr_ordinal_at(p, total_cost * (blockIdx.x + 1) / gridDim.x);
  const int count = (int)(g1 - g0);
  unsigned st = 0, ph = 0;         // ring slot and its phase

  // registers: 56 for the four auxiliary warps, the rest of the launch's share for the softmax warps
  if (warp < 4) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 56;\n");
    if (warp == 0) {
      // ---------------------------------------------------------------- producer: lanes 0 .. 2 NT - 1 copy Q, K, V; lane 31 the bias
      const bool colmode = p.mode == FR_MODE_PAIR_COL;
      const int t = lane >> 1, part = lane & 1;      // Q: tile and 64-query half; keys: tile and K / V
      FrItem<NT> it;
      if (count > 0) it.seek(p, g0);
      int blocks = 0;
      bool ok = true;
      for (int n = 0; n < count && ok; ++n, it.next(p)) {
        const unsigned qb = n & 1, qph = (n >> 1) & 1;
        const int tiles = it.tiles(p);
        if (lane == 0) {
          ok = fr_wait_idle(&qempty[qb], qph ^ 1, ab);
          mbar_expect_tx(&qfull[qb], tiles * Q_BYTES);
        }
        ok = __shfl_sync(0xffffffffu, ok, 0);
        if (!ok) break;
        const bool mine = t < tiles;
        const int x = it.head(p, t) * D, row = it.kvrow(p, t), col = it.g * NT + t;
        const CUtensorMap* cmap = &p.cmap[it.s];
        const CUtensorMap* map = part ? &p.vmap : &p.kmap;
        if (mine) {
          unsigned char* dst = sQ + (qb * NT + t) * Q_BYTES + part * KV_BYTES;
          const int q0 = it.jb * 128 + part * 64;
          if (colmode) tma_load_4d(dst, cmap, &qfull[qb], x, q0, col, 0);
          else tma_load_2d(dst, &p.qmap, &qfull[qb], x, row + q0);
        }
        for (int k0 = 0; k0 < it.N; k0 += FR_KEYS) {
          unsigned char* stg = sStage + st * STAGE_BYTES;
          if (lane == 0) {
            ok = blocks++ != p.drop && fr_wait_idle(&empty[st], ph ^ 1, ab);
            if (ok && k0 == 0) {    // (after a wait that ran out nothing is written: the softmax warps may still be at an older item)
              FrInfo& f = info[n % FR_MAXSTAGE];
              f.N = it.N;
              f.q0 = it.jb * 128;
              f.tiles = tiles;
              f.step = colmode ? it.N : 1;
              f.orow = colmode ? (int)(p.m.pair_off[it.s] - p.row0) + it.jb * 128 * it.N + it.g * NT : it.kvrow(p, 0) + it.jb * 128;
              f.head = it.head(p, 0);
              f.tile_row = p.mode == FR_MODE_TOKEN ? 0 : colmode ? 1 : it.N;
              f.tile_head = p.mode == FR_MODE_TOKEN ? 1 : 0;
              f.ld = round_up8(it.N);
              f.bias_plane = (long long)p.H * p.m.cm_off[it.s] + (long long)f.head * it.N * f.ld;
            }
            if (ok) mbar_expect_tx(&full[st], BIAS_BYTES + tiles * 2 * KV_BYTES);
          }
          ok = __shfl_sync(0xffffffffu, ok, 0);
          if (!ok) break;
          if (mine) {
            unsigned char* dst = stg + BIAS_BYTES + (t * 2 + part) * KV_BYTES;
            if (colmode) tma_load_4d(dst, cmap, &full[st], x, k0, col, 1 + part);
            else tma_load_2d(dst, map, &full[st], x, row + k0);
          }
          if (HAS_BIAS && lane == 31) tma_load_3d(stg, &p.bmap[it.s], &full[st], k0, it.jb * 128, it.head(p, 0));
          if (++st == nstage) { st = 0; ph ^= 1; }
        }
      }
    } else if (warp <= NT) {
      // ---------------------------------------------------------------- score MMAs: one issuing warp per tile, so that
      // no tile waits for another one's buffers (whole warp, one elected lane issues)
      const int t = warp - 1;
      const unsigned q_base = smem_u32(sQ) + t * Q_BYTES, k_base = smem_u32(sStage) + BIAS_BYTES + t * 2 * KV_BYTES;
      const unsigned d_base = tmem_base + t * 2 * FR_KEYS;
      const unsigned idesc = idesc_f16(128, FR_KEYS, 0, 0, FMT_BF16, FMT_BF16);
      unsigned cnt = 0;
      FrItem<NT> it;
      if (count > 0) it.seek(p, g0);
      bool ok = true;                                // false once a wait has run out
      for (int n = 0; n < count; ++n, it.next(p)) {
        const unsigned qb = n & 1, qph = (n >> 1) & 1;
        const bool valid = t < it.tiles(p);
        ok = fr_wait_idle(&qfull[qb], qph, ab);
        const unsigned long long qd = fr_desc(q_base + qb * NT * Q_BYTES, SPAN);
        for (int k0 = 0; k0 < it.N; k0 += FR_KEYS) {
          // every block, also of an item in which this tile has no row: a parity wait tells one phase from the next only,
          // and a warp that left blocks out could take a slot's load of one ring turn ago, still in flight, for its own
          ok &= fr_wait_idle(&full[st], ph, ab);
          if (valid) {
            const unsigned b = cnt & 1, bph = (cnt >> 1) & 1;
            ok &= fr_wait_idle(&sempty[t * 2 + b], bph ^ 1, ab);
            tc_fence_after();
            const unsigned long long kd = fr_desc(k_base + st * STAGE_BYTES, SPAN);
            if (!__all_sync(0xffffffffu, ok)) break;
            if (elect_one()) {
#pragma unroll
              for (int ks = 0; ks < D / 16; ++ks) umma_bf16(d_base + b * FR_KEYS, qd + ks * 2, kd + ks * 2, idesc, ks ? 1u : 0u);
              tc_commit(&sfull[t * 2 + b]);
            }
            __syncwarp();
            ++cnt;
          }
          if (++st == nstage) { st = 0; ph ^= 1; }
        }
        if (!__all_sync(0xffffffffu, ok)) break;
        if (valid) {
          if (elect_one()) tc_commit(&qempty[qb]);
        } else if (lane == 0) {
          mbar_arrive(&qempty[qb]);
        }
        __syncwarp();
      }
    }
  } else {
    // ------------------------------------------------------------------ softmax and P V
    if (NT == 3) asm volatile("setmaxnreg.inc.sync.aligned.u32 152;\n");      // 4 x 128 = 56 + 3 x 152
    else asm volatile("setmaxnreg.inc.sync.aligned.u32 224;\n");              // 3 x 168 = 56 + 2 x 224
    const int t = (warp - 4) >> 2, quarter = warp & 3;
    const unsigned s_base = tmem_base + ((unsigned)(quarter * 32) << 16) + t * 2 * FR_KEYS;
    const float sc2 = p.sc2;
    // this lane's ldmatrix addresses inside a stage (the stage base is 1024-byte aligned)
    const unsigned bias_off = (unsigned)((quarter * 32 + (lane & 15)) * 128 + (((lane >> 4) ^ (lane & 7)) << 4));
    const unsigned v_off = BIAS_BYTES + (t * 2 + 1) * KV_BYTES + (lane & 15) * SPAN +
                           ((unsigned)((lane >> 4) ^ ((((lane & 15) * SPAN) >> 7) & (SPAN / 16 - 1))) << 4);
    const unsigned stage_base = smem_u32(sStage), empty_bar = smem_u32(empty), sempty_bar = smem_u32(sempty + 2 * t);
    unsigned long long* sfull_t = sfull + 2 * t;
    float nref[4] = {0.f, 0.f, 0.f, 0.f};            // minus the references of the lane's query rows
    bool have_ref = false;
    unsigned cnt = 0;                                // blocks of this tile so far
#pragma unroll 1
    for (int n = 0; n < count; ++n) {
      if (!__all_sync(0xffffffffu, mbar_wait(&full[st], ph, ab))) break;   // the item's first stage: its description is there too
      const FrInfo& inf = info[n % FR_MAXSTAGE];
      const int N = __shfl_sync(0xffffffffu, inf.N, 0), q0 = __shfl_sync(0xffffffffu, inf.q0, 0) + quarter * 32;
      const bool valid = t < __shfl_sync(0xffffffffu, inf.tiles, 0);
      if (!valid || q0 >= N) {    // no row, or no query in this warp's quarter: follow the barriers only
        for (int k0 = 0; k0 < N; k0 += FR_KEYS) {
          if (!__all_sync(0xffffffffu, mbar_wait(&full[st], ph, ab))) goto gone;
          if (valid) {
            if (!__all_sync(0xffffffffu, mbar_wait(&sfull_t[cnt & 1], (cnt >> 1) & 1, ab))) goto gone;
            fr_arrive(sempty_bar + (cnt & 1) * 8, lane);
            ++cnt;
          }
          __syncwarp();
          fr_arrive(empty_bar + st * 8, lane);
          if (++st == nstage) { st = 0; ph ^= 1; }
        }
        continue;
      }
      float o[2][D / 8][4];
      float2 l[4];
      // Chunks of 32 keys in pairs: the even ones in sa / pa, the odd ones in sb / pb (a block boundary lies between an
      // odd and an even chunk).  The previous chunk's product is issued beside each chunk's exponentials, so a stage is
      // let go of one chunk after its last; the row's first chunk has zero weights before it.
      unsigned sa[2][16], sb[2][16], pa[2][2][4], pb[2][2][4];
#pragma unroll
      for (int mt = 0; mt < 2; ++mt)
#pragma unroll
        for (int k = 0; k < D / 8; ++k)
#pragma unroll
          for (int e = 0; e < 4; ++e) o[mt][k][e] = 0.f;
#pragma unroll
      for (int r = 0; r < 4; ++r) l[r] = make_float2(0.f, 0.f);
#pragma unroll
      for (int k = 0; k < 16; ++k) pb[k >> 3][(k >> 2) & 1][k & 3] = 0u;
      unsigned stage = stage_base + st * STAGE_BYTES, v_prev = stage + v_off, s_addr = s_base + (cnt & 1) * FR_KEYS;
      int left = N;                                  // keys left in the row
      unsigned held = 0;                             // empty barrier of the stage whose last product is pending
      if (!__all_sync(0xffffffffu, mbar_wait(&sfull_t[cnt & 1], (cnt >> 1) & 1, ab))) break;
      tc_fence_after();
      fr_request_scores(s_addr, sa);
      tmem_ld_wait2(sa[0], sa[1]);
      if (!have_ref) {
        unsigned m[2][16];
#pragma unroll
        for (int e = 0; e < 16; ++e) { m[0][e] = sa[0][e]; m[1][e] = sa[1][e]; }
        if (left < 32) fr_mask(m, left, lane);
        fr_first_reference<HAS_BIAS>(m, stage + bias_off, sc2, nref);
        have_ref = true;
      }
#pragma unroll 1
      while (true) {
        // (at the end of the row the scores requested are nobody's, but readable)
        const bool more = left > FR_KEYS;
        const unsigned wrap = st + 1 == nstage, nst = wrap ? 0u : st + 1, nph = ph ^ wrap, ncnt = cnt + 1;
        fr_request_scores(s_addr + 32, sb);
        if (left < 32) fr_mask(sa, left, lane);
        fr_weights<D, HAS_BIAS>(sa, stage + bias_off, 0, sc2, nref, l, pa, o, pb, v_prev);
        // the next block's barriers are looked at a chunk ahead, so that their latency is not waited for
        const bool ready = more ? fr_ready(&full[nst], nph) & fr_ready(&sfull_t[ncnt & 1], (ncnt >> 1) & 1) : true;
        tmem_ld_wait2(sb[0], sb[1]);
        if (held) fr_arrive(held, lane);             // the last product of the previous block is issued
        if (left <= 32) break;
        const unsigned bias_odd = stage + bias_off, v_odd = stage + v_off, buf = sempty_bar + (cnt & 1) * 8;
        if (more) {
          if (!__all_sync(0xffffffffu, ready)) {
            const bool there = mbar_wait(&full[nst], nph, ab) & mbar_wait(&sfull_t[ncnt & 1], (ncnt >> 1) & 1, ab);
            if (!__all_sync(0xffffffffu, there)) goto gone;
          }
          tc_fence_after();
          held = empty_bar + st * 8;
          st = nst;
          ph = nph;
          cnt = ncnt;
          stage = stage_base + st * STAGE_BYTES;
          s_addr = s_base + (cnt & 1) * FR_KEYS;
        }
        fr_request_scores(s_addr, sa);
        if (left < 64) fr_mask(sb, left - 32, lane);
        fr_weights<D, HAS_BIAS>(sb, bias_odd, 1, sc2, nref, l, pb, o, pa, v_odd);
        tmem_ld_wait2(sa[0], sa[1]);
        v_prev = v_odd + 32 * SPAN;
        if (!more) break;
        tc_fence_before();                           // the block's scores have all been read
        fr_arrive(buf, lane);
        left -= FR_KEYS;
      }
      if (left <= 32) fr_pv<D>(o, pa, stage + v_off);      // the last chunk's product
      else fr_pv<D>(o, pb, v_prev);
      tc_fence_before();
      __syncwarp();
      // ---- the row is finished: sums over the quads, the next row's references
      float inv[4];
      bool off = false;
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        float x = l[r].x + l[r].y;
        x += __shfl_xor_sync(0xffffffffu, x, 1);
        x += __shfl_xor_sync(0xffffffffu, x, 2);
        asm("rcp.approx.ftz.f32 %0, %1;\n" : "=f"(inv[r]) : "f"(x));
        const int q = q0 + (r >> 1) * 16 + (r & 1) * 8 + (lane >> 2);
        // (a sum that is not a number comes from a score that is none, and nothing would change that: the row stays as it is)
        const bool bad = x <= FR_LOW || x >= FR_HIGH;
        off |= bad & (q < N);
        nref[r] -= bad || x != x ? 0.f : (float)((int)(__float_as_uint(x) >> 23) - 127) + FR_MARGIN;
      }
      const bool again = __any_sync(0xffffffffu, off);
      if (again) {
        const float4 e = fr_exact_row<D, HAS_BIAS>(p, inf, t, quarter, lane);
        const float lse[4] = {e.x, e.y, e.z, e.w};
        __syncwarp();
#pragma unroll
        for (int r = 0; r < 4; ++r) nref[r] = fabsf(lse[r]) < 1e30f ? -(lse[r] + FR_MARGIN) : nref[r];
      } else {
        // O / l.  Quads transpose four words so that a lane stores 16 bytes (a quarter of the store instructions and of
        // the lines they touch)
        const int4 out = *reinterpret_cast<const int4*>(&inf.orow);
        const int Hd = p.H * D, step = inf.step;
        const int orow0 = out.x + t * out.z + quarter * 32 * step;
        __nv_bfloat16* op = p.o + p.row0 * Hd + (out.y + t * out.w) * D;
        unsigned w[4][D / 8];
#pragma unroll
        for (int r = 0; r < 4; ++r)
#pragma unroll
          for (int k = 0; k < D / 8; ++k) w[r][k] = fr_pack(o[r >> 1][k][(r & 1) * 2] * inv[r], o[r >> 1][k][(r & 1) * 2 + 1] * inv[r]);
        constexpr int RPT = D == 16 ? 2 : 1;         // rows per transpose (at d = 16 a row has two words only)
#pragma unroll
        for (int r = 0; r < 4; r += RPT) {
#pragma unroll
          for (int k = 0; k < D / 8; k += 4) {
            const uint4 v = D == 16 ? fr_quad_transpose(w[r][0], w[r][1], w[r + RPT - 1][0], w[r + RPT - 1][1], lane)
                                    : fr_quad_transpose(w[r][k], w[r][(k + 1) % (D / 8)], w[r][(k + 2) % (D / 8)], w[r][(k + 3) % (D / 8)], lane);
            const int rr = D == 16 ? r + ((lane >> 1) & 1) : r;
            const int q = (rr >> 1) * 16 + (rr & 1) * 8 + (lane >> 2);
            const int ch = D == 16 ? (lane & 1) * 8 : (k + (lane & 3)) * 8;
            const long long orow = orow0 + (long long)q * step;
            if (q0 + q < N && NT_IN(orow, p.rows, NT_SITE_FRAG_ATTN_OUT)) *reinterpret_cast<uint4*>(op + orow * Hd + ch) = v;
          }
        }
      }
      // the item's last stage goes back only now: its description is in use until here
      __syncwarp();
      fr_arrive(sempty_bar + (cnt & 1) * 8, lane);
      fr_arrive(empty_bar + st * 8, lane);
      ++cnt;
      if (++st == nstage) { st = 0; ph ^= 1; }
    }
  }
gone:
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  abort_linger(ab);
  if (warp == 1) tmem_dealloc(tmem_base, 512);
}

// ---------------------------------------------------------------------------------- host
constexpr int fr_tiles(int d) { return d == 64 ? 2 : 3; }

static size_t fr_smem_bytes(int d, bool has_bias, int nstage) {
  const size_t span = 2 * d, nt = fr_tiles(d);
  return 2 * nt * 128 * span + (size_t)nstage * ((has_bias ? FR_BIAS_BYTES : 0) + nt * 2 * FR_KEYS * span) + 1024;
}
static const size_t FR_SMEM_LIMIT = 232448 - 1024;     // the static part (barriers, item descriptions) is small

static int fr_pick_stages(int d, bool has_bias) {
  int n = FR_MAXSTAGE;
  while (n > 2 && fr_smem_bytes(d, has_bias, n) > FR_SMEM_LIMIT) --n;
  return n;
}

bool fast_attn_fr_supported(int H, int d) { return H >= 1 && (d == 16 || d == 32 || d == 64); }

template <int D, bool HAS_BIAS>
static nt_status launch_attn_fr(AttnFrParams& p, int n_min, cudaStream_t st) {
  constexpr int NT = fr_tiles(D);
  static bool attr_set[64] = {};
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev < 0 || dev >= 64) return NT_ERR_UNSUPPORTED;
  if (!attr_set[dev]) {
    if (cudaFuncSetAttribute(attn_fr_kernel<D, HAS_BIAS, NT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)FR_SMEM_LIMIT) !=
        cudaSuccess)
      return cuda_fail("attention smem attribute");
    attr_set[dev] = true;
  }
  // items and their cost
  p.item_off[0] = p.cost_off[0] = 0;
  for (int s = 0; s < p.m.B; ++s) {
    const long long N = p.m.N[s], njb = N <= n_min ? 0 : (N + 127) / 128;
    const long long items = p.mode == FR_MODE_TOKEN ? njb * (p.single_tile ? p.H : (p.H + NT - 1) / NT) : njb * p.H * ((N + NT - 1) / NT);
    p.item_off[s + 1] = p.item_off[s] + items;
    p.cost_off[s + 1] = p.cost_off[s] + items * ((N + 31) / 32 + FR_ITEM_COST);
  }
  const long long items = p.item_off[p.m.B];
  if (items == 0) return NT_OK;
  const int sms = sm_count();
  const unsigned grid = (unsigned)(items < sms ? items : sms);
  {
    LaunchScope ls(p.mode == FR_MODE_TOKEN ? "attn_core_tok" : p.mode == FR_MODE_PAIR_COL ? "attn_core_col" : "attn_core", st);
    launch_kernel(attn_fr_kernel<D, HAS_BIAS, NT>, grid, 128 + 128 * NT, fr_smem_bytes(D, HAS_BIAS, p.nstage), st, p);
  }
  return cuda_ok("attention launch");
}

nt_status fast_attn_core_fr(const void* q, const void* k, const void* v, const void* bias, void* o, int H, int d,
                            int mode, const BatchMeta& m, int* status, cudaStream_t st, int n_min) {
  if (!fast_attn_fr_supported(H, d)) return NT_ERR_UNSUPPORTED;
  AttnFrParams p;
  memset(&p, 0, sizeof(p));
  p.m = m;
  p.q = (const __nv_bfloat16*)q;
  p.k = (const __nv_bfloat16*)k;
  p.v = (const __nv_bfloat16*)v;
  p.bias = (const __nv_bfloat16*)bias;
  p.o = (__nv_bfloat16*)o;
  p.H = H;
  p.mode = mode;
  p.status = status;
  p.sc2 = FR_LOG2E / sqrtf((float)d);
  p.nstage = fr_pick_stages(d, bias != nullptr);
  p.drop = g_fr_drop;
  const bool token = mode == FR_MODE_TOKEN;
  p.single_tile = token && bias != nullptr;   // every head has bias planes of its own: nothing to share between two rows
  p.row0 = token ? m.tok_off[0] : m.pair_off[0];
  const long long rows = (token ? m.tok_off[m.B] : m.pair_off[m.B]) - p.row0;
  if (rows <= 0) return NT_OK;
  if (rows > 0x7FFFFF00ll) return NT_ERR_UNSUPPORTED;
  p.rows = rows;
  const int Hd = H * d;
  const int promo = 2 * d >= 128 ? 128 : 2 * d;
  if (mode == FR_MODE_PAIR_COL) {
    // q, k, v must be three equally spaced buffers (they are carved that way): the map's outermost dimension picks one
    const long long gap = (const char*)k - (const char*)q;
    if (gap <= 0 || (const char*)v - (const char*)k != gap || gap % 16 != 0) return NT_ERR_UNSUPPORTED;
    for (int s = 0; s < m.B; ++s) {
      const int N = m.N[s];
      if (N < 1 || N <= n_min) continue;
      const unsigned long long dims[4] = {(unsigned long long)Hd, (unsigned long long)N, (unsigned long long)N, 3};
      const unsigned long long strides[3] = {(unsigned long long)N * Hd * 2, (unsigned long long)Hd * 2, (unsigned long long)gap};
      const unsigned box[4] = {(unsigned)d, 64, 1, 1};
      if (!make_tmap_16bit(&p.cmap[s], p.q + m.pair_off[s] * Hd, 4, dims, strides, box, 2 * d, promo))
        return cuda_fail("attention column map");
    }
  } else {
    const unsigned long long dims[2] = {(unsigned long long)Hd, (unsigned long long)rows};
    const unsigned long long strides[1] = {(unsigned long long)Hd * 2};
    const unsigned box[2] = {(unsigned)d, 64};
    if (!make_tmap_16bit(&p.qmap, p.q + p.row0 * Hd, 2, dims, strides, box, 2 * d, promo)) return cuda_fail("attention q map");
    if (!make_tmap_16bit(&p.kmap, p.k + p.row0 * Hd, 2, dims, strides, box, 2 * d, promo)) return cuda_fail("attention k map");
    if (!make_tmap_16bit(&p.vmap, p.v + p.row0 * Hd, 2, dims, strides, box, 2 * d, promo)) return cuda_fail("attention v map");
  }
  if (bias) {
    for (int s = 0; s < m.B; ++s) {
      const int N = m.N[s];
      if (N < 1 || N <= n_min) continue;
      const unsigned long long ld = (unsigned long long)round_up8(N);
      const unsigned long long dims[3] = {(unsigned long long)N, (unsigned long long)N, (unsigned long long)H};
      const unsigned long long strides[2] = {ld * 2, (unsigned long long)N * ld * 2};
      const unsigned box[3] = {64, 128, 1};
      if (!make_tmap_16bit(&p.bmap[s], p.bias + (long long)H * m.cm_off[s], 3, dims, strides, box, 128, 128))
        return cuda_fail("attention bias map");
    }
    if (d == 16) return launch_attn_fr<16, true>(p, n_min, st);
    if (d == 32) return launch_attn_fr<32, true>(p, n_min, st);
    return launch_attn_fr<64, true>(p, n_min, st);
  }
  if (d == 16) return launch_attn_fr<16, false>(p, n_min, st);
  if (d == 32) return launch_attn_fr<32, false>(p, n_min, st);
  return launch_attn_fr<64, false>(p, n_min, st);
}

}  // namespace ntp
