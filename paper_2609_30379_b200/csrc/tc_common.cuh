// sm_100a building blocks for the tensor-core kernels: mbarrier with bounded waits, TMA tiled
// loads / stores, tcgen05 MMA with shared-memory operand descriptors, TMEM allocation and loads.
// Every wait is bounded (a probe count and about a second of SM clocks); on expiry the kernel records NT_ERR_TIMEOUT in the status
// word, raises a CTA-wide abort flag (later waits give up after a short spin) and still runs to
// its normal end, so TMEM is released and the context stays usable.
#pragma once

#include <cuda.h>

#include "common.cuh"

namespace ntp {

// ---------------------------------------------------------------------------------- host: TMA maps
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
EncodeTiledFn get_encode_tiled();

// bf16 tensor map with 128-byte swizzle; dims / strides fastest first (strides in bytes for dims 1..rank-1)
bool make_tmap_bf16(CUtensorMap* map, const void* base, int rank, const unsigned long long* dims,
                    const unsigned long long* strides_bytes, const unsigned* box);
// same with a 32-, 64- or 128-byte swizzle span (the inner box extent in bytes must not exceed it); 0 = no swizzle.
// l2_promotion_bytes: granularity at which L2 fetches around a request (128, 64 or 0 = none); boxes narrower than a
// 128-byte line that other CTAs read at other times should not promote, or DRAM delivers their neighbours in vain.
bool make_tmap_16bit(CUtensorMap* map, const void* base, int rank, const unsigned long long* dims,
                     const unsigned long long* strides_bytes, const unsigned* box, int swizzle_bytes,
                     int l2_promotion_bytes = 128);

#ifdef __CUDACC__
// ---------------------------------------------------------------------------------- device helpers
constexpr unsigned WAIT_PROBES = 1u << 22;            // probes before a wait gives up, whatever the clock says
constexpr long long WAIT_CLOCKS = 1ll << 31;          // SM clocks before a wait gives up (about a second)
constexpr long long WAIT_CLOCKS_ABORTED = 1ll << 14;  // once the CTA has given up, later waits return quickly

struct AbortCtx {
  int* status;            // global status word (nullable)
  volatile int* flag;     // CTA-shared abort flag
};

// A CTA that gave up on a wait may still have bulk copies in flight into its shared memory (loads it had requested
// before the wait expired); they land within a few microseconds.  Before such a CTA returns, and its shared memory
// goes to the next one, it sits out a bounded interval far longer than that (about 70 microseconds).  On the normal
// path every copy has been consumed through its barrier and this is one shared-memory read.
__device__ inline void abort_linger(const AbortCtx& ab) {
  if (*ab.flag) {
    const long long t0 = clock64();
    while (clock64() - t0 < (1ll << 17)) {
    }
  }
}

__device__ inline unsigned smem_u32(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }

__device__ inline void mbar_init(void* bar, unsigned count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(smem_u32(bar)), "r"(count));
}
__device__ inline void mbar_fence_init() { asm volatile("fence.mbarrier_init.release.cluster;\n" ::); }
__device__ inline void mbar_expect_tx(void* bar, unsigned bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}
__device__ inline void mbar_arrive(void* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(smem_u32(bar)) : "memory");
}
__device__ inline bool mbar_try(void* bar, unsigned parity) {
  unsigned ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.b32 %0, 1, 0, p;\n\t}\n"
      : "=r"(ok) : "r"(smem_u32(bar)), "r"(parity) : "memory");
  return ok != 0;
}
// Bounded wait; returns false (after flagging) if the limit was reached.  A failing probe parks the warp in
// hardware for a few microseconds at most and returns at once when the phase completes, so the loop needs no
// sleep of its own; the abort flag and the clock are looked at every 16th probe.
__device__ inline bool mbar_wait(void* bar, unsigned parity, const AbortCtx& ab, long long limit_clocks = WAIT_CLOCKS) {
  if (mbar_try(bar, parity)) return true;
  const long long t0 = clock64();
  const long long limit = *ab.flag ? WAIT_CLOCKS_ABORTED : limit_clocks;
  for (unsigned it = 0; it < WAIT_PROBES; ++it) {
    if (mbar_try(bar, parity)) return true;
    if ((it & 15u) == 15u && (clock64() - t0 > limit || *ab.flag)) break;
  }
  if (!*ab.flag) {
    *ab.flag = 1;
    if (ab.status) atomicCAS(ab.status, 0, (int)NT_ERR_TIMEOUT);
  }
  return false;
}

__device__ inline void fence_proxy_async_smem() { asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory"); }

__device__ inline void tma_load_2d(void* dst, const CUtensorMap* map, void* bar, int c0, int c1) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];\n"
      ::"r"(smem_u32(dst)), "l"(map), "r"(smem_u32(bar)), "r"(c0), "r"(c1) : "memory");
}
__device__ inline void tma_load_3d(void* dst, const CUtensorMap* map, void* bar, int c0, int c1, int c2) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5}], [%2];\n"
      ::"r"(smem_u32(dst)), "l"(map), "r"(smem_u32(bar)), "r"(c0), "r"(c1), "r"(c2) : "memory");
}
__device__ inline void tma_load_4d(void* dst, const CUtensorMap* map, void* bar, int c0, int c1, int c2, int c3) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5, %6}], [%2];\n"
      ::"r"(smem_u32(dst)), "l"(map), "r"(smem_u32(bar)), "r"(c0), "r"(c1), "r"(c2), "r"(c3) : "memory");
}
__device__ inline void tma_store_2d(const CUtensorMap* map, const void* src, int c0, int c1) {
  asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%2, %3}], [%1];\n"
               ::"l"(map), "r"(smem_u32(src)), "r"(c0), "r"(c1) : "memory");
}
__device__ inline void tma_store_4d(const CUtensorMap* map, const void* src, int c0, int c1, int c2, int c3) {
  asm volatile("cp.async.bulk.tensor.4d.global.shared::cta.bulk_group [%0, {%2, %3, %4, %5}], [%1];\n"
               ::"l"(map), "r"(smem_u32(src)), "r"(c0), "r"(c1), "r"(c2), "r"(c3) : "memory");
}
__device__ inline void tma_store_commit() { asm volatile("cp.async.bulk.commit_group;\n" ::: "memory"); }
__device__ inline void tma_store_wait_read0() { asm volatile("cp.async.bulk.wait_group.read 0;\n" ::: "memory"); }
__device__ inline void tma_store_wait_all0() { asm volatile("cp.async.bulk.wait_group 0;\n" ::: "memory"); }

// ---- TMEM
__device__ inline void tmem_alloc(unsigned* dst_smem, unsigned ncols) {   // whole warp
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(smem_u32(dst_smem)), "r"(ncols)
               : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
}
__device__ inline void tmem_dealloc(unsigned taddr, unsigned ncols) {     // whole warp
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(taddr), "r"(ncols) : "memory");
}
__device__ inline void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory"); }
__device__ inline void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory"); }
__device__ inline void tc_commit(void* bar) {   // arrives on the mbarrier when all prior MMAs of this thread finish
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(smem_u32(bar))
               : "memory");
}
__device__ inline void tmem_ld_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory"); }

// 32 lanes x 32 consecutive columns of 32-bit: thread t gets row (lane base + t), columns c..c+31
__device__ inline void tmem_ld32(unsigned taddr, unsigned (&r)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
      "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,"
      "%29,%30,%31}, [%32];\n"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
        "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
        "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr) : "memory");
}

// 32 lanes x 16 consecutive columns
__device__ inline void tmem_ld16(unsigned taddr, unsigned (&r)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];\n"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr) : "memory");
}

// 32 lanes x 8 / 2 consecutive columns
// registers -> TMEM: thread t writes row (lane base + t), 16 or 8 consecutive columns
__device__ inline void tmem_st8(unsigned taddr, const unsigned (&r)[8]) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};\n"
               ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]) : "memory");
}
__device__ inline void tmem_st_wait() { asm volatile("tcgen05.wait::st.sync.aligned;\n" ::: "memory"); }
// D[tmem] (+)= A[tmem] * B[smem]: the A tile (128 rows x 16 elements, two 16-bit elements per column) is read from TMEM
__device__ inline void umma_ts(unsigned d_tmem, unsigned a_tmem, unsigned long long bdesc, unsigned idesc,
                               unsigned accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}\n"
      ::"r"(d_tmem), "r"(a_tmem), "l"(bdesc), "r"(idesc), "r"(accumulate) : "memory");
}
// Waits for the TMEM loads in flight and then passes their destination registers through an empty statement, so that
// no use of them can be scheduled ahead of the wait.  Two statements on purpose: the copies the compiler may make of
// tied operands stand in front of the statement that ties them, and in front of the wait the loads have not landed.
#define NT_TIE16(a)                                                                                                    \
  asm volatile("" : "+r"(a[0]), "+r"(a[1]), "+r"(a[2]), "+r"(a[3]), "+r"(a[4]), "+r"(a[5]), "+r"(a[6]), "+r"(a[7]),   \
                    "+r"(a[8]), "+r"(a[9]), "+r"(a[10]), "+r"(a[11]), "+r"(a[12]), "+r"(a[13]), "+r"(a[14]), "+r"(a[15])::"memory")
__device__ inline void tmem_ld_wait16(unsigned (&a)[16]) {
  tmem_ld_wait();
  NT_TIE16(a);
}
__device__ inline void tmem_ld_wait2(unsigned (&a)[16], unsigned (&b)[16]) {
  tmem_ld_wait();
  NT_TIE16(a);
  NT_TIE16(b);
}

// ---- MMA descriptors (bf16 operands, float accumulate)
// K-major operand tile in the 128-byte-swizzled layout TMA writes for a {64 elements, rows} box:
// row r at r * 128 bytes, 16-byte chunks XOR-swizzled by (r & 7); groups of 8 rows are 1024 bytes
// apart (stride byte offset).  The tile base must be 1024-byte aligned; advancing K by 16 elements
// adds 32 bytes to the start address.
__device__ inline unsigned long long desc_kmajor_sw128(unsigned saddr) {
  unsigned long long d = 0;
  d |= (unsigned long long)((saddr & 0x3FFFFu) >> 4);            // start address, bits [0,14)
  d |= (unsigned long long)1 << 16;                              // leading byte offset (unused with swizzle)
  d |= (unsigned long long)(1024 >> 4) << 32;                    // stride byte offset, bits [32,46)
  d |= (unsigned long long)1 << 46;                              // descriptor version (Blackwell)
  d |= (unsigned long long)2 << 61;                              // SWIZZLE_128B
  return d;
}
// MN-major operand: 64 MN-elements (128 bytes) contiguous per K row, 8 K rows form a 1024-byte
// swizzle atom; the next 64 MN-elements live `lbo` bytes further, the next 8 K rows `sbo` bytes further.
__device__ inline unsigned long long desc_mnmajor_sw128(unsigned saddr, unsigned lbo, unsigned sbo) {
  unsigned long long d = 0;
  d |= (unsigned long long)((saddr & 0x3FFFFu) >> 4);
  d |= (unsigned long long)((lbo >> 4) & 0x3FFF) << 16;
  d |= (unsigned long long)((sbo >> 4) & 0x3FFF) << 32;
  d |= (unsigned long long)1 << 46;
  d |= (unsigned long long)2 << 61;
  return d;
}
// K-major operand without swizzle ("interleaved" core matrices): a core matrix is 8 rows x 16 bytes stored
// contiguously (128 bytes); the next 8 rows are `sbo` bytes further, the next 8 K-elements `lbo` bytes further.
__device__ inline unsigned long long desc_kmajor_nosw(unsigned saddr, unsigned lbo, unsigned sbo) {
  unsigned long long d = 0;
  d |= (unsigned long long)((saddr & 0x3FFFFu) >> 4);
  d |= (unsigned long long)((lbo >> 4) & 0x3FFF) << 16;
  d |= (unsigned long long)((sbo >> 4) & 0x3FFF) << 32;
  d |= (unsigned long long)1 << 46;
  return d;
}
// instruction descriptor of kind::f16: D = f32, M x N tile, operand majors (0 = K-major, 1 = MN-major)
// and the 16-bit format, FMT_F16 or FMT_BF16, the same for both operands
constexpr int FMT_F16 = 0, FMT_BF16 = 1;
__device__ inline unsigned idesc_f16(int M, int N, int a_mn_major, int b_mn_major, int a_fmt, int b_fmt) {
  return (1u << 4) | ((unsigned)a_fmt << 7) | ((unsigned)b_fmt << 10) | ((unsigned)a_mn_major << 15) |
         ((unsigned)b_mn_major << 16) | ((unsigned)(N >> 3) << 17) | ((unsigned)(M >> 4) << 24);
}
// Four K steps of 16 (one 64-column slab of two K-major 128-byte-swizzled operands): D[tmem] (+)= A[smem] * B[smem].  Called by a
// converged warp; one elected lane issues.  One election and one block of code for the four: an issuer that shares
// its scheduler with busy warps pays for every instruction between two MMAs.
__device__ inline void umma_k4(unsigned d_tmem, unsigned long long adesc, unsigned long long bdesc, unsigned idesc, unsigned accumulate) {
  asm volatile(
      "{\n\t.reg .pred p, t, e;\n\t.reg .b64 a, b;\n\t"
      "elect.sync _|e, 0xffffffff;\n\t"
      "setp.ne.b32 p, %4, 0;\n\tsetp.eq.b32 t, 0, 0;\n\t"
      "@e tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t"
      "add.s64 a, %1, 2;\n\tadd.s64 b, %2, 2;\n\t"
      "@e tcgen05.mma.cta_group::1.kind::f16 [%0], a, b, %3, t;\n\t"
      "add.s64 a, %1, 4;\n\tadd.s64 b, %2, 4;\n\t"
      "@e tcgen05.mma.cta_group::1.kind::f16 [%0], a, b, %3, t;\n\t"
      "add.s64 a, %1, 6;\n\tadd.s64 b, %2, 6;\n\t"
      "@e tcgen05.mma.cta_group::1.kind::f16 [%0], a, b, %3, t;\n\t}\n"
      ::"r"(d_tmem), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate) : "memory");
}
// D[tmem] (+)= A[smem] * B[smem]; issued by one thread
__device__ inline void umma_bf16(unsigned d_tmem, unsigned long long adesc, unsigned long long bdesc, unsigned idesc,
                                 unsigned accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n"
      ::"r"(d_tmem), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate) : "memory");
}

// true in exactly one lane of a converged warp.  The MMA issuer runs its loop with the whole warp and puts only
// the tcgen05 instructions under this predicate: descriptors and addresses then stay warp-uniform, which keeps
// the cost of issuing one MMA at a few instructions.
__device__ inline bool elect_one() {
  unsigned pred;
  asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.b32 %0, 1, 0, p;\n\t}\n" : "=r"(pred));
  return pred != 0;
}

__device__ inline void named_bar_sync(int id, int nthreads) {
  asm volatile("bar.sync %0, %1;\n" ::"r"(id), "r"(nthreads) : "memory");
}

// two floats (given as bit patterns) -> packed bf16x2, first in the low half
__device__ inline unsigned pack2(unsigned lo, unsigned hi) {
  __nv_bfloat162 h = __floats2bfloat162_rn(__uint_as_float(lo), __uint_as_float(hi));
  return *reinterpret_cast<unsigned*>(&h);
}

// two floats (bit patterns) scaled and packed as fp16x2 (saturating), first in the low half

// byte offset of 16-byte chunk `chunk` of row `row` inside a 128-byte-swizzled tile
__device__ inline unsigned sw128_off(int row, int chunk) { return row * 128 + ((chunk ^ (row & 7)) << 4); }

// Both MMA operands must have the same 16-bit format.  The folded weights are fp16 (three more
// significant bits than bf16), so the bf16 activation tile is rewritten as fp16 in place before the
// MMA; a bf16 value is exactly representable in fp16 while its magnitude is in [2^-14, 65504], and
// loses only bits below 2^-24 otherwise.  One thread converts one row of a K-major 128-byte-swizzled
// tile made of `nslab` 64-column slabs and returns the row's sum and sum of squares.
__device__ inline void convert_row_bf16_to_f16(unsigned char* tile, int nslab, int slab_bytes, int row, float& sum,
                                               float& sq) {
  float s4[4] = {0.f, 0.f, 0.f, 0.f}, q4[4] = {0.f, 0.f, 0.f, 0.f};   // four independent chains instead of one
  for (int sl = 0; sl < nslab; ++sl) {
    uint4 v[8];
#pragma unroll
    for (int ch = 0; ch < 8; ++ch) v[ch] = *reinterpret_cast<const uint4*>(tile + sl * slab_bytes + sw128_off(row, ch));
#pragma unroll
    for (int ch = 0; ch < 8; ++ch) {
      unsigned w[4] = {v[ch].x, v[ch].y, v[ch].z, v[ch].w};
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const float lo = __uint_as_float(w[e] << 16), hi = __uint_as_float(w[e] & 0xffff0000u);
        s4[e] += lo + hi;
        q4[e] = fmaf(lo, lo, q4[e]);
        q4[e] = fmaf(hi, hi, q4[e]);
        __half2 h = __floats2half2_rn(lo, hi);
        w[e] = *reinterpret_cast<unsigned*>(&h);
      }
      *reinterpret_cast<uint4*>(tile + sl * slab_bytes + sw128_off(row, ch)) = make_uint4(w[0], w[1], w[2], w[3]);
    }
  }
  sum = (s4[0] + s4[1]) + (s4[2] + s4[3]);
  sq = (q4[0] + q4[1]) + (q4[2] + q4[3]);
}

// 32 bytes of one row to global memory.  `wide`: the buffer is aligned to 32 bytes (callers guarantee 16); one store then
// fills a sector that two 16-byte stores would each write in part.
__device__ inline void store_32b(void* to, const unsigned (&w)[8], bool wide) {
  if (wide) {
    asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};\n" ::"l"(to), "r"(w[0]), "r"(w[1]), "r"(w[2]), "r"(w[3]),
                 "r"(w[4]), "r"(w[5]), "r"(w[6]), "r"(w[7]) : "memory");
  } else {
    *reinterpret_cast<uint4*>(to) = make_uint4(w[0], w[1], w[2], w[3]);
    *(reinterpret_cast<uint4*>(to) + 1) = make_uint4(w[4], w[5], w[6], w[7]);
  }
}

// LayerNorm folded into the MMA for a tile that stays as it is.  One more K step adds s c0 - mean c1 to the raw product,
// s = 1 / rstd, so that rstd times the accumulator is the normalised projection and a reader of the accumulator needs no
// tables.  The step multiplies bf16 whatever the tile holds: a bf16 state reaches far beyond fp16, and so do its means and
// spreads.  Three bf16 parts carry the 24 bits of a float; of the nine products of two such triples eight fit the columns
// (0-7 mean and c1, 8-15 s and c0), and the one left out, third part times third part, is 2^-34 of the whole or less.
__device__ inline void bf16_parts(float x, unsigned (&p)[3]) {
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    const __nv_bfloat16 h = __float2bfloat16_rn(x);
    p[i] = __bfloat16_as_ushort(h);
    x -= __bfloat162float(h);
  }
}
__device__ inline uint4 ln_aug_row_cols(float x) {
  unsigned p[3];
  bf16_parts(x, p);
  return make_uint4(p[0] | p[0] << 16, p[1] | p[1] << 16, p[0] | p[2] << 16, p[1] | p[2] << 16);
}
__device__ inline uint4 ln_aug_weight_cols(float x) {
  unsigned p[3];
  bf16_parts(x, p);
  return make_uint4(p[0] | p[1] << 16, p[0] | p[1] << 16, p[2] | p[0] << 16, p[2] | p[1] << 16);
}
// The row's columns 0-7 to `at`, 8-15 `region` bytes further on; returns the rstd to apply to the accumulator.  rstd = 0 (the
// row's sum of squares passed the float range): the offset alone, at a scale that no product reaches.
__device__ inline float ln_aug_row(unsigned char* at, int region, float mean, float rstd) {
  const bool none = rstd == 0.f;
  rstd = none ? 7.8886091e-31f : rstd;                   // 2^-100
  *reinterpret_cast<uint4*>(at) = ln_aug_row_cols(none ? 0.f : -mean);
  float s;
  asm("rcp.approx.ftz.f32 %0, %1;\n" : "=f"(s) : "f"(rstd));
  *reinterpret_cast<uint4*>(at + region) = ln_aug_row_cols(s);
  return rstd;
}
__device__ inline void ln_aug_weight(unsigned char* at, int region, float2 c01) {
  *reinterpret_cast<uint4*>(at) = ln_aug_weight_cols(c01.y);
  *reinterpret_cast<uint4*>(at + region) = ln_aug_weight_cols(c01.x);
}

// LayerNorm folded into the MMA, activation side.  Two threads per tile row (hf = 0 / 1), each owning four of the
// eight 16-byte chunks of every 64-channel slab of a K-major 128-byte-swizzled bf16 tile: the row is rewritten in
// place as fp16 scaled by its rstd, and hf = 0 writes the row's augmentation columns (m_hi, m_lo, m_hi, 1, 1, 0, 0, 0),
// m = -mean * rstd, to `aug_row` (16 bytes of a K-major no-swizzle region).  Against weight columns
// (c1_hi, c1_hi, c1_lo, c0_hi, c0_lo) one more K step then adds m * c1 + c0, so the accumulator holds LN(z) W^T.
// The two threads of a row must be neighbouring lanes of a converged warp.
__device__ inline void convert_row_ln_fp16(unsigned char* tile, int nslab, int slab_bytes, unsigned char* aug_row, int row,
                                           int hf, int c, float eps, float2* stats_out = nullptr) {
  uint4 raw[2][4];
#pragma unroll
  for (int sl = 0; sl < 2; ++sl)
#pragma unroll
    for (int j = 0; j < 4; ++j)
      raw[sl][j] = sl < nslab ? *reinterpret_cast<const uint4*>(tile + sl * slab_bytes + sw128_off(row, hf * 4 + j))
                              : make_uint4(0, 0, 0, 0);
  float s4[4] = {0.f, 0.f, 0.f, 0.f}, q4[4] = {0.f, 0.f, 0.f, 0.f};   // four independent chains
#pragma unroll
  for (int sl = 0; sl < 2; ++sl)
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const unsigned w[4] = {raw[sl][j].x, raw[sl][j].y, raw[sl][j].z, raw[sl][j].w};
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const float lo = __uint_as_float(w[e] << 16), hi = __uint_as_float(w[e] & 0xffff0000u);
        s4[e] += lo + hi;
        q4[e] = fmaf(lo, lo, q4[e]);
        q4[e] = fmaf(hi, hi, q4[e]);
      }
    }
  float sum = (s4[0] + s4[1]) + (s4[2] + s4[3]), sq = (q4[0] + q4[1]) + (q4[2] + q4[3]);
  sum += __shfl_xor_sync(0xffffffffu, sum, 1);
  sq += __shfl_xor_sync(0xffffffffu, sq, 1);
  const float mean = sum / (float)c;
  const float rstd = rsqrtf(fmaxf(sq / (float)c - mean * mean, 0.f) + eps);
#pragma unroll
  for (int sl = 0; sl < 2; ++sl)
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      if (sl < nslab) {
        unsigned w[4] = {raw[sl][j].x, raw[sl][j].y, raw[sl][j].z, raw[sl][j].w};
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          __half2 h = __floats2half2_rn(__uint_as_float(w[e] << 16) * rstd, __uint_as_float(w[e] & 0xffff0000u) * rstd);
          w[e] = *reinterpret_cast<unsigned*>(&h);
        }
        *reinterpret_cast<uint4*>(tile + sl * slab_bytes + sw128_off(row, hf * 4 + j)) = make_uint4(w[0], w[1], w[2], w[3]);
      }
    }
  if (hf == 0 && stats_out) *stats_out = make_float2(mean, rstd);   // for a later stage that normalises the same row
  if (hf == 0) {
    const float mm = -mean * rstd;
    const __half mh = __float2half_rn(mm), ml = __float2half_rn(mm - __half2float(mh));
    const __half one = __float2half_rn(1.0f), zero = __float2half_rn(0.0f);
    __half2 p0 = __halves2half2(mh, ml), p1 = __halves2half2(mh, one), p2 = __halves2half2(one, zero),
            p3 = __halves2half2(zero, zero);
    *reinterpret_cast<uint4*>(aug_row) = make_uint4(*reinterpret_cast<unsigned*>(&p0), *reinterpret_cast<unsigned*>(&p1),
                                                    *reinterpret_cast<unsigned*>(&p2), *reinterpret_cast<unsigned*>(&p3));
  }
}

__device__ inline float2 unpack_h2(unsigned w) {
  return __half22float2(*reinterpret_cast<const __half2*>(&w));
}
#endif  // __CUDACC__

}  // namespace ntp
