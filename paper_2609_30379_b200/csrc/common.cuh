// Shared declarations of libnested_pair's CUDA sources: batch metadata passed by value to
// kernels, dtype helpers, launch bookkeeping.
#pragma once

#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>
#include <stdio.h>

#include <atomic>

#include "../../include/nested_pair.h"

namespace ntp {

constexpr int MAXB = 64;  // samples per launch group; larger batches are processed in groups

// Per-group batch metadata, computed on the host from the canonical lengths (App. A: canonical
// sizes stay on the host) and passed by value, so kernels decode positions without a global read.
// Offsets are absolute (they index the caller's full packed buffers).
struct BatchMeta {
  int B;
  int N[MAXB];
  long long tok_off[MAXB + 1];
  long long pair_off[MAXB + 1];
  // prefix of N_s * ld_s with ld_s = round_up(N_s, 8): size of one channel plane of the
  // channel-major intermediates; element (s, c, i, k) of a C-channel buffer lives at
  // C * cm_off[s] + c * N_s * ld_s + i * ld_s + k.
  long long cm_off[MAXB + 1];
};

__host__ __device__ inline int round_up8(int n) { return (n + 7) & ~7; }

// largest s with off[s] <= p (p < off[B]); empty samples are skipped because their successor
// shares the offset.
__device__ inline int find_sample(const long long* off, int B, long long p) {
  int lo = 0, hi = B;  // invariant: off[lo] <= p < off[hi]
  while (hi - lo > 1) {
    int mid = (lo + hi) >> 1;
    if (off[mid] <= p) lo = mid; else hi = mid;
  }
  return lo;
}

template <typename T> struct Cvt;
template <> struct Cvt<float> {
  __device__ static inline float ld(const float* p) { return *p; }
  __device__ static inline void st(float* p, float v) { *p = v; }
};
template <> struct Cvt<__nv_bfloat16> {
  __device__ static inline float ld(const __nv_bfloat16* p) { return __bfloat162float(*p); }
  __device__ static inline void st(__nv_bfloat16* p, float v) { *p = __float2bfloat16_rn(v); }
};

// ---- checked build (-DNT_DEBUG_BOUNDS -rdc=true): the tool that would find a stray index is not available where
// this library is developed, so the kernels can check themselves.  Every global index a kernel derives from the
// offsets is tested against the extent its buffer was given at the boundary; a stray one is counted, the first one is
// recorded (site, index) and the access is SKIPPED, so the checked build never faults.  In the normal build NT_IN is
// the constant true and costs nothing.  nt_debug_bounds_report reads the record.
enum NtBoundSite {
  NT_SITE_DECODE = 1, NT_SITE_PROJ_OUT, NT_SITE_CONTRACT_OUT, NT_SITE_BROADCAST_OUT, NT_SITE_ATTN_OUT, NT_SITE_SEGMENT_OUT,
  NT_SITE_FAST_BROADCAST, NT_SITE_FAST_SEGMENT, NT_SITE_FRAG_ATTN_OUT, NT_SITE_ROW_ATTN_OUT, NT_SITE_ATTN_IN_BIAS,
  NT_SITE_TOKEN_GEMM_OUT, NT_SITE_RECT_BROADCAST
};
#ifdef NT_DEBUG_BOUNDS
extern __device__ int g_nt_bounds[4];     // violations, site of the first, its index (low / high word)
__device__ inline bool nt_in_bounds(long long idx, long long extent, int site) {
  if (idx >= 0 && idx < extent) return true;
  if (atomicAdd(&g_nt_bounds[0], 1) == 0) {
    g_nt_bounds[1] = site;
    g_nt_bounds[2] = (int)(idx & 0xffffffffll);
    g_nt_bounds[3] = (int)(idx >> 32);
  }
  return false;
}
#define NT_IN(idx, extent, site) ::ntp::nt_in_bounds((long long)(idx), (long long)(extent), (site))
#else
#define NT_IN(idx, extent, site) true
#endif

extern std::atomic<long long> g_launches;
extern int g_force_generic;

// Counts a kernel launch and, while per-kernel profiling is on (nt_profile_begin), brackets it with
// CUDA events on the launching stream.  Construct before the launch, destroy after it.
struct LaunchScope {
  LaunchScope(const char* name, cudaStream_t st);
  ~LaunchScope();
  cudaStream_t st;
  int slot;
};

// Launch with programmatic stream serialisation: the kernel may be set up while its predecessor in the stream drains, and
// waits for it in pdl_begin, which every kernel of the library calls before it touches global memory.  (2.4 -> 1.9 us of
// host time per launch, and the launch latency, barrier set-up and TMEM allocation of a small kernel run in the shadow of
// the one before.)
template <typename... KArgs, typename... Args>
inline void launch_kernel(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, Args&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at;
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
}
#ifdef __CUDACC__
// Every thread: waits until the kernels before this one in the stream are complete and their writes visible.  A grid that
// leaves SMs free lets its successor in at once (the successor then waits in its own pdl_begin); a grid that fills the GPU
// does not: the successor's blocks could only sit beside it (2.37 -> 2.41 ms for the near-uniform stack when they did).  The
// line lies at 128 blocks, an eighth below the 148 SMs this library is built for.
// Loads before this point, and loads the compiler may move there (const __restrict__, __ldg), must not read what an
// earlier kernel wrote.
__device__ inline void pdl_begin() {
  if ((unsigned long long)gridDim.x * gridDim.y < 128) asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory");
  asm volatile("griddepcontrol.wait;\n" ::: "memory");
}
#endif

// Reports the pending CUDA error (and where it was seen) on stderr and maps it to NT_ERR_CUDA.
nt_status cuda_fail(const char* where);

inline nt_status cuda_ok(const char* where = "kernel launch") {
  return cudaPeekAtLastError() == cudaSuccess ? NT_OK : cuda_fail(where);
}

// Builds the metadata of samples [s0, s1) (s1 - s0 <= MAXB) given absolute prefix arrays.
void fill_meta(BatchMeta& m, const int64_t* lengths_h, int s0, int s1, long long tok0, long long pair0,
               long long cm0);

struct GroupIter {  // walks a batch in groups of MAXB samples
  const int64_t* len;
  int B, s0 = 0;
  long long tok = 0, pair = 0, cm = 0;
  GroupIter(const int64_t* l, int b) : len(l), B(b) {}
  bool next(BatchMeta& m);
};

// one tiny launch whose only wait runs out (testing aid)
nt_status launch_expire_wait(int* status, long long limit_clocks, int* observed, cudaStream_t st);

// exponential-rate microbenchmark (one CTA of 512 threads per block index; see exp_rate.cu)
nt_status launch_exp_rate(int variant, int iters, int blocks, float* sink, long long* clocks, cudaStream_t st);

// multiprocessors of the current device (queried once per device)
int sm_count();

static inline size_t align_up(size_t v, size_t a) { return (v + a - 1) / a * a; }

}  // namespace ntp
