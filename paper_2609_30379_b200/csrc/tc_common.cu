// Host side of the TMA plumbing: resolves cuTensorMapEncodeTiled through the runtime (no link-time
// dependency on the driver library) and encodes tiled maps for 16-bit elements.
#include "tc_common.cuh"

namespace ntp {

EncodeTiledFn get_encode_tiled() {
  static EncodeTiledFn fn = nullptr;
  static bool tried = false;
  if (!tried) {
    tried = true;
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = (EncodeTiledFn)p;
  }
  return fn;
}

bool make_tmap_16bit(CUtensorMap* map, const void* base, int rank, const unsigned long long* dims,
                     const unsigned long long* strides_bytes, const unsigned* box, int swizzle_bytes, int l2_promotion_bytes) {
  EncodeTiledFn enc = get_encode_tiled();
  if (!enc) return false;
  cuuint64_t gdim[5];
  cuuint64_t gstr[5];
  cuuint32_t bdim[5], estr[5];
  for (int i = 0; i < rank; ++i) {
    gdim[i] = dims[i];
    bdim[i] = box[i];
    estr[i] = 1;
    if (i + 1 < rank) gstr[i] = strides_bytes[i];
  }
  const CUtensorMapSwizzle sw = swizzle_bytes == 0    ? CU_TENSOR_MAP_SWIZZLE_NONE
                               : swizzle_bytes == 32 ? CU_TENSOR_MAP_SWIZZLE_32B
                               : swizzle_bytes == 64 ? CU_TENSOR_MAP_SWIZZLE_64B
                                                     : CU_TENSOR_MAP_SWIZZLE_128B;
  // bf16 and fp16 tiles move identically (no conversion on the way), so one 16-bit type serves both
  CUresult r = enc(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, (cuuint32_t)rank, const_cast<void*>(base), gdim, gstr, bdim,
                   estr, CU_TENSOR_MAP_INTERLEAVE_NONE, sw,
                   l2_promotion_bytes >= 128 ? CU_TENSOR_MAP_L2_PROMOTION_L2_128B
                   : l2_promotion_bytes == 64 ? CU_TENSOR_MAP_L2_PROMOTION_L2_64B : CU_TENSOR_MAP_L2_PROMOTION_NONE,
                   CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS;
}

bool make_tmap_bf16(CUtensorMap* map, const void* base, int rank, const unsigned long long* dims,
                    const unsigned long long* strides_bytes, const unsigned* box) {
  return make_tmap_16bit(map, base, rank, dims, strides_bytes, box, 128);
}

// Testing aid behind nt_debug_expire_wait: the bounded wait every tensor-core kernel uses, on a barrier nobody arrives
// at, with a limit of a few thousand clocks.  The warp records NT_ERR_TIMEOUT in the status word, raises the CTA's
// abort flag and the kernel ends normally: exactly what a kernel does when one of its waits runs out.
__global__ void expire_wait_kernel(int* status, long long limit_clocks, int* observed) {
  pdl_begin();
  __shared__ __align__(8) unsigned long long bar;
  __shared__ int abort_flag;
  if (threadIdx.x == 0) {
    abort_flag = 0;
    mbar_init(&bar, 1);
    mbar_fence_init();
  }
  __syncthreads();
  AbortCtx ab{status, &abort_flag};
  bool ok = true;
  if (threadIdx.x == 0) ok = mbar_wait(&bar, 0, ab, limit_clocks);      // phase 0 never completes
  __syncthreads();
  // a later wait of the same CTA gives up after the short limit, as in the real kernels
  if (threadIdx.x == 32) mbar_wait(&bar, 0, ab);
  if (threadIdx.x == 0 && observed) *observed = (ok ? 0 : 1) | (abort_flag ? 2 : 0);
}

nt_status launch_expire_wait(int* status, long long limit_clocks, int* observed, cudaStream_t st) {
  {
    LaunchScope ls("debug_expire_wait", st);
    launch_kernel(expire_wait_kernel, 1, 64, 0, st, status, limit_clocks, observed);
  }
  return cuda_ok("expire wait launch");
}

}  // namespace ntp
