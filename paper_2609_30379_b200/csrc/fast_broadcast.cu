// The gather + LayerNorm pair broadcast (Eq. 1 line 1; Sec. 3.2 "Creating axes through broadcasting"):
//   z[s,i,j,:] = LN(u[s,i,:] + v[s,j,:]) * gamma + beta, bf16 out, a pure streaming write of the packed pair state.
//
// The normalisation is taken apart into per-token and per-pair pieces so that the loop over positions holds no
// reduction.  With uc, vc the rows minus their own channel means, x = uc_i + vc_j has zero mean and
//   var_ij = (|uc_i|^2 + |vc_j|^2 + 2 uc_i . vc_j) / c ,      z = (uc_i g + vc_j g) rstd_ij + beta .
// Everything per token is done once by a small kernel over the T1 token rows (broadcast_prep_kernel: centred rows,
// the column rows already times gamma, bf16 copies of both for the dot products, squared norms).  The c-long dot
// products of a band of rows with a chunk of columns are a small matrix product, taken with mma.sync on bf16
// operands.  Each centred row is kept as a high and a low bf16 part (x = hi + lo up to 2^-17 |x|) and the product
// is hi.hi + hi.lo + lo.hi with float accumulation: when the row and column terms nearly cancel the variance is a
// small difference of the moments, and single bf16 operands (2^-9 per factor) were measured to miss the tolerance
// there.  What is left per position and channel pair is one packed add, one packed fma, one conversion and an
// eighth of a 16-byte store.
//
// Work split of the streaming kernel: the state is cut into bands of BI pair rows; the columns of all bands, laid
// end to end, are split evenly over a persistent grid; a block walks its share in chunks of up to BJ columns of one
// band.  Per chunk: the column rows arrive by asynchronous copies (the next chunk's during the current one), the
// warps take the BI x BJ dot products and leave rstd in shared memory, then every warp streams its rows of the band.
// LP = c / 16 lanes share a position; a lane owns two runs of 8 channels, c / 2 apart, so a position's lanes write
// c contiguous bytes per store instruction.  Float rows in shared memory are c + 4 floats apart and 16-byte slot f of
// a row sits at f ^ ((f >> 3) & 1), bf16 rows are c + 8 elements apart: streaming reads (slots 2 cl, 2 cl + 1) and
// MMA fragment reads are free of bank conflicts.
#include "fast.cuh"

namespace ntp {

constexpr int BL_BI = 32;                       // pair rows per band
#ifndef BL_OCC
#define BL_OCC 2                                // resident blocks per SM the kernel is compiled for
#endif
#define BL_BJ(C) ((C) <= 128 ? 32 : 16)         // columns per chunk

__device__ inline int bl_swz(int f) { return f ^ ((f >> 3) & 1); }
__device__ inline float2 bl_f2(float x, float y) { return make_float2(x, y); }
__device__ inline unsigned bl_pack(float2 v) {
  unsigned y;
  asm("cvt.rn.bf16x2.f32 %0, %1, %2;\n" : "=r"(y) : "f"(v.y), "f"(v.x));
  return y;
}
__device__ inline float2 bl_lo(unsigned w) { return bl_f2(__uint_as_float(w << 16), __uint_as_float(w & 0xffff0000u)); }
__device__ inline void bl_cp16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src));
}
__device__ inline void bl_cp4(void* dst, const void* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src));
}

// ------------------------------------------------------------------------------------------
// Per-token preparation, in place: rows [0, rows_u) of u become uc; rows of v become vc * gamma; bf16 copies of
// uc and vc and the squared norms of both go to their own arrays.  One warp per row (two rows for c = 64).
// ------------------------------------------------------------------------------------------
template <int C>
__global__ void __launch_bounds__(256) broadcast_prep_kernel(BcastPrepared p, long long rows_u, long long rows_v,
                                                             const __nv_bfloat16* gamma) {
  pdl_begin();
  constexpr int FPL = C > 128 ? C / 128 : 1;       // 16-byte pieces per lane
  constexpr int RPI = C < 128 ? 128 / C : 1;       // rows per warp
  constexpr int LR = 32 / RPI;                     // lanes per row
  const int lane = threadIdx.x & 31;
  const long long row = ((long long)blockIdx.x * 8 + (threadIdx.x >> 5)) * RPI + lane / LR;
  const bool live = row < rows_u + rows_v;         // dead lanes go through the shuffles with zeros
  const bool is_v = row >= rows_u;
  const long long r = is_v ? row - rows_u : row;
  float* src = (is_v ? p.v : p.u) + r * C;
  float4 x[FPL];
  float s = 0.f;
#pragma unroll
  for (int q = 0; q < FPL; ++q) {
    x[q] = live ? reinterpret_cast<const float4*>(src)[(lane % LR) + 32 * q] : make_float4(0.f, 0.f, 0.f, 0.f);
    s += (x[q].x + x[q].y) + (x[q].z + x[q].w);
  }
#pragma unroll
  for (int o = LR / 2; o; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  const float mean = s * (1.0f / C);
  float ss = 0.f;
#pragma unroll
  for (int q = 0; q < FPL; ++q) {
    x[q].x -= mean; x[q].y -= mean; x[q].z -= mean; x[q].w -= mean;
    ss = fmaf(x[q].x, x[q].x, fmaf(x[q].y, x[q].y, fmaf(x[q].z, x[q].z, fmaf(x[q].w, x[q].w, ss))));
  }
#pragma unroll
  for (int o = LR / 2; o; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
  if (!live) return;
  __nv_bfloat16* bdst = (is_v ? p.vb : p.ub) + r * C;
  __nv_bfloat16* ldst = (is_v ? p.vbl : p.ubl) + r * C;
#pragma unroll
  for (int q = 0; q < FPL; ++q) {
    const int f = (lane % LR) + 32 * q;
    const uint2 hi = make_uint2(bl_pack(bl_f2(x[q].x, x[q].y)), bl_pack(bl_f2(x[q].z, x[q].w)));
    const float2 h0 = bl_lo(hi.x), h1 = bl_lo(hi.y);
    reinterpret_cast<uint2*>(bdst)[f] = hi;
    reinterpret_cast<uint2*>(ldst)[f] = make_uint2(bl_pack(bl_f2(x[q].x - h0.x, x[q].y - h0.y)),
                                                   bl_pack(bl_f2(x[q].z - h1.x, x[q].w - h1.y)));
    if (is_v) {
      const uint2 w = *reinterpret_cast<const uint2*>(gamma + f * 4);
      const float2 ga = bl_lo(w.x), gb = bl_lo(w.y);
      x[q].x *= ga.x; x[q].y *= ga.y; x[q].z *= gb.x; x[q].w *= gb.y;
    }
    reinterpret_cast<float4*>(src)[f] = x[q];
  }
  if (lane % LR == 0) (is_v ? p.nv : p.nu)[r] = ss;
}

struct BlChunk { int s, i0, j, len; };
__device__ inline BlChunk bl_chunk(const long long* band_off, const BcastGeom& m, long long cur, long long end,
                                   int bj) {
  BlChunk c{0, 0, 0, 0};
  if (cur >= end) return c;
  c.s = find_sample(band_off, m.B, cur);
  const int N = m.cols[c.s];
  const int r = (int)(cur - band_off[c.s]);
  c.i0 = (r / N) * BL_BI;
  c.j = r % N;
  c.len = (int)min((long long)min(bj, N - c.j), end - cur);
  return c;
}

// Copy `rows` prepared token rows (float row, the two bf16 rows, squared norm) starting at token row `t0` into shared
// memory.
template <int C>
__device__ inline void bl_stage(const BcastPrepared& p, bool col_side, long long t0, int rows, float4* dF,
                                __nv_bfloat16* dB, __nv_bfloat16* dL, float* dN) {
  constexpr int F4 = C / 4, VS = F4 + 1, B8 = C / 8, BP = C + 8;
  const float4* sf = reinterpret_cast<const float4*>((col_side ? p.v : p.u) + t0 * C);
  const uint4* sb = reinterpret_cast<const uint4*>((col_side ? p.vb : p.ub) + t0 * C);
  const uint4* sl = reinterpret_cast<const uint4*>((col_side ? p.vbl : p.ubl) + t0 * C);
  const float* sn = (col_side ? p.nv : p.nu) + t0;
  for (int e = threadIdx.x; e < rows * F4; e += 256) bl_cp16(dF + (e / F4) * VS + bl_swz(e % F4), sf + e);
  for (int e = threadIdx.x; e < rows * B8; e += 256) {
    bl_cp16(dB + (e / B8) * BP + (e % B8) * 8, sb + e);
    bl_cp16(dL + (e / B8) * BP + (e % B8) * 8, sl + e);
  }
  if (threadIdx.x < rows) bl_cp4(dN + threadIdx.x, sn + threadIdx.x);
}

template <int C, bool ACC>       // ACC: z += the broadcast (persistent pair stream) instead of z = the broadcast
__global__ void __launch_bounds__(256, BL_OCC) broadcast_ln_moments_kernel(BcastPrepared p,
                                                                           const __nv_bfloat16* gamma,
                                                                           const __nv_bfloat16* beta,
                                                                           float eps, __nv_bfloat16* z,
                                                                           BcastGeom m, long long n_cols) {
  pdl_begin();
  constexpr int LP = C / 16;                       // lanes per position in the streaming loop
  constexpr int PPW = 32 / LP;                     // positions per warp-wide instruction
  constexpr int VS = C / 4 + 1;                    // float row pitch in 16-byte pieces
  constexpr int BP = C + 8;                        // bf16 row pitch in elements
  constexpr int BJ = BL_BJ(C);
  constexpr int RS = BJ + 1;                       // pitch of the rstd tile
  extern __shared__ float4 bl_smem[];
  float4* sU = bl_smem;                            // [BI][VS] centred u rows of the band
  float4* sV = sU + BL_BI * VS;                    // [2][BJ][VS] centred v rows of the chunk, times gamma
  __nv_bfloat16* sUb = reinterpret_cast<__nv_bfloat16*>(sV + 2 * BJ * VS);   // [BI][BP] high bf16 parts
  __nv_bfloat16* sUl = sUb + BL_BI * BP;           // [BI][BP] low parts
  __nv_bfloat16* sVb = sUl + BL_BI * BP;           // [2][BJ][BP]
  __nv_bfloat16* sVl = sVb + 2 * BJ * BP;          // [2][BJ][BP]
  float* sR = reinterpret_cast<float*>(sVl + 2 * BJ * BP);                   // [BI][RS] rstd of the chunk's positions
  float* sNu = sR + BL_BI * RS;                    // [BI] squared norms of the centred u rows
  float* sNv = sNu + BL_BI;                        // [2][BJ]
  __shared__ long long band_off[MAXB + 1];         // prefix of bands x columns per sample
  if (threadIdx.x == 0) {
    long long acc = 0;
    for (int s = 0; s < m.B; ++s) {
      band_off[s] = acc;
      acc += (long long)((m.rows[s] + BL_BI - 1) / BL_BI) * m.cols[s];
    }
    band_off[m.B] = acc;
  }
  __syncthreads();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, sub = lane / LP, cl = lane % LP;
  // streaming loop: the lane's channels are (g c/2 + cl 8) .. + 8 for g = 0, 1 = pieces g c/8 + 2 cl + {0, 1}
  int pf[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) pf[q] = bl_swz((q >> 1) * (C / 8) + 2 * cl + (q & 1));
  float2 g2[8], b2[8];
#pragma unroll
  for (int g = 0; g < 2; ++g) {
    const uint4 gw = *reinterpret_cast<const uint4*>(gamma + g * (C / 2) + cl * 8);
    const uint4 bw = *reinterpret_cast<const uint4*>(beta + g * (C / 2) + cl * 8);
    g2[4 * g] = bl_lo(gw.x); g2[4 * g + 1] = bl_lo(gw.y); g2[4 * g + 2] = bl_lo(gw.z); g2[4 * g + 3] = bl_lo(gw.w);
    b2[4 * g] = bl_lo(bw.x); b2[4 * g + 1] = bl_lo(bw.y); b2[4 * g + 2] = bl_lo(bw.z); b2[4 * g + 3] = bl_lo(bw.w);
  }
  long long cur = n_cols * blockIdx.x / gridDim.x;
  const long long end = n_cols * (blockIdx.x + 1) / gridDim.x;
  BlChunk ck = bl_chunk(band_off, m, cur, end, BJ);
  if (ck.len > 0) bl_stage<C>(p, true, m.v_off[ck.s] + ck.j, ck.len, sV, sVb, sVl, sNv);
  asm volatile("cp.async.commit_group;\n" ::);
  int band_s = -1, band_i0 = -1;
  for (int k = 0; ck.len > 0; ++k) {
    cur += ck.len;
    const BlChunk nx = bl_chunk(band_off, m, cur, end, BJ);
    const int N = m.cols[ck.s], R = m.rows[ck.s];
    if (ck.s != band_s || ck.i0 != band_i0) {            // a new band: fetch its rows (the last reader left at the
      band_s = ck.s;                                     // barrier that closed the previous chunk)
      band_i0 = ck.i0;
      bl_stage<C>(p, false, m.u_off[ck.s] + ck.i0, min(BL_BI, R - ck.i0), sU, sUb, sUl, sNu);
    }
    asm volatile("cp.async.commit_group;\n" ::);
    const int nb = (k + 1) & 1;
    if (nx.len > 0)
      bl_stage<C>(p, true, m.v_off[nx.s] + nx.j, nx.len, sV + nb * BJ * VS, sVb + nb * BJ * BP, sVl + nb * BJ * BP,
                  sNv + nb * BJ);
    asm volatile("cp.async.commit_group;\n" ::);
    asm volatile("cp.async.wait_group 1;\n" ::);         // all but the next chunk's copies
    __syncthreads();
    const float4* sVk = sV + (k & 1) * BJ * VS;
    const __nv_bfloat16* sVbk = sVb + (k & 1) * BJ * BP;
    const __nv_bfloat16* sVlk = sVl + (k & 1) * BJ * BP;
    const float* sNvk = sNv + (k & 1) * BJ;
    // dot products of the chunk's columns (MMA rows) with the band's rows (MMA columns) -> rstd.  Rows past the
    // band's or the chunk's end hold stale shared memory: their results are computed and never read.
    {
      constexpr int MT = BJ / 16, UNITS = MT * (BL_BI / 8);
      if (warp < UNITS) {
        const int mt = warp % MT, nt = warp / MT, gq = lane >> 2, t = lane & 3;
        const int oa = (mt * 16 + gq) * (BP / 2) + t, ob = (nt * 8 + gq) * (BP / 2) + t;
        const unsigned* fa = reinterpret_cast<const unsigned*>(sVbk) + oa;
        const unsigned* la = reinterpret_cast<const unsigned*>(sVlk) + oa;
        const unsigned* fb = reinterpret_cast<const unsigned*>(sUb) + ob;
        const unsigned* lb = reinterpret_cast<const unsigned*>(sUl) + ob;
        float d[2][4] = {};
        auto mma = [](float* dd, const unsigned (&a)[4], unsigned b0, unsigned b1) {
          asm volatile(
              "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};\n"
              : "+f"(dd[0]), "+f"(dd[1]), "+f"(dd[2]), "+f"(dd[3])
              : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
        };
#pragma unroll
        for (int ks = 0; ks < C / 16; ++ks) {
          const unsigned ah[4] = {fa[ks * 8], fa[8 * (BP / 2) + ks * 8], fa[ks * 8 + 4], fa[8 * (BP / 2) + ks * 8 + 4]};
          const unsigned al[4] = {la[ks * 8], la[8 * (BP / 2) + ks * 8], la[ks * 8 + 4], la[8 * (BP / 2) + ks * 8 + 4]};
          const unsigned bh0 = fb[ks * 8], bh1 = fb[ks * 8 + 4], bl0 = lb[ks * 8], bl1 = lb[ks * 8 + 4];
          mma(d[0], ah, bh0, bh1);          // hi . hi
          mma(d[1], ah, bl0, bl1);          // hi . lo
          mma(d[1], al, bh0, bh1);          // lo . hi
        }
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const int jj = mt * 16 + gq + (e >> 1) * 8, ii = nt * 8 + 2 * t + (e & 1);
          const float var = (sNu[ii] + sNvk[jj] + 2.f * (d[0][e] + d[1][e])) * (1.0f / C);
          sR[ii * RS + jj] = rsqrtf(fmaxf(var, 0.f) + eps);
        }
      }
    }
    __syncthreads();
    // stream the band's rows: z = (uc g + vc g) rstd + beta
    const long long z_end = m.z_off[m.B - 1] + (long long)m.rows[m.B - 1] * m.cols[m.B - 1];
    const int nj = ck.len;
#pragma unroll 1
    for (int rr = 0; rr < BL_BI / 8; ++rr) {
      const int r = warp * (BL_BI / 8) + rr, i = ck.i0 + r;
      if (i >= R) break;
      float2 ug[8];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const float4 t4 = sU[r * VS + pf[q]];
        ug[2 * q] = __fmul2_rn(bl_f2(t4.x, t4.y), g2[2 * q]);
        ug[2 * q + 1] = __fmul2_rn(bl_f2(t4.z, t4.w), g2[2 * q + 1]);
      }
      const long long pos0 = m.z_off[ck.s] + (long long)i * N + ck.j;
      uint4* zp = reinterpret_cast<uint4*>(z + (pos0 + sub) * C) + cl;
      const float4* vp = sVk + sub * VS;
      const float* rp = sR + r * RS + sub;
#pragma unroll 2
      for (int jb = 0; jb < nj; jb += PPW, zp += PPW * (C / 8), vp += PPW * VS, rp += PPW) {
        const bool ok = jb + sub < nj && NT_IN(pos0 + jb + sub, z_end, NT_SITE_FAST_BROADCAST);
        const float rs = *rp;                // positions past the run: stale shared memory, computed, never stored
        const float2 r2 = bl_f2(rs, rs);
        float2 y[8];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const float4 t4 = vp[pf[q]];
          y[2 * q] = __ffma2_rn(__fadd2_rn(ug[2 * q], bl_f2(t4.x, t4.y)), r2, b2[2 * q]);
          y[2 * q + 1] = __ffma2_rn(__fadd2_rn(ug[2 * q + 1], bl_f2(t4.z, t4.w)), r2, b2[2 * q + 1]);
        }
        if (ok) {
#pragma unroll
          for (int g = 0; g < 2; ++g) {
            if (ACC) {
              const uint4 old = zp[g * (C / 16)];
              y[4 * g] = __fadd2_rn(y[4 * g], bl_lo(old.x));
              y[4 * g + 1] = __fadd2_rn(y[4 * g + 1], bl_lo(old.y));
              y[4 * g + 2] = __fadd2_rn(y[4 * g + 2], bl_lo(old.z));
              y[4 * g + 3] = __fadd2_rn(y[4 * g + 3], bl_lo(old.w));
            }
            zp[g * (C / 16)] = make_uint4(bl_pack(y[4 * g]), bl_pack(y[4 * g + 1]), bl_pack(y[4 * g + 2]),
                                          bl_pack(y[4 * g + 3]));
          }
        }
      }
    }
    __syncthreads();                           // the chunk's readers are done before its buffers are refilled
    ck = nx;
  }
  asm volatile("cp.async.wait_group 0;\n" ::);
}

bool fast_broadcast_supported(int c_z) { return c_z == 64 || c_z == 128 || c_z == 256; }

size_t fast_broadcast_scratch_bytes(long long rows_u, long long rows_v, int c_z) {
  const size_t ru = (size_t)rows_u, rv = (size_t)rows_v, c = (size_t)c_z;
  return align_up(ru * c * 4, 256) + align_up(rv * c * 4, 256) + 2 * align_up(ru * c * 2, 256) +
         2 * align_up(rv * c * 2, 256) + align_up(ru * 4, 256) + align_up(rv * 4, 256);
}

BcastPrepared fast_broadcast_carve(void* ws, long long rows_u, long long rows_v, int c_z) {
  const size_t ru = (size_t)rows_u, rv = (size_t)rows_v, c = (size_t)c_z;
  char* b = (char*)ws;
  BcastPrepared p;
  p.u = (float*)b; b += align_up(ru * c * 4, 256);
  p.v = (float*)b; b += align_up(rv * c * 4, 256);
  p.ub = (__nv_bfloat16*)b; b += align_up(ru * c * 2, 256);
  p.vb = (__nv_bfloat16*)b; b += align_up(rv * c * 2, 256);
  p.ubl = (__nv_bfloat16*)b; b += align_up(ru * c * 2, 256);
  p.vbl = (__nv_bfloat16*)b; b += align_up(rv * c * 2, 256);
  p.nu = (float*)b; b += align_up(ru * 4, 256);
  p.nv = (float*)b;
  return p;
}

nt_status fast_broadcast_prep(const BcastPrepared& p, long long rows_u, long long rows_v, const void* gamma, int c_z,
                              cudaStream_t st, const char* scope) {
  const long long rows = rows_u + rows_v;
  if (rows == 0) return NT_OK;
  const int rpb = 8 * (c_z < 128 ? 128 / c_z : 1);
  const unsigned blocks = (unsigned)((rows + rpb - 1) / rpb);
  const __nv_bfloat16* g = (const __nv_bfloat16*)gamma;
  LaunchScope ls(scope, st);
  if (c_z == 64) launch_kernel(broadcast_prep_kernel<64>, blocks, 256, 0, st, p, rows_u, rows_v, g);
  else if (c_z == 128) launch_kernel(broadcast_prep_kernel<128>, blocks, 256, 0, st, p, rows_u, rows_v, g);
  else launch_kernel(broadcast_prep_kernel<256>, blocks, 256, 0, st, p, rows_u, rows_v, g);
  return cuda_ok();
}

template <int C>
static size_t bl_smem_bytes() {
  constexpr int VS = C / 4 + 1, BJ = BL_BJ(C), BP = C + 8;
  return (size_t)(BL_BI + 2 * BJ) * VS * 16 + (size_t)(BL_BI + 2 * BJ) * BP * 2 * 2 +
         (size_t)(BL_BI * (BJ + 1) + BL_BI + 2 * BJ) * 4;
}

template <int C, bool ACC>
static nt_status bl_launch(const BcastPrepared& p, const __nv_bfloat16* g, const __nv_bfloat16* b, float eps,
                           __nv_bfloat16* z, const BcastGeom& m, long long items, cudaStream_t st,
                           const char* scope) {
  static bool attr_set_dev[64] = {};
  int dev = 0;
  cudaGetDevice(&dev);
  const size_t smem = bl_smem_bytes<C>();
  if (dev >= 0 && dev < 64 && !attr_set_dev[dev]) {
    if (cudaFuncSetAttribute(broadcast_ln_moments_kernel<C, ACC>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)smem) != cudaSuccess)
      return cuda_ok();
    attr_set_dev[dev] = true;
  }
  // a chunk of columns per block while that fills the GPU; smaller pieces for small states (a 32 x 32 piece is a chain of
  // 32 dependent steps per warp: 12.6 us on lengths 7-61, 8.2 with eight columns per block)
  const long long cap = (long long)sm_count() * BL_OCC;
  long long blocks = (items + 7) / 8;
  if (blocks > cap) blocks = cap;
  LaunchScope ls(scope, st);
  launch_kernel(broadcast_ln_moments_kernel<C, ACC>, (unsigned)blocks, 256, smem, st, p, g, b, eps, z, m, items);
  return NT_OK;
}

nt_status fast_broadcast_ln_geom(const BcastPrepared& p, const void* gamma, const void* beta, float eps, int c_z,
                                 void* z, const BcastGeom& m, cudaStream_t st, bool accumulate, const char* scope) {
  long long items = 0;      // columns of all bands of BL_BI pair rows, laid end to end
  for (int s = 0; s < m.B; ++s) items += (long long)((m.rows[s] + BL_BI - 1) / BL_BI) * m.cols[s];
  if (items == 0) return NT_OK;
  const __nv_bfloat16* g = (const __nv_bfloat16*)gamma;
  const __nv_bfloat16* b = (const __nv_bfloat16*)beta;
  __nv_bfloat16* zz = (__nv_bfloat16*)z;
  nt_status rc = NT_OK;
  if (accumulate) {
    if (c_z == 64) rc = bl_launch<64, true>(p, g, b, eps, zz, m, items, st, scope);
    else if (c_z == 128) rc = bl_launch<128, true>(p, g, b, eps, zz, m, items, st, scope);
    else rc = bl_launch<256, true>(p, g, b, eps, zz, m, items, st, scope);
  } else {
    if (c_z == 64) rc = bl_launch<64, false>(p, g, b, eps, zz, m, items, st, scope);
    else if (c_z == 128) rc = bl_launch<128, false>(p, g, b, eps, zz, m, items, st, scope);
    else rc = bl_launch<256, false>(p, g, b, eps, zz, m, items, st, scope);
  }
  if (rc != NT_OK) return rc;
  return cuda_ok();
}

nt_status fast_broadcast_ln(const BcastPrepared& p, const void* gamma, const void* beta, float eps, int c_z, void* z,
                            const BatchMeta& m, cudaStream_t st, bool accumulate) {
  BcastGeom g;
  g.B = m.B;
  for (int s = 0; s < MAXB; ++s) {
    g.rows[s] = g.cols[s] = s < m.B ? m.N[s] : 0;
    g.u_off[s] = g.v_off[s] = m.tok_off[s];
    g.z_off[s] = m.pair_off[s];
  }
  return fast_broadcast_ln_geom(p, gamma, beta, eps, c_z, z, g, st, accumulate,
                                accumulate ? "broadcast_ln_add" : "broadcast_ln");
}

}  // namespace ntp
