// Triangle-update output stage on tcgen05 (float accumulate), in place on the pair state:
//   z += sigmoid(LN_in(z) W_g^T) * (LN_out(t) W_o^T)
// t is the contraction result in channel-major layout (t[c][i][j], j contiguous), so a run of 64
// positions of one pair row is, per channel, 128 contiguous bytes: exactly the MN-major operand
// form of the MMA (positions are M, channels are K).  The output gate is recomputed here from z
// instead of being stored by the input projection, which saves one write and one read of a
// [T2, c_z] buffer.  Both LayerNorms are folded into the weights (W' = W gamma; W_o' fp16 against the
// fp16 t, W_g' bf16 against the bf16 state itself), so NOTHING has to touch the tiles between the TMA
// load and the MMA: the MMAs start as soon as the tiles land, four warps take the row statistics of t
// and z from the same tiles meanwhile and write them as one more K step of either product (ln_aug_row), and the epilogue is
//   z += (tanh(g / 2) + 1) (o / 2),  o / 2 = (rstd_t / 2) acc_o,  g / 2 = (rstd_z / 2) acc_g.
// Bound: the life of a z stage -- load, statistics, epilogue, store -- with room for two of them beside the weights.
// Tables of the LayerNorm constants in the epilogue (four 16-byte reads per four channels and warp) were two fifths of
// the shared-memory traffic, which is why the constants travel through the tensor cores instead.
// Measured at eight samples of about 215 positions: 76.4 us with eight storing epilogue warps, 72.4 us with sixteen and a
// store warp, 70.3 us without the tables.  (Without statistics and arithmetic it takes 62 us.  Storing from registers, 78 us,
// and eight statistics warps, 73 us, were slower.)
//
// A tile is two 64-position chunks (s, i, j0).  The t chunks and the z tile travel through rings of
// their own: a t stage is free once the MMAs and the statistics have read it, a z stage only after the
// epilogue has written the new z into it and the TMA stores have read it (clipped at the row end, so
// nothing outside sum N^2 is touched) -- so the t loads of the tile after next start one epilogue early.
#include <cstring>

#include "fast.cuh"
#include "tc_common.cuh"

namespace ntp {

constexpr int TO_EPI = 16;                              // epilogue warps
constexpr int TO_STORE = 6 + TO_EPI;                    // the warp that stores finished tiles
constexpr int TO_THREADS = 32 * (TO_STORE + 1);         // producer, MMA, 4 statistics warps, epilogue, store
constexpr int TO_MAXB = 12;

struct TriOutParams {
  CUtensorMap zmap[TO_MAXB];     // {c_z, N (j), N (i), 1}, box {64, 32, 1, 1}
  CUtensorMap tmap[TO_MAXB];     // {N (j), N (i), c_h, 1}, box {64, 1, c_h, 1}
  CUtensorMap womap;             // {c_h, c_z}, box {64, c_z}
  CUtensorMap wgmap;             // {c_z, c_z}, box {64, c_z}
  long long chunk_off[TO_MAXB + 1];
  int N[TO_MAXB];
  int B, c_z, c_h;
  float eps;
  const float2* c01o;            // [c_z]
  const float2* c01g;            // [c_z]
  int* status;
  const float2* zstats;          // nullable: (mean, rstd) of every z row by packed position, left by the input projection
  long long pos_off[TO_MAXB];
};

__device__ inline bool to_decode(const TriOutParams& p, long long q, int& s, int& i, int& j0) {
  if (q >= p.chunk_off[p.B]) return false;
  s = 0;
  while (s + 1 < p.B && q >= p.chunk_off[s + 1]) ++s;
  const int cpr = (p.N[s] + 63) / 64;
  // a sample's chunk count N * ceil(N / chunk) is far below 2^32 (N < 2^20 is checked on the host): 32-bit division
  const unsigned r = (unsigned)(q - p.chunk_off[s]);
  i = (int)(r / (unsigned)cpr);
  j0 = (int)(r - (unsigned)i * (unsigned)cpr) * 64;
  return true;
}

__device__ inline float to_tanh(float x) {
  float t;
  asm("tanh.approx.f32 %0, %1;\n" : "=f"(t) : "f"(x));
  return t;
}

__global__ void __launch_bounds__(TO_THREADS, 1) tri_out_kernel(const __grid_constant__ TriOutParams p) {
  extern __shared__ unsigned char smem_raw[];
  __shared__ __align__(8) unsigned long long bars[19];
  __shared__ float2 sStats[2][128];        // per z stage and position: (rstd_t / 2, rstd_z / 2)
  __shared__ unsigned tmem_base_s;
  __shared__ int abort_flag;
  unsigned char* smem = smem_raw + ((1024 - (smem_u32(smem_raw) & 1023)) & 1023);
  const int c_z = p.c_z, c_h = p.c_h;
  const int zslab = c_z / 64, hslab = c_h / 64;
  const int wo_slab = c_z * 128, wg_slab = c_z * 128;        // one 64-wide K slab of [c_z rows]
  const int wo_bytes = hslab * wo_slab, wg_bytes = zslab * wg_slab;
  const int t_chunk = c_h * 128;                             // [c_h][64 positions]
  const int z_slab = 128 * 128;                              // [128 positions][64 channels]
  const int t_stage = 2 * t_chunk, z_stage = zslab * z_slab;
  unsigned char* sWo = smem;
  unsigned char* sWg = sWo + wo_bytes;
  unsigned char* sT = sWg + wg_bytes;                        // 2 stages of the two t chunks
  unsigned char* sZ = sT + 2 * t_stage;                      // 2 stages of the z tile
  unsigned char* sAx = sZ + 2 * z_stage;                     // [2 stages][t | z][2][128][8] bf16: augmentation columns 0-7, 8-15 of the rows
  unsigned char* sBx = sAx + 4 * 4096;                       // [W_o | W_g][2][c_z][8] bf16: the same of the weights
  unsigned long long* tfullb = bars;        // [2] t chunks landed
  unsigned long long* tfree = bars + 2;     // [2] MMAs and statistics have read them
  unsigned long long* zfullb = bars + 4;    // [2] z tile landed
  unsigned long long* zfree = bars + 6;     // [2] MMAs have read it, the new z has been stored from it
  unsigned long long* tfull = bars + 8;     // [2] accumulators complete
  unsigned long long* tempty = bars + 10;   // [2]
  unsigned long long* sconv = bars + 12;    // [2] statistics published
  unsigned long long* wfull = bars + 14;
  unsigned long long* zdone = bars + 15;    // [2] the new z is in the tile

  const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;   // warp-uniform for the compiler too
  if (threadIdx.x == 0) {
    abort_flag = 0;
    for (int s = 0; s < 2; ++s) {
      mbar_init(&tfullb[s], 1);
      mbar_init(&tfree[s], 1 + 4);                   // MMA commit + the four statistics warps
      mbar_init(&zfullb[s], 1);
      mbar_init(&zfree[s], 1 + 4 + 1);               // MMA commit + the statistics warps + the store warp
      mbar_init(&tfull[s], 1);
      mbar_init(&tempty[s], TO_EPI);
      mbar_init(&zdone[s], TO_EPI);
      mbar_init(&sconv[s], 4);
    }
    mbar_init(wfull, 1);
    mbar_fence_init();
  }
  if (warp == 1) tmem_alloc(&tmem_base_s, 512);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  pdl_begin();
  for (int n = threadIdx.x; n < 2 * c_z; n += TO_THREADS) {
    const int g = n >= c_z ? 1 : 0, r = n - g * c_z;
    ln_aug_weight(sBx + g * c_z * 32 + r * 16, c_z * 16, g ? p.c01g[r] : p.c01o[r]);
  }
  fence_proxy_async_smem();
  __syncthreads();
  const unsigned tmem_base = __shfl_sync(0xffffffffu, tmem_base_s, 0);
  AbortCtx ab{p.status, &abort_flag};
  const long long nchunks = p.chunk_off[p.B];
  const long long ntiles = (nchunks + 1) / 2;

  if (warp == 0) {
    // ------------------------------------------------------------------ producer (lane q decodes and loads chunk q)
    if (lane == 0) {
      mbar_expect_tx(wfull, wo_bytes + wg_bytes);
      for (int sl = 0; sl < hslab; ++sl) tma_load_2d(sWo + sl * wo_slab, &p.womap, wfull, sl * 64, 0);
      for (int sl = 0; sl < zslab; ++sl) tma_load_2d(sWg + sl * wg_slab, &p.wgmap, wfull, sl * 64, 0);
    }
    int stage = 0;
    unsigned phase = 0;
    for (long long t = blockIdx.x; t < ntiles; t += gridDim.x) {
      int s = 0, i = 0, j0 = 0;
      const bool valid = lane < 2 && to_decode(p, 2 * t + lane, s, i, j0);
      const int nvalid = (2 * t + 1 < nchunks) ? 2 : 1;
      if (lane == 0) {
        mbar_wait(&tfree[stage], phase ^ 1, ab);
        mbar_expect_tx(&tfullb[stage], nvalid * t_chunk);
      }
      __syncwarp();
      if (valid) tma_load_4d(sT + stage * t_stage + lane * t_chunk, &p.tmap[s], &tfullb[stage], j0, i, 0, 0);
      if (lane == 0) {
        mbar_wait(&zfree[stage], phase ^ 1, ab);
        mbar_expect_tx(&zfullb[stage], nvalid * zslab * 64 * 128);
      }
      __syncwarp();
      if (valid)
        for (int sl = 0; sl < zslab; ++sl)
          for (int sub = 0; sub < 2; ++sub)      // 32-position boxes (the size the epilogue warps store)
            tma_load_4d(sZ + stage * z_stage + sl * z_slab + (lane * 64 + sub * 32) * 128, &p.zmap[s], &zfullb[stage], sl * 64,
                        j0 + sub * 32, i, 0);
      if (++stage == 2) { stage = 0; phase ^= 1; }
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------------ MMA issuer (whole warp, one elected lane issues)
    mbar_wait(wfull, 0, ab);
    int stage = 0;
    unsigned phase = 0, tph0 = 0, tph1 = 0;
    unsigned n = 0;
    const unsigned idesc_t = idesc_f16(128, c_z, 1, 0, FMT_F16, FMT_F16);     // A = t (fp16, MN-major), W_o' fp16
    const unsigned idesc_z = idesc_f16(128, c_z, 0, 0, FMT_BF16, FMT_BF16);   // A = the bf16 z tile, W_g' bf16
    const unsigned long long wo_desc = desc_kmajor_sw128(smem_u32(sWo)), wg_desc = desc_kmajor_sw128(smem_u32(sWg));
    const unsigned long long bxo_desc = desc_kmajor_nosw(smem_u32(sBx), c_z * 16, 128);
    const unsigned long long bxg_desc = desc_kmajor_nosw(smem_u32(sBx + c_z * 32), c_z * 16, 128);
    const unsigned wo16 = (unsigned)wo_slab >> 4, wg16 = (unsigned)wg_slab >> 4, z16 = (unsigned)z_slab >> 4;
    for (long long t = blockIdx.x; t < ntiles; t += gridDim.x, ++n) {
      const unsigned buf = n & 1;
      if (buf == 0) { mbar_wait(&tempty[0], tph0 ^ 1, ab); tph0 ^= 1; }
      else { mbar_wait(&tempty[1], tph1 ^ 1, ab); tph1 ^= 1; }
      const unsigned d1 = tmem_base + buf * 256, d2 = d1 + c_z;
      mbar_wait(&tfullb[stage], phase, ab);
      tc_fence_after();
      const unsigned long long t_desc = desc_mnmajor_sw128(smem_u32(sT + stage * t_stage), t_chunk, 1024);
#pragma unroll
      for (int ks = 0; ks < 8; ++ks)                       // K = channels of t, 16 per step (2048 bytes of the MN-major tile)
        if (ks < c_h / 16 && elect_one())
          umma_bf16(d1, t_desc + ks * 128, wo_desc + ((ks >> 2) * wo16 + (ks & 3) * 2), idesc_t, ks != 0);
      if (elect_one()) tc_commit(&tfree[stage]);
      __syncwarp();
      mbar_wait(&zfullb[stage], phase, ab);
      tc_fence_after();
      const unsigned long long z_desc = desc_kmajor_sw128(smem_u32(sZ + stage * z_stage));
#pragma unroll
      for (int sl = 0; sl < 2; ++sl)
        if (sl < zslab) umma_k4(d2, z_desc + sl * z16, wg_desc + sl * wg16, idesc_z, sl);
      mbar_wait(&sconv[stage], phase, ab);                 // the rows' augmentation columns are written
      tc_fence_after();
      if (elect_one()) umma_bf16(d1, desc_kmajor_nosw(smem_u32(sAx + stage * 8192), 2048, 128), bxo_desc, idesc_z, 1);
      if (elect_one()) umma_bf16(d2, desc_kmajor_nosw(smem_u32(sAx + stage * 8192 + 4096), 2048, 128), bxg_desc, idesc_z, 1);
      if (elect_one()) {
        tc_commit(&tfull[buf]);
        tc_commit(&zfree[stage]);
      }
      __syncwarp();
      if (++stage == 2) { stage = 0; phase ^= 1; }
    }
  } else if (warp >= 2 && warp < 6) {
    // ------------------------------------------------------------------ statistics (4 warps, one position per thread)
    const int row = (warp - 2) * 32 + lane;
    const int q = row >> 6;
    int stage = 0;
    unsigned phase = 0;
    for (long long t = blockIdx.x; t < ntiles; t += gridDim.x) {
      // this row's chunk: scale of eps for t, and the z statistics the input projection left (requested early)
      float eps_t = p.eps;
      float2 zst = make_float2(0.f, 1.f);
      {
        int s_, i_, j_;
        if (to_decode(p, 2 * t + q, s_, i_, j_)) {
          eps_t = p.eps / ((float)p.N[s_] * (float)p.N[s_]);
          const int j = j_ + (row & 63);
          if (p.zstats && j < p.N[s_]) zst = *(p.zstats + p.pos_off[s_] + (long long)i_ * p.N[s_] + j);
        }
      }
      mbar_wait(&tfullb[stage], phase, ab);
      // Statistics of t over channels (columns of the MN-major fp16 tile).  Eight lanes share a group of eight
      // positions: lane cg sums channels cg, cg + 8, ... with 16-byte loads (8 positions each), then a
      // reduce-scatter over the eight lanes leaves every lane with the two sums of one position -- its own row.
      float ts, tq;
      {
        const int cg = lane & 7, pgl = ((warp - 2) * 4 + (lane >> 3)) & 7;      // position group inside the 64-position chunk
        float2 a2[4] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f), make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
        float2 q2[4] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f), make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
        const unsigned char* tb = sT + stage * t_stage + q * t_chunk + cg * 128 + ((pgl ^ cg) << 4);   // channel c = cc * 8 + cg: c & 7 = cg
#pragma unroll 4
        for (int cc = 0; cc < c_h / 8; ++cc) {
          const uint4 v = *reinterpret_cast<const uint4*>(tb + cc * 1024);
          const unsigned w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            const float2 f = unpack_h2(w[e]);
            a2[e] = __fadd2_rn(a2[e], f);
            q2[e] = __ffma2_rn(f, f, q2[e]);
          }
        }
        float a8[8] = {a2[0].x, a2[0].y, a2[1].x, a2[1].y, a2[2].x, a2[2].y, a2[3].x, a2[3].y};
        float q8[8] = {q2[0].x, q2[0].y, q2[1].x, q2[1].y, q2[2].x, q2[2].y, q2[3].x, q2[3].y};
        // reduce-scatter: after the step with lane bit b, a lane keeps the half of the positions whose bit b equals its own
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const bool up = cg & 4;
          const float sa = up ? a8[e] : a8[e + 4], sq_ = up ? q8[e] : q8[e + 4];
          const float ka = up ? a8[e + 4] : a8[e], kq = up ? q8[e + 4] : q8[e];
          a8[e] = ka + __shfl_xor_sync(0xffffffffu, sa, 4);
          q8[e] = kq + __shfl_xor_sync(0xffffffffu, sq_, 4);
        }
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          const bool up = cg & 2;
          const float sa = up ? a8[e] : a8[e + 2], sq_ = up ? q8[e] : q8[e + 2];
          const float ka = up ? a8[e + 2] : a8[e], kq = up ? q8[e + 2] : q8[e];
          a8[e] = ka + __shfl_xor_sync(0xffffffffu, sa, 2);
          q8[e] = kq + __shfl_xor_sync(0xffffffffu, sq_, 2);
        }
        {
          const bool up = cg & 1;
          const float sa = up ? a8[0] : a8[1], sq_ = up ? q8[0] : q8[1];
          const float ka = up ? a8[1] : a8[0], kq = up ? q8[1] : q8[0];
          ts = ka + __shfl_xor_sync(0xffffffffu, sa, 1);
          tq = kq + __shfl_xor_sync(0xffffffffu, sq_, 1);
        }
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(&tfree[stage]);
      // t arrives scaled by 1 / N_s (see the contraction); LayerNorm is scale-free once eps is scaled alike
      const float tmean = ts / (float)c_h;
      const float trstd = rsqrtf(fmaxf(tq / (float)c_h - tmean * tmean, 0.f) + eps_t);
      // z row: statistics of the bf16 tile (read only)
      mbar_wait(&zfullb[stage], phase, ab);
      float zs = 0.f, zq = 0.f;
      if (!p.zstats) {
        float s4[4] = {0.f, 0.f, 0.f, 0.f}, q4[4] = {0.f, 0.f, 0.f, 0.f};
        const unsigned char* zt = sZ + stage * z_stage;
        for (int g8 = 0; g8 < c_z / 8; ++g8) {
          const uint4 v = *reinterpret_cast<const uint4*>(zt + (g8 >> 3) * z_slab + sw128_off(row, g8 & 7));
          const unsigned w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            const float lo = __uint_as_float(w[e] << 16), hi = __uint_as_float(w[e] & 0xffff0000u);
            s4[e] += lo + hi;
            q4[e] = fmaf(lo, lo, q4[e]);
            q4[e] = fmaf(hi, hi, q4[e]);
          }
        }
        zs = (s4[0] + s4[1]) + (s4[2] + s4[3]);
        zq = (q4[0] + q4[1]) + (q4[2] + q4[3]);
      }
      const float zmean = p.zstats ? zst.x : zs / (float)c_z;
      const float zrstd = p.zstats ? zst.y : rsqrtf(fmaxf(zq / (float)c_z - zmean * zmean, 0.f) + p.eps);
      // (the z tile has landed, so the MMAs that read this stage's columns for the tile before are complete)
      unsigned char* ax = sAx + stage * 8192 + row * 16;
      const float tr = ln_aug_row(ax, 2048, tmean, trstd), zr = ln_aug_row(ax + 4096, 2048, zmean, zrstd);
      sStats[stage][row] = make_float2(0.5f * tr, 0.5f * zr);
      fence_proxy_async_smem();
      __syncwarp();
      if (lane == 0) {
        mbar_arrive(&sconv[stage]);
        mbar_arrive(&zfree[stage]);
      }
      if (++stage == 2) { stage = 0; phase ^= 1; }
    }
  } else if (warp < TO_STORE) {
    // ------------------------------------------------------------------ epilogue (16 warps: four per TMEM lane quarter, a
    // quarter of the channels each).  With 8 warps that also stored, this stage was the kernel's period: 2560 clocks of
    // arithmetic and 1770 of waiting for the store engine per tile of 128 positions, against 4950 for the tile.
    const int quarter = warp & 3;
    const int part = (warp - 6) >> 2;
    const int row = quarter * 32 + lane;           // position inside the tile
    int stage = 0;
    unsigned phase = 0;
    for (long long t = blockIdx.x; t < ntiles; t += gridDim.x) {
      unsigned char* zrow = sZ + stage * z_stage;
      mbar_wait(&tfull[stage], phase, ab);         // accumulator buffers and z stages advance together; the MMAs waited for the statistics
      tc_fence_after();
      const float2 stt = sStats[stage][row];
      const float2 tr2 = make_float2(stt.x, stt.x), zr2 = make_float2(stt.y, stt.y);
      const unsigned taddr = tmem_base + ((unsigned)(quarter * 32) << 16) + stage * 256;
#pragma unroll 1
      for (int c0 = part * (c_z / 4); c0 < (part + 1) * (c_z / 4); c0 += 16) {
        unsigned r1[16], r2[16];
        tmem_ld16(taddr + c0, r1);
        tmem_ld16(taddr + c_z + c0, r2);
        tmem_ld_wait2(r1, r2);
        unsigned char* zp = zrow + (c0 >> 6) * z_slab;
#pragma unroll
        for (int ch = 0; ch < 2; ++ch) {
          const int chunk16 = ((c0 & 63) >> 3) + ch;
          uint4* ptr = reinterpret_cast<uint4*>(zp + sw128_off(row, chunk16));
          uint4 v = *ptr;
          unsigned w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            const int n0 = ch * 8 + e * 2;
            const float2 z2 = make_float2(__uint_as_float(w[e] << 16), __uint_as_float(w[e] & 0xffff0000u));   // the bf16 state
            const float2 oh = __fmul2_rn(tr2, make_float2(__uint_as_float(r1[n0]), __uint_as_float(r1[n0 + 1])));
            const float2 ta = __fmul2_rn(zr2, make_float2(__uint_as_float(r2[n0]), __uint_as_float(r2[n0 + 1])));
            const float2 th = make_float2(to_tanh(ta.x), to_tanh(ta.y));
            const float2 res = __fadd2_rn(__ffma2_rn(oh, th, oh), z2);
            __nv_bfloat162 hh = __floats2bfloat162_rn(res.x, res.y);
            w[e] = *reinterpret_cast<unsigned*>(&hh);
          }
          *ptr = make_uint4(w[0], w[1], w[2], w[3]);
        }
      }
      tc_fence_before();
      fence_proxy_async_smem();
      __syncwarp();
      if (lane == 0) {
        mbar_arrive(&tempty[stage]);
        mbar_arrive(&zdone[stage]);
      }
      if (++stage == 2) { stage = 0; phase ^= 1; }
    }
  } else {
    // ------------------------------------------------------------------ store: lane l takes 32 positions of a 64-channel slab
    int stage = 0;
    unsigned phase = 0;
    for (long long t = blockIdx.x; t < ntiles; t += gridDim.x) {
      const int quarter = lane & 3, sl = lane >> 2, sub = quarter & 1;
      int s, i, j0;
      const bool any = sl < zslab && to_decode(p, 2 * t + (quarter >> 1), s, i, j0) && j0 + sub * 32 < p.N[s];
      mbar_wait(&zdone[stage], phase, ab);
      if (any) tma_store_4d(&p.zmap[s], sZ + stage * z_stage + sl * z_slab + quarter * 32 * 128, sl * 64, j0 + sub * 32, i, 0);
      tma_store_commit();
      tma_store_wait_read0();
      __syncwarp();
      if (lane == 0) mbar_arrive(&zfree[stage]);
      if (++stage == 2) { stage = 0; phase ^= 1; }
    }
    tma_store_wait_all0();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  abort_linger(ab);
  if (warp == 1) tmem_dealloc(tmem_base, 512);
}

bool fast_tri_out_supported(int c_z, int c_h) { return (c_z == 64 || c_z == 128) && (c_h == 64 || c_h == 128); }

nt_status fast_tri_out(void* z, const void* t, const TriPrep& tp, float eps, int c_z, int c_h, const BatchMeta& m,
                       int* status, cudaStream_t st, const float2* zstats) {
  const void* wo = tp.wo;
  const void* wg = tp.wg;
  const float2* c01o = (const float2*)tp.c01o;
  const float2* c01g = (const float2*)tp.c01g;
  const int zslab = c_z / 64, hslab = c_h / 64;
  const size_t smem = (size_t)hslab * c_z * 128 + (size_t)zslab * c_z * 128 +
                      2 * ((size_t)2 * c_h * 128 + (size_t)zslab * 128 * 128) + 4 * 4096 + (size_t)c_z * 64 + 1024;
  // the attribute belongs to a (kernel, device) pair: one flag per device
  static bool attr_set_dev[64] = {};
  int attr_dev = 0;
  cudaGetDevice(&attr_dev);
  bool& attr_set = attr_set_dev[attr_dev & 63];
  if (!attr_set) {
    if (cudaFuncSetAttribute(tri_out_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 220 * 1024) != cudaSuccess)
      return cuda_fail("tri_out smem attribute");
    attr_set = true;
  }
  for (int g0 = 0; g0 < m.B; g0 += TO_MAXB) {
    TriOutParams p;
    memset(&p, 0, sizeof(p));
    p.B = m.B - g0 < TO_MAXB ? m.B - g0 : TO_MAXB;
    p.c_z = c_z;
    p.c_h = c_h;
    p.eps = eps;
    p.c01o = c01o;
    p.c01g = c01g;
    p.status = status;
    p.zstats = zstats;
    {
      const unsigned long long dims[2] = {(unsigned long long)c_h, (unsigned long long)c_z};
      const unsigned long long strides[1] = {(unsigned long long)c_h * 2};
      const unsigned box[2] = {64, (unsigned)c_z};
      if (!make_tmap_bf16(&p.womap, wo, 2, dims, strides, box)) return cuda_fail("tri_out W_o map");
      const unsigned long long dims2[2] = {(unsigned long long)c_z, (unsigned long long)c_z};
      const unsigned long long strides2[1] = {(unsigned long long)c_z * 2};
      if (!make_tmap_bf16(&p.wgmap, wg, 2, dims2, strides2, box)) return cuda_fail("tri_out W_g map");
    }
    p.chunk_off[0] = 0;
    for (int l = 0; l < TO_MAXB; ++l) {
      const int N = l < p.B ? m.N[g0 + l] : 0;
      p.N[l] = N;
      p.pos_off[l] = l < p.B ? m.pair_off[g0 + l] : 0;
      p.chunk_off[l + 1] = p.chunk_off[l] + (long long)N * ((N + 63) / 64);
      if (N > 0) {
        const int ld = round_up8(N);
        {
          const unsigned long long dims[4] = {(unsigned long long)c_z, (unsigned long long)N, (unsigned long long)N, 1};
          const unsigned long long strides[3] = {(unsigned long long)c_z * 2, (unsigned long long)N * c_z * 2,
                                                 (unsigned long long)N * N * c_z * 2};
          const unsigned box[4] = {64, 32, 1, 1};
          const char* base = (const char*)z + (size_t)m.pair_off[g0 + l] * c_z * 2;
          if (!make_tmap_bf16(&p.zmap[l], base, 4, dims, strides, box)) return cuda_fail("tri_out z map");
        }
        {
          const unsigned long long dims[4] = {(unsigned long long)N, (unsigned long long)N, (unsigned long long)c_h, 1};
          const unsigned long long strides[3] = {(unsigned long long)ld * 2, (unsigned long long)N * ld * 2,
                                                 (unsigned long long)c_h * N * ld * 2};
          const unsigned box[4] = {64, 1, (unsigned)c_h, 1};
          const char* base = (const char*)t + (size_t)c_h * m.cm_off[g0 + l] * 2;
          if (!make_tmap_bf16(&p.tmap[l], base, 4, dims, strides, box)) return cuda_fail("tri_out t map");
        }
      }
    }
    const long long ntiles = (p.chunk_off[p.B] + 1) / 2;
    if (ntiles == 0) continue;
    const unsigned grid = (unsigned)(ntiles < sm_count() ? ntiles : sm_count());
    {
      LaunchScope ls("tri_out", st);
      launch_kernel(tri_out_kernel, grid, TO_THREADS, smem, st, p);
    }
    if (cudaPeekAtLastError() != cudaSuccess) return cuda_fail("tri_out launch");
  }
  return NT_OK;
}

}  // namespace ntp
