// Block-scaled 4-bit quantiser for Q and K (the paper's quantisation format is NVFP4; it prints no formula).
// Per (b, h): tensor scale g = amax / (6 * 448) (1 if amax = 0).  Per token and 16 consecutive elements of the
// head dimension: sf = e4m3((amax_block / 6) / g), code = e2m1(x / (value(sf) * g)), both round-to-nearest-even
// and saturating; every scalar step is one fp32 operation rounded to nearest, so the bytes are reproducible.
//
// Output layout, chosen for the block-scaled tensor-core MMA that consumes it:
//   codes   [B*H][Nb*128 tokens][64 bytes]   two codes per byte (even element in the low nibble), rows >= N zero
//   scales  [B*H][Nb][2][32][4][4] bytes     per 128-token block and half of the head dimension (64 elements = 4
//                                            scale blocks) one 512-byte group: byte ((t % 32) * 4 + t / 32) * 4 + kb
//                                            holds the scale of token t (within the block), scale block kb -- the
//                                            order in which a 32-lane x 128-bit copy into tensor memory wants them
// Two kernels: the per-(b,h) amax (an integer atomicMax on the non-negative fp32 bit pattern), then the cast.
#include <cuda_fp4.h>

#include "common.cuh"

namespace sva {

static constexpr int Q4_THREADS = 256;

// amax[tensor * BH + bh] (as fp32 bits; the launcher zeroes it) = max |x| over the existing tokens
// From the end of the tensors, which a kernel that has just written them (the prologue) leaves in the L2.
// A CTA per 128-token block, its second half's loads in flight behind the first half's maxima, and one atomicMax.  (An atomic per
// warp, 98 304 of them on 48 words, took 100 us for 403 MB.  Runs of blocks per CTA, as pooling has them, are slower: there is no
// reduction per block to hide.
// The whole quantiser, us, inputs not in the L2, runs of four / a block per CTA: 24 heads x 32 760 tokens 155.9 / 153.5,
// 16 x 16 384 61.2 / 56.1, 16 x 8 192 33.3 / 32.8, 8 x 4 096 16.4 / 13.4; inputs in the L2, 16 x 8 192 30.4 / 28.7.)
__global__ void __launch_bounds__(Q4_THREADS)
amax_kernel(const __nv_bfloat16* __restrict__ q, const __nv_bfloat16* __restrict__ k, Strides sq, Strides sk, int H, int N,
            int BH, uint32_t* __restrict__ amax) {
  const int bh = gridDim.y - 1 - blockIdx.y + grid_dep_wait(), which = 1 - blockIdx.z;
  const Strides s = which ? sk : sq;
  const __nv_bfloat16* base = (which ? k : q) + (long long)(bh / H) * s.b + (long long)(bh % H) * s.h;
  const int lo = (gridDim.x - 1 - blockIdx.x) * 128, hi = min(lo + 128, N);
  const int row = threadIdx.x >> 4, vec = threadIdx.x & 15;   // 16 vectors of 8 elements per token, 16 tokens at a time
  uint4 u[4];
  auto load = [&](int t0) {
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const int t = t0 + 16 * r + row;
      u[r] = make_uint4(0u, 0u, 0u, 0u);
      if (t < hi) u[r] = __ldg(reinterpret_cast<const uint4*>(base + (long long)t * s.n) + vec);
    }
  };
  uint32_t m = 0u;                                            // max of the |x| bit patterns (bf16 in the upper half)
  load(lo);
  for (int t0 = lo; t0 < hi; t0 += 64) {
    uint4 c[4];
#pragma unroll
    for (int r = 0; r < 4; ++r) c[r] = u[r];
    load(t0 + 64);
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const uint32_t w[4] = {c[r].x, c[r].y, c[r].z, c[r].w};
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        m = max(m, (w[e] << 16) & 0x7fffffffu);
        m = max(m, w[e] & 0x7fff0000u);
      }
    }
  }
  __shared__ uint32_t wm[Q4_THREADS / 32];
  m = __reduce_max_sync(0xffffffffu, m);
  if ((threadIdx.x & 31) == 0) wm[threadIdx.x >> 5] = m;
  __syncthreads();
  if (threadIdx.x == 0) {
#pragma unroll
    for (int i = 1; i < Q4_THREADS / 32; ++i) m = max(m, wm[i]);
    if (m) atomicMax(amax + which * BH + bh, m);
  }
}

__device__ __noinline__ float div_slow(float a, float b) { return __fdiv_rn(a, b); }

// the larger of two bf16 pairs, lane by lane; a NaN loses against a number
__device__ __forceinline__ uint32_t max_bf16x2(uint32_t a, uint32_t b) {
  uint32_t r;
  asm("max.bf16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
  return r;
}

// One CTA per (128-token block, head, tensor), in the reverse of the order in which amax_kernel read them, so that the tensors'
// beginnings are still in the L2; a thread casts four 16-element scale blocks, whose loads are all in flight.  Issue-bound (75 % of
// the issue slots at 105 us): the divisions are three FMA-pipe operations each, element pairs in packed ones, with true
// divisions out of line for magnitudes whose residuals could underflow; scales leave through shared memory.  Q and K of
// 24 heads x 32 760 tokens (403 MB in, 113 MB out): 105 -> 85 us alone
// (in a call at the power cap 94).  Registers matter: with 72 of them, three CTAs per SM, the cast took 102 us.
__global__ void __launch_bounds__(Q4_THREADS)
quantize4_kernel(const __nv_bfloat16* __restrict__ q, const __nv_bfloat16* __restrict__ k, Strides sq, Strides sk, int H,
                 int N, int Nb, int BH, const uint32_t* __restrict__ amax, uint8_t* __restrict__ q4,
                 uint8_t* __restrict__ k4, uint8_t* __restrict__ q_sf, uint8_t* __restrict__ k_sf, float* __restrict__ q_g,
                 float* __restrict__ k_g) {
  const int I = blockIdx.x, bh = blockIdx.y + grid_dep_wait(), which = blockIdx.z;
  const Strides s = which ? sk : sq;
  const __nv_bfloat16* base = (which ? k : q) + (long long)(bh / H) * s.b + (long long)(bh % H) * s.h;
  uint8_t* codes = (which ? k4 : q4) + ((long long)bh * Nb + I) * 128 * 64;
  uint8_t* sfo = (which ? k_sf : q_sf) + ((long long)bh * Nb + I) * 1024;
  const float am = __uint_as_float(__ldg(amax + which * BH + bh));
  const float g = am > 0.f ? __fdiv_rn(am, 2688.0f) : 1.0f;
  __shared__ __align__(16) uint8_t sf_tile[1024];              // the block's scales in tile order: single bytes to the HBM are partial sectors
  const bool g_fast = div_fast_ok(g);
  const float g_rcp = __frcp_rn(g);
  if (I == 0 && threadIdx.x == 0) (which ? k_g : q_g)[bh] = g;
  const int lo = I * 128;
  constexpr int PER = 128 * 8 / Q4_THREADS;                   // scale blocks per thread, all their loads in flight
  uint4 in[PER][2];
#pragma unroll
  for (int r = 0; r < PER; ++r) {
    const int i = threadIdx.x + r * Q4_THREADS, t = i >> 3, kb = i & 7;
    in[r][0] = in[r][1] = make_uint4(0u, 0u, 0u, 0u);
    if (lo + t < N) {
      const uint4* src = reinterpret_cast<const uint4*>(base + (long long)(lo + t) * s.n + kb * 16);
      in[r][0] = __ldg(src); in[r][1] = __ldg(src + 1);
    }
  }
#pragma unroll
  for (int r = 0; r < PER; ++r) {
    const int i = threadIdx.x + r * Q4_THREADS;
    const int t = i >> 3, kb = i & 7;                         // token of the block, scale block of the token
    const uint32_t w[8] = {in[r][0].x, in[r][0].y, in[r][0].z, in[r][0].w, in[r][1].x, in[r][1].y, in[r][1].z, in[r][1].w};
    uint32_t mx = 0u;                                         // max |x| of the pairs, NaNs left out (an integer maximum would take them)
#pragma unroll
    for (int e = 0; e < 8; ++e) mx = max_bf16x2(mx, w[e] & 0x7fff7fffu);
    const float a = __uint_as_float(max(mx << 16, mx & 0xffff0000u));
    const float u = g_fast && (a == 0.f || a >= 8.077935669463161e-28f)                       // 2^-90
                        ? div_fast(div_fast(a, 6.0f, 0.16666667163372039795f), g, g_rcp)
                        : div_slow(div_slow(a, 6.0f), g);
    uint8_t sf = (uint8_t)__nv_cvt_float_to_fp8(u, __NV_SATFINITE, __NV_E4M3);
    const float sd = e4m3_to_float(sf);
    uint2 out = make_uint2(0u, 0u);
    if (sd > 0.f) {                                           // (a token beyond N is all zeros: scale and codes 0)
      const float sc = __fmul_rn(sd, g);
      uint32_t pk[2] = {0u, 0u};
      if (div_fast_ok(sc)) {
        // x / sc: the correctly rounded quotient from one reciprocal per scale block (div_fast, two elements at a time)
        const float rc = __frcp_rn(sc);
        const uint64_t sc2 = pack2(sc, sc), rc2 = pack2(rc, rc), nrc2 = pack2(-rc, -rc), one = pack2(-1.f, -1.f), nz = pack2(-0.f, -0.f);
#pragma unroll
        for (int e = 0; e < 8; ++e) {
          const uint64_t x = pack2(bf16lo(w[e]), bf16hi(w[e]));
          const uint64_t q0 = fma2(x, rc2, nz), res = fma2(q0, sc2, fma2(x, one, nz));
          float2 y;
          unpack2(fma2(res, nrc2, q0), y.x, y.y);
          pk[e >> 2] |= ((uint32_t)__nv_cvt_float2_to_fp4x2(y, __NV_E2M1, cudaRoundNearest) & 0xffu) << (8 * (e & 3));
        }
      } else {
        // (kept out of the loop's way: the unrolled divisions stalled the kernel on instruction fetch)
#pragma unroll 1
        for (int e = 0; e < 8; ++e) {
          const uint32_t we = reinterpret_cast<const uint32_t*>(base + (long long)(lo + t) * s.n + kb * 16)[e];
          const float2 y = make_float2(div_slow(bf16lo(we), sc), div_slow(bf16hi(we), sc));
          const uint32_t c = ((uint32_t)__nv_cvt_float2_to_fp4x2(y, __NV_E2M1, cudaRoundNearest) & 0xffu) << (8 * (e & 3));
          if (e < 4) pk[0] |= c; else pk[1] |= c;
        }
      }
      out = make_uint2(pk[0], pk[1]);
    } else {
      sf = 0;
    }
    *reinterpret_cast<uint2*>(codes + t * 64 + kb * 8) = out;
    sf_tile[(kb >> 2) * 512 + ((t & 31) * 4 + (t >> 5)) * 4 + (kb & 3)] = sf;
  }
  __syncthreads();
  if (threadIdx.x < 64) reinterpret_cast<uint4*>(sfo)[threadIdx.x] = reinterpret_cast<const uint4*>(sf_tile)[threadIdx.x];
}

int launch_quantize4(const Dims& m, const sva_problem_t* p, const void* q, const void* k, void* q4, void* k4,
                     void* q_sf, void* k_sf, float* q_g, float* k_g, void* ws, cudaStream_t st) {
  if (m.d != 128 || m.block != 128) return SVA_ERR_UNSUPPORTED;
  const int BH = m.B * m.H;
  uint32_t* amax = static_cast<uint32_t*>(ws);
  if (cudaMemsetAsync(amax, 0, (size_t)2 * BH * sizeof(uint32_t), st) != cudaSuccess) return SVA_ERR_CUDA;
  const Strides sq = make_strides(p->q_stride), sk = make_strides(p->k_stride);
  const int rc = launch_dep(amax_kernel, dim3(m.Nb, BH, 2), Q4_THREADS, 0, st, (const __nv_bfloat16*)q, (const __nv_bfloat16*)k, sq, sk, m.H,
                            m.N, BH, amax);
  if (rc != SVA_OK) return rc;
  return launch_dep(quantize4_kernel, dim3(m.Nb, BH, 2), Q4_THREADS, 0, st, (const __nv_bfloat16*)q, (const __nv_bfloat16*)k, sq, sk,
                    m.H, m.N, m.Nb, BH, amax, (uint8_t*)q4, (uint8_t*)k4, (uint8_t*)q_sf, (uint8_t*)k_sf, q_g, k_g);
}

}  // namespace sva
