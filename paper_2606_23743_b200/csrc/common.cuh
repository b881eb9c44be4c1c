// Shared host/device helpers of the sva library (CUDA side only).
#pragma once
#include <cuda_bf16.h>
#include <cuda_fp8.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <mutex>

#include "../../include/sva.h"

namespace sva {

struct Dims {
  int B, H, N, d, block, Nb, R;
  float scale;
  bool fp8;
};

inline Dims make_dims(const sva_problem_t* p) {
  Dims m;
  m.B = p->B; m.H = p->H; m.N = p->N; m.d = p->d; m.block = p->block;
  m.Nb = (p->N + p->block - 1) / p->block;
  m.R = p->B * p->H * m.Nb;
  m.scale = p->softmax_scale > 0.f ? p->softmax_scale : 1.0f / sqrtf((float)p->d);
  m.fp8 = p->qk_dtype == SVA_FP8_E4M3;
  return m;
}

struct Strides { long long b, h, n; };
inline Strides make_strides(const int64_t s[3]) { return Strides{(long long)s[0], (long long)s[1], (long long)s[2]}; }

__device__ __forceinline__ float bf16lo(uint32_t u) { return __uint_as_float(u << 16); }
__device__ __forceinline__ float bf16hi(uint32_t u) { return __uint_as_float(u & 0xffff0000u); }

// e4m3 byte -> float (exact)
__device__ __forceinline__ float e4m3_to_float(uint32_t byte) {
  __half_raw h = __nv_cvt_fp8_to_halfraw((__nv_fp8_storage_t)byte, __NV_E4M3);
  return __half2float(__half(h));
}

// two e4m3 bytes (the low 16 bits) -> two floats (exact), the low byte first
__device__ __forceinline__ float2 e4m3x2_to_float2(uint32_t pair) {
  return __half22float2(__half2(__nv_cvt_fp8x2_to_halfraw2((__nv_fp8x2_storage_t)pair, __NV_E4M3)));
}

// x / s for the e4m3 cast, s and y = RN(1/s) fixed for a whole block: q0 = x*y, one exact residual, one
// correction -- the correctly rounded quotient (Markstein's sequence) in three FMA-pipe operations instead of
// the dozen of a general division, valid while s is in [2^-60, 2^60] and its significand is not all ones
// (div_fast_ok; otherwise the caller divides).  |x| below s*2^-12 may come out one unit off, which the cast
// sends to zero all the same.  The residual is formed negated, t = q0*s - x, so that a zero x keeps its
// sign through both steps (-0 stays -0, as in a true division).
__device__ __forceinline__ bool div_fast_ok(float s) {
  return s >= 8.673617379884035e-19f && s <= 1.152921504606847e18f && (__float_as_uint(s) & 0x7fffffu) != 0x7fffffu;
}
__device__ __forceinline__ float div_fast(float x, float s, float y) {
  const float q0 = x * y;
  const float t = fmaf(q0, s, -x);
  return fmaf(-t, y, q0);
}
// two fp32 -> two e4m3 bytes (round to nearest even, saturating), first value in the low byte
__device__ __forceinline__ uint32_t e4m3x2(float lo, float hi) {
  return (uint32_t)__nv_cvt_float2_to_fp8x2(make_float2(lo, hi), __NV_SATFINITE, __NV_E4M3);
}

// Kernels of one call follow one another in a stream; each is launched so that it may be set up while its predecessor ends
// (programmatic stream serialisation), and starts with grid_dep_wait(), which returns when every earlier kernel of the
// stream has completed and its writes are visible.  It returns 0, which the compiler does not know: added to the indices that a
// kernel's first loads are made from, it keeps read-only loads from being moved in front of it.
// grid_dep_launch() lets the next kernel be set up once every CTA has called it or ended -- whatever the size of the grid, none
// of its CTAs can then be kept from an SM by one that waits for it.  The short kernels call it at their start (block scores,
// selection, CSR, tile lists, mean key, remainder weights, row counters; none of them holds tensor memory); the streaming
// ones, the tensor-core ones and the attention kernel do not, so that their successors come in when they end: called
// there too, the successors' waiting CTAs made everything from a medium clip on 0.3 to 0.9 % slower than plain launches.  As
// it is: a 5 580-token clip 95.3 -> 83.7 us for the whole call, 8 192 tokens x 16 heads 172 -> 166.5 us.
// (The diagnostic CUDA-core attention kernel is launched plainly: it starts when everything before it has ended.)
__device__ __forceinline__ int grid_dep_wait() {
  int zero;
  asm volatile("griddepcontrol.wait;\n\tmov.u32 %0, 0;" : "=r"(zero)::"memory");
  return zero;
}
__device__ __forceinline__ void grid_dep_launch() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
// (cluster: CTAs per thread-block cluster; the grid is then a multiple of it in x)
template <typename... P, typename... A>
inline int launch_dep_cluster(int cluster, void (*kern)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, A&&... args) {
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = (unsigned)cluster;
  attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cfg.attrs = attr;
  cfg.numAttrs = cluster > 1 ? 2 : 1;
  if (cudaLaunchKernelEx(&cfg, kern, static_cast<P>(args)...) == cudaSuccess) return SVA_OK;
  (void)cudaGetLastError();                    // (reported by the status; not left behind for the caller's next check)
  return SVA_ERR_CUDA;
}

template <typename... P, typename... A>
inline int launch_dep(void (*kern)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, A&&... args) {
  return launch_dep_cluster(1, kern, grid, block, smem, st, static_cast<A&&>(args)...);
}

// Function attributes of a kernel, set once per device and instantiation instead of per call.
struct DeviceOnce {
  std::mutex mutex;
  bool done[64] = {false};
  template <typename F>
  int run(F set) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return SVA_ERR_CUDA;
    std::lock_guard<std::mutex> lock(mutex);
    if (!done[dev]) {
      if (!set()) return SVA_ERR_CUDA;
      done[dev] = true;
    }
    return SVA_OK;
  }
};

// Consecutive token blocks per CTA of the kernels that stream a tensor's blocks (`blocks` of them over all heads and tensors, of
// block_bytes) with the next block's loads in flight while they reduce: runs of up to 128 KB, as long as the CTAs' first loads
// together still come to 16 MB (512 blocks of 32 KB: 3.5 CTAs per SM).  16 heads x 8 192 tokens, pooling of Q and K: one block of
// 32 KB per CTA 15.5 us, two 14.8, four 14.3; 32 heads x 4 096 tokens in blocks of 16 KB: two 15.8, four 16.1, eight 17.9;
// 24 x 32 760 in them: two 80.9, four 78.0, eight 74.3.
inline int blocks_per_cta(long long blocks, int block_bytes) {
  const long long run = blocks * block_bytes >> 24;
  const int most = (128 << 10) / block_bytes;
  return run < 1 ? 1 : run > most ? most : (int)run;
}

// host-side argument checks shared by the entry points
int validate_problem(const sva_problem_t* p);

// launchers (each returns an sva_status_t)
int launch_select(const Dims& m, const sva_problem_t* p, const sva_select_t* s, const void* q,
                  const void* k, const float* q_scale, const float* k_scale, int32_t* row_ptr,
                  int32_t* col_idx, float* block_scores, void* ws, size_t ws_bytes,
                  cudaStream_t st);
size_t select_workspace_bytes(const Dims& m, const sva_select_t* s);
int launch_pool(const Dims& m, const sva_problem_t* p, const void* q, const void* k, const float* q_scale,
                const float* k_scale, float* qbar, float* kbar, cudaStream_t st);
int launch_select_pooled(const Dims& m, const sva_problem_t* p, const sva_select_t* s, const float* qbar,
                         const float* kbar, int32_t* row_ptr, int32_t* col_idx, float* block_scores, void* ws,
                         size_t ws_bytes, cudaStream_t st);
int launch_prologue(const Dims& m, const sva_problem_t* p, const void* q, const void* k, const float* gq,
                    const float* gk, const float* cosn, const float* sinn, float eps, void* qo, void* ko,
                    float* qbar, float* kbar, void* q8, void* k8, float* qs, float* ks, cudaStream_t st);
int launch_select_noalloc(const Dims& m, const sva_problem_t* p, const sva_select_t* s,
                          const void* q, const void* k, const float* q_scale, const float* k_scale,
                          int32_t* row_ptr, int32_t* col_idx, float* block_scores, cudaStream_t st);
int select_row_cap(const Dims& m, const sva_select_t* s);
size_t smooth_workspace_bytes(const Dims& m);
int launch_quantize(const Dims& m, const sva_problem_t* p, const void* q, const void* k, void* q8,
                    void* k8, float* qs, float* ks, float* k_mean, float* lse_shift, void* ws, cudaStream_t st);
int launch_quantize4(const Dims& m, const sva_problem_t* p, const void* q, const void* k, void* q4, void* k4,
                     void* q_sf, void* k_sf, float* q_g, float* k_g, void* ws, cudaStream_t st);
int launch_token_move(bool scatter, const void* src, const int64_t ss[3], void* dst, const int64_t sd[3],
                      const int32_t* idx, int B, int H, int M, int n_full, int d, int elem_bytes,
                      int32_t* status, cudaStream_t st);
int launch_attn_simt(const Dims& m, const sva_problem_t* p, const void* q, const void* k,
                     const void* v, const float* qs, const float* ks, const int32_t* row_ptr,
                     const int32_t* col_idx, void* o, float* lse, int32_t* status, cudaStream_t st);
int launch_attn_ts(const Dims& m, const sva_problem_t* p, const void* q, const void* k, const void* v,
                   const float* q_scale, const float* k_scale, const int32_t* row_ptr, const int32_t* col_idx, void* o, float* lse, int32_t* status,
                   void* ws, size_t ws_bytes, cudaStream_t st, int remainder_order = -1,
                   const float* block_scores = nullptr);
int launch_attn_ts_fp4(const Dims& m, const sva_problem_t* p, const void* q4, const void* k4, const void* q_sf,
                       const void* k_sf, const float* q_g, const float* k_g, const void* v, const int32_t* row_ptr,
                       const int32_t* col_idx, void* o, float* lse, int32_t* status, void* ws, size_t ws_bytes,
                       cudaStream_t st);
bool attn_ts_fp4_serves(const Dims& m);
size_t attn_ts_workspace_bytes(const Dims& m);
size_t attn_ts_one_call_workspace_bytes(const Dims& m);
size_t attn_ts_remainder_workspace_bytes(const Dims& m, int order);
bool attn_ts_remainder_serves(const Dims& m);
bool attn_ts_serves(const Dims& m);    // d = 128 or 64, bf16 or e4m3 Q/K, 128- or 64-token blocks
int launch_prepare_v_ts(const Dims& m, const sva_problem_t* p, const void* v, void* ws, size_t ws_bytes,
                        cudaStream_t st);

// two fp32 lanes in one instruction (sm_100): d = a * b + c, d = a + b
__device__ __forceinline__ uint64_t pack2(float lo, float hi) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ void unpack2(uint64_t v, float& lo, float& hi) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {
  uint64_t d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}

}  // namespace sva
