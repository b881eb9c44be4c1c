// First-order term of the approximate remainder (the paper's "first-order Taylor" compensation of dropped
// blocks, as this build reads it): for a query block I
//     T_i = scale * A_I^T q_i,   A_I = sum_{J dropped by I} exp(sbar_IJ) C_J,   C_J = sum_{j in J} (k_j - kbar_J) v_j^T,
// one d x d matrix per query block.  Three kernels prepare A_I for the attention kernel, which then treats it as one
// more tile of the row (its "P" are the scaled query values, its "V" is A_I -- or, for the attention kernel that runs
// on a transposed copy of V, its "V^T" is A_I^T; the kernels below are written for the transposed form and produce
// the other one when the launcher hands the covariance kernel K and V in each other's place):
//   cov_kernel        C_J^T = V_J^T K_J - n_J vbar_J kbar_J^T per key block: one 128 x 128 x block tcgen05 MMA, both
//                     operands read where they lie (MN-major), the rank-one centring in the epilogue; bf16 out
//   weights_kernel    W[I][J] = exp(sbar_IJ - mu_I) for the dropped J (0 for the kept ones), mu_I = their maximum
//   aggregate_kernel  A_I^T = sum_J W[I][J] C_J^T: per head a [Nb x Nb] x [Nb x d*d] GEMM on tcgen05
// All waits are bounded (tc_ptx.cuh); a wait that runs out sets SVA_DEV_TIMEOUT and the CTA leaves.
#include "tc_ptx.cuh"

namespace sva {

static __device__ __forceinline__ bool wait_or_report(uint32_t bar, uint32_t parity, volatile int* abort_flag, int32_t* status) {
  if (mbar_wait(bar, parity, abort_flag)) return true;
  if (status) atomicOr(status, SVA_DEV_TIMEOUT);
  return false;
}

// A wait has run out: copies and MMAs still in flight get time to land before shared memory and TMEM go away.
static __device__ __noinline__ void settle() {
  const long long t0 = clock64();
  while (clock64() - t0 < 2000000LL) __nanosleep(1000);
}

namespace rem {
constexpr int D = 128;
constexpr int TILE = BS * D * 2;                  // 32 KB: 128 rows x 256 bytes as two 128-byte panels
}

// 32 finished values of a thread's row (columns c0 .. c0+31 of 128, c0 a multiple of 32) as bf16 into a staging tile: 128 rows as two
// 128-byte panels, 128-byte swizzle, which two TMA stores then write out.  (A bulk copy of 256 bytes per row, 128 per tile, keeps the
// copy engine busy for some 3 000 cycles; 16-byte stores from registers touch 32 rows per instruction, half a sector at a time.)
static __device__ __forceinline__ void stage_row(uint8_t* tile, int row, int c0, const uint32_t (&o)[16]) {
  uint8_t* p = tile + (c0 >> 6) * (rem::TILE / 2) + row * 128;
#pragma unroll
  for (int e = 0; e < 4; ++e)
    *reinterpret_cast<uint4*>(p + (((((c0 & 63) >> 3) + e) ^ (row & 7)) << 4)) = make_uint4(o[4 * e], o[4 * e + 1], o[4 * e + 2], o[4 * e + 3]);
}

// ------------------------------------------------------------------ C_J^T
// grid (Nb, B*H), 128 threads.  Shared memory: K tile, V tile ([keys][d] as two 64-element panels, 128-byte swizzle).
// Bound by the CTA's latency (three per SM): the MMA runs beside the column sums, which read 16 bytes at a time, and the finished
// matrix leaves as two TMA stores.  20 heads x 138 blocks: 73 -> 61 us (sums of a column per thread, 2 bytes at a time, and 16-byte
// stores of 32 rows per warp before), and the block means with it.
// mean_k, mean_v (of the tensors behind tm_k and tm_v; both or neither): the block means that the attention kernel's block-mean tiles read,
// [B*H][Nbp][128] bf16, rows >= Nb zero.  They are at hand here: without the pass that makes them from K and V again
// (pool_kv_kernel) a call on the same 20 x 138 blocks is 46 to 53 us shorter.  (fp32 both, but in eight partial sums per column
// where that kernel has sixteen: a mean whose sums are not exact in fp32 can round to the neighbouring bf16 value.)
__global__ void __launch_bounds__(128)
cov_kernel(const __grid_constant__ CUtensorMap tm_k, const __grid_constant__ CUtensorMap tm_v, const __grid_constant__ CUtensorMap tm_ct,
           int H, int N, int block, int Nb, __nv_bfloat16* __restrict__ mean_k, __nv_bfloat16* __restrict__ mean_v, int Nbp,
           int32_t* __restrict__ row_counter, int debug, int32_t* __restrict__ status) {
  using namespace rem;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  const uint32_t sbase = smem_u32(smem);
  __shared__ __align__(8) unsigned long long bars[2];
  __shared__ uint32_t tmem_base_s;
  __shared__ int abort_s;
  __shared__ float part[8][D], kb_s[D], vb_s[D];
  volatile int* abort_flag = &abort_s;
  const uint32_t bar_full = smem_u32(&bars[0]), bar_mma = smem_u32(&bars[1]);
  const int J = blockIdx.x, bh = blockIdx.y, hh = bh % H, bb = bh / H;
  const int warp = threadIdx.x >> 5;
  const int cnt = min(block, N - J * block);
  const uint32_t panel = (uint32_t)block * 128u;             // bytes of one 64-element panel of the tile
  if (threadIdx.x == 0) {
    mbar_init(bar_full, 1);
    mbar_init(bar_mma, 1);
    abort_s = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base_s)), "r"(128u) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = tmem_base_s;
  grid_dep_wait();
  if (mean_k) {
    if (J == 0 && bh == 0 && threadIdx.x < 2) row_counter[threadIdx.x] = 0;        // the attention kernel draws its rows from it
    if (J == Nb - 1) {
      for (int r = Nb; r < Nbp; ++r) {
        const long long at = ((long long)bh * Nbp + r) * D + threadIdx.x;
        mean_k[at] = mean_v[at] = __float2bfloat16_rn(0.f);
      }
    }
  }
  if (threadIdx.x == 0) {
    mbar_expect_tx(bar_full, 4u * panel);
    tma_load_4d(sbase, &tm_k, bar_full, 0, J * block, hh, bb);
    tma_load_4d(sbase + panel, &tm_k, bar_full, 64, J * block, hh, bb);
    tma_load_4d(sbase + TILE, &tm_v, bar_full, 0, J * block, hh, bb);
    if (!(debug & 256)) tma_load_4d(sbase + TILE + panel, &tm_v, bar_full, 64, J * block, hh, bb);      // (test aid: the wait runs out)
  }
  bool ok = wait_or_report(bar_full, 0u, abort_flag, status);
  ok = __syncthreads_and(ok);                                   // (every thread or none goes on: there are barriers below)
  if (ok) {
    if (threadIdx.x == 0) {
      // D[e][c] = sum_j V[j][e] K[j][c]: A = V^T and B = K^T, both MN-major from the tiles as they lie
      tc_fence_after();
      const uint32_t idesc = instr_desc(128, 128, 1, true) | (1u << 15);
      const uint64_t ad = smem_desc(sbase + TILE, panel, 1024), bd = smem_desc(sbase, panel, 1024);
      for (int kk = 0; kk < block / 16; ++kk)
        tc_mma_ss_bf16(tmem_base, ad + (uint64_t)(kk * 128), bd + (uint64_t)(kk * 128), idesc, kk > 0 ? 1u : 0u);
      tc_commit(bar_mma, 1u);
    }
    // column means of the two tiles (rows beyond N arrive as zeros): a thread adds 8 columns of every eighth row, 16 bytes at a time,
    // then the eight partial sums of a column in order
    const int vec = threadIdx.x & 15, grp = threadIdx.x >> 4;
    for (int which = 0; which < 2; ++which) {
      const uint8_t* tp = smem + which * TILE + (vec >> 3) * panel;
      float acc[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
#pragma unroll 4
      for (int j = grp; j < block; j += 8) {                    // (row j % 8 = grp: one swizzle pattern per thread)
        const uint4 u = *reinterpret_cast<const uint4*>(tp + j * 128 + (((vec & 7) ^ grp) << 4));
        const uint32_t wd[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
        for (int e = 0; e < 4; ++e) { acc[2 * e] += bf16lo(wd[e]); acc[2 * e + 1] += bf16hi(wd[e]); }
      }
#pragma unroll
      for (int e = 0; e < 8; ++e) part[grp][vec * 8 + e] = acc[e];
      __syncthreads();
      float sum = 0.f;
#pragma unroll
      for (int g = 0; g < 8; ++g) sum += part[g][threadIdx.x];
      const float mean = sum / (float)cnt;
      (which ? vb_s : kb_s)[threadIdx.x] = mean;
      if (mean_k) (which ? mean_v : mean_k)[((long long)bh * Nbp + J) * D + threadIdx.x] = __float2bfloat16_rn(mean);
      __syncthreads();
    }
  }
  __syncthreads();
  ok = ok && wait_or_report(bar_mma, 0u, abort_flag, status);
  if (ok) {
    tc_fence_after();
    const int e = threadIdx.x;                                // TMEM lane = row e of C_J^T
    const float nv = (float)cnt * vb_s[e];
    const uint32_t lane_addr = tmem_base + ((uint32_t)(warp * 32) << 16);
#pragma unroll 1
    for (int c0 = 0; c0 < D; c0 += 32) {
      uint32_t v[32];
      tmem_ld32(lane_addr + c0, v);
      tc_wait_ld();
      uint32_t o[16];
#pragma unroll
      for (int t = 0; t < 32; t += 2)
        o[t >> 1] = pack_bf16(__uint_as_float(v[t]) - nv * kb_s[c0 + t], __uint_as_float(v[t + 1]) - nv * kb_s[c0 + t + 1]);
      stage_row(smem, e, c0, o);                              // (the MMA has read the tiles)
    }
    fence_async_smem();
  }
  ok = __syncthreads_and(ok);
  if (ok && threadIdx.x == 0) {
    tma_store_3d(&tm_ct, sbase, 0, J * D, bh);
    tma_store_3d(&tm_ct, sbase + TILE / 2, 64, J * D, bh);
    bulk_commit();
    bulk_wait0();
  }
  if (abort_s) settle();
  tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(128u) : "memory");
  }
}

// ------------------------------------------------------------------ W and mu
// (20 heads x 138 blocks, 22 kept: 14 -> 5.8 us with the kept blocks as a bit mask; every block was compared with every entry before.)
// One warp per CSR row: W[r][J] (bf16, Nbw columns, zero beyond Nb and for kept J), mu[r].
__global__ void __launch_bounds__(256)
weights_kernel(const float* __restrict__ scores, const int32_t* __restrict__ row_ptr, const int32_t* __restrict__ col_idx,
               int R, int Nb, int Nbw, __nv_bfloat16* __restrict__ w, float* __restrict__ mu) {
  __shared__ uint32_t bm_s[8][32];
  const int lane = threadIdx.x & 31;
  uint32_t* bm = bm_s[threadIdx.x >> 5];
  grid_dep_launch();
  const int zero = grid_dep_wait(), r = blockIdx.x * 8 + (threadIdx.x >> 5) + zero;
  if (r >= R) return;
  const float* srow = scores + (long long)r * Nb;
  const int nnz = __ldg(row_ptr + R + zero);
  int cb = __ldg(row_ptr + r), ce = __ldg(row_ptr + r + 1);
  if (cb < 0 || ce < cb || ce - cb > Nb || ce > nnz) ce = cb;          // corrupt pair: treated as keeping nothing
  // the kept blocks of the row as a bit mask, 1024 blocks at a time
  auto mark = [&](int base) {
    bm[lane] = 0u;
    __syncwarp();
    for (int t = cb + lane; t < ce; t += 32) {
      const int J = __ldg(col_idx + t);
      if (J >= base && J - base < 1024) atomicOr(&bm[(J - base) >> 5], 1u << (J & 31));
    }
    __syncwarp();
  };
  // first pass: the maximum over the dropped blocks
  float mx = -INFINITY;
  for (int base = 0; base < Nb; base += 1024) {
    mark(base);
    for (int J0 = base; J0 < min(Nb, base + 1024); J0 += 32) {
      const int J = J0 + lane;
      const float s = J < Nb ? __ldg(srow + J) : -INFINITY;
      if (!(bm[(J0 - base) >> 5] >> lane & 1u)) mx = fmaxf(mx, s);
    }
    __syncwarp();
  }
#pragma unroll
  for (int o = 16; o; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  const bool none = mx == -INFINITY;                                      // nothing dropped
  for (int base = 0; base < Nbw; base += 1024) {
    if (Nb > 1024) mark(base);
    for (int J0 = base; J0 < min(Nbw, base + 1024); J0 += 32) {
      const int J = J0 + lane;
      const bool kept = J >= Nb || (bm[(J0 - base) >> 5] >> lane & 1u);
      float x = 0.f;
      if (!kept && !none) x = __expf(__ldg(srow + J) - mx);
      if (J < Nbw) w[(long long)r * Nbw + J] = __float2bfloat16_rn(x);
    }
    __syncwarp();
  }
  // (nothing dropped: -inf, so that the first-order tile's factor exp(mu - m) is 0 for every reference m, also one far below 0)
  if (lane == 0) mu[r] = mx;
}

// ------------------------------------------------------------------ A_I^T = sum_J W[I][J] C_J^T
// Columns: the flattened (e, c) index, in 128 n-tiles of 128.  A operand: W tile [128 I][64 J] K-major; B operand: C^T rows [64 J][128 n]
// as two 64-element panels, MN-major.  A CTA keeps the W tiles of one or two I-tiles in shared memory and walks through a run of
// n-tiles, the C^T chunks in a ring, two accumulators per I-tile so that one is read while the next is made.
// What bounds it is the way from the L2: with W fetched again for every n-tile (a CTA per tile) that was 490 MB for 90 MB read and
// 90 MB written (20 heads x 138 blocks), 79 us inside the attention call; now 51 (16 heads x 64 blocks: 18.3 -> 16.7).
// grid (runs, groups of I-tiles, B*H), 192 threads: warps 0-3 read the accumulators and write A^T, one lane of warp 4 loads, one of
// warp 5 issues the MMAs.
namespace agg {
constexpr uint32_t A_BYTES = 128 * 128, B_PANEL = 64 * 128;           // 16 KB W tile; two 8 KB panels of C^T rows
constexpr int MAX_STAGES = 6, OUT_STAGE = rem::TILE;
struct Plan { int tiles, resident, stages, smem; };                    // I-tiles per CTA; is W kept; ring stages
// Two I-tiles up to 256 blocks (128 KB of W), one up to 512; beyond that W comes through the ring with its chunk.
inline Plan plan(int Nb, int chunks) {
  Plan p;
  p.tiles = Nb > 128 && chunks <= 4 ? 2 : 1;
  p.resident = chunks <= 8 ? 1 : 0;
  const int w = p.resident ? p.tiles * chunks * (int)A_BYTES : 0, stage = (int)(p.resident ? 2 * B_PANEL : 2 * B_PANEL + A_BYTES);
  p.stages = (225 * 1024 - w - OUT_STAGE) / stage;
  if (p.stages > MAX_STAGES) p.stages = MAX_STAGES;
  p.smem = 1024 + w + p.stages * stage + OUT_STAGE;
  return p;
}
// Runs of n-tiles per group of I-tiles: the number that gives the shortest longest SM of the B200's 148 (a run costs about two
// n-tiles to begin), up to an n-tile each: one or two groups -- a call of one or two heads -- would leave most SMs idle otherwise.
// The whole call, us, at most 32 runs / so: 1 head x 4 blocks of 128 24.3 / 22.4, x 64 28.0 / 25.6, x 129 42.2 / 37.1, x 256
// 77.9 / 70.0, 2 heads x 64 29.7 / 28.3, 3 x 64 38.9 / 38.2.
inline int runs(int groups) {
  int best = 1, cost = 1 << 30;
  for (int r = 1; r <= rem::D; ++r) {
    const int c = (groups * r + 147) / 148 * ((rem::D + r - 1) / r + 2);
    if (c < cost) { cost = c; best = r; }
  }
  return best;
}
}
// barrier of the four epilogue warps, and whether all of them may go on
static __device__ __forceinline__ bool epilogue_all(bool ok) {
  uint32_t r;
  asm volatile("{\n.reg .pred p, q;\nsetp.ne.b32 p, %1, 0;\nbarrier.cta.red.and.pred q, 1, 128, p;\nselp.u32 %0, 1, 0, q;\n}"
               : "=r"(r) : "r"((uint32_t)ok) : "memory");
  return r != 0u;
}
__global__ void __launch_bounds__(192, 1)
aggregate_kernel(const __grid_constant__ CUtensorMap tm_w, const __grid_constant__ CUtensorMap tm_c, const __grid_constant__ CUtensorMap tm_at,
                 int Nb, int chunks, int tiles_per_cta, int resident, int stages, int debug, int32_t* __restrict__ status) {
  using namespace rem;
  using namespace agg;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  __shared__ __align__(8) unsigned long long bars[2 * MAX_STAGES + 5];
  __shared__ uint32_t tmem_base_s;
  __shared__ int abort_s;
  volatile int* abort_flag = &abort_s;
  const uint32_t bar_full = smem_u32(&bars[0]), bar_empty = smem_u32(&bars[MAX_STAGES]), bar_w = smem_u32(&bars[2 * MAX_STAGES]),
                 bar_acc = bar_w + 8, bar_acc_free = bar_w + 24;
  const uint32_t w_area = smem_u32(smem), stage_bytes = resident ? 2 * B_PANEL : 2 * B_PANEL + A_BYTES;
  const uint32_t ring = w_area + (resident ? tiles_per_cta * chunks * A_BYTES : 0u);
  uint8_t* out_stage = smem + (ring - w_area) + stages * stage_bytes;
  const int bh = blockIdx.z, it0 = tiles_per_cta * blockIdx.y, tiles = min(tiles_per_cta, (Nb + 127) / 128 - it0);
  const int per = (D + (int)gridDim.x - 1) / (int)gridDim.x, nt0 = blockIdx.x * per, nt1 = min(nt0 + per, D);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t cols = tiles_per_cta == 2 ? 512u : 256u;               // two accumulators of 128 columns per I-tile
  if (threadIdx.x == 0) {
    for (int b = 0; b < MAX_STAGES; ++b) { mbar_init(bar_full + 8 * b, 1); mbar_init(bar_empty + 8 * b, 1); }
    mbar_init(bar_w, 1);
    for (int b = 0; b < 2; ++b) { mbar_init(bar_acc + 8 * b, 1); mbar_init(bar_acc_free + 8 * b, 128); }
    abort_s = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base_s)), "r"(cols) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = tmem_base_s;
  grid_dep_wait();
  bool ok = true;
  if (warp == 4) {
    if (lane == 0) {
      if (resident) {
        mbar_expect_tx(bar_w, tiles * chunks * A_BYTES);
        for (int ch = 0; ch < chunks; ++ch)
          for (int t = 0; t < tiles; ++t) tma_load_3d(w_area + (ch * tiles_per_cta + t) * A_BYTES, &tm_w, bar_w, ch * 64, (it0 + t) * 128, bh);
      }
      int st = 0;
      uint32_t ph = 0;
      for (int nt = nt0; nt < nt1 && ok; ++nt) {
        if ((debug & 512) && nt > nt0) break;                              // test aid: starve the ring so that waits run out
        for (int ch = 0; ch < chunks; ++ch) {
          ok = wait_or_report(bar_empty + 8 * st, ph ^ 1u, abort_flag, status);
          if (!ok) break;
          const uint32_t dst = ring + st * stage_bytes, bar = bar_full + 8 * st;
          mbar_expect_tx(bar, stage_bytes);
          tma_load_3d(dst, &tm_c, bar, nt * 128, ch * 64, bh);
          tma_load_3d(dst + B_PANEL, &tm_c, bar, nt * 128 + 64, ch * 64, bh);
          if (!resident) tma_load_3d(dst + 2 * B_PANEL, &tm_w, bar, ch * 64, it0 * 128, bh);
          if (++st == stages) { st = 0; ph ^= 1u; }
        }
      }
    }
  } else if (warp == 5) {
    if (lane == 0) {
      const uint32_t idesc = instr_desc(128, 128, 1, true);
      int st = 0;
      uint32_t ph = 0;
      if (resident) ok = wait_or_report(bar_w, 0u, abort_flag, status);
      for (int i = 0; i < nt1 - nt0 && ok; ++i) {
        const uint32_t acc = tmem_base + (i & 1) * tiles_per_cta * 128;
        if (i >= 2) ok = wait_or_report(bar_acc_free + 8 * (i & 1), (uint32_t)(i / 2 - 1) & 1u, abort_flag, status);
        for (int ch = 0; ch < chunks && ok; ++ch) {
          ok = wait_or_report(bar_full + 8 * st, ph, abort_flag, status);
          if (!ok) break;
          tc_fence_after();
          const uint32_t src = ring + st * stage_bytes;
          const uint64_t bd = smem_desc(src, B_PANEL, 1024);
          for (int t = 0; t < tiles; ++t) {
            const uint64_t ad = smem_desc(resident ? w_area + (ch * tiles_per_cta + t) * A_BYTES : src + 2 * B_PANEL, 16, 1024);
            for (int kk = 0; kk < 4; ++kk)                                 // 16 J per instruction
              tc_mma_ss_bf16(acc + 128 * t, ad + (uint64_t)(kk * 2), bd + (uint64_t)(kk * 128), idesc, (ch > 0 || kk > 0) ? 1u : 0u);
          }
          tc_commit(bar_empty + 8 * st, 1u);
          if (++st == stages) { st = 0; ph ^= 1u; }
        }
        if (ok) tc_commit(bar_acc + 8 * (i & 1), 1u);
      }
    }
  } else {
    for (int i = 0; i < nt1 - nt0; ++i) {
      ok = wait_or_report(bar_acc + 8 * (i & 1), (uint32_t)(i / 2) & 1u, abort_flag, status);
      if (!(ok = epilogue_all(ok))) break;
      tc_fence_after();
      for (int t = 0; t < tiles; ++t) {
        if (threadIdx.x == 0) bulk_wait_read0();             // the tile staged before has been read
        epilogue_all(true);
        if ((it0 + t) * 128 + warp * 32 < Nb) {              // (a row of this warp exists; TMEM lane = query block of the tile)
          const uint32_t lane_addr = tmem_base + ((i & 1) * tiles_per_cta + t) * 128 + ((uint32_t)(warp * 32) << 16);
#pragma unroll 1
          for (int c0 = 0; c0 < 128; c0 += 32) {
            uint32_t v[32];
            tmem_ld32(lane_addr + c0, v);
            tc_wait_ld();
            uint32_t o[16];
#pragma unroll
            for (int e = 0; e < 32; e += 2) o[e >> 1] = pack_bf16(__uint_as_float(v[e]), __uint_as_float(v[e + 1]));
            stage_row(out_stage, threadIdx.x, c0, o);
          }
        }
        if (t == tiles - 1) {
          tc_fence_before();
          mbar_arrive(bar_acc_free + 8 * (i & 1));
        }
        fence_async_smem();
        epilogue_all(true);
        if (threadIdx.x == 0) {                              // (rows beyond Nb are clipped by the map)
          tma_store_3d(&tm_at, smem_u32(out_stage), (nt0 + i) * 128, (it0 + t) * 128, bh);
          tma_store_3d(&tm_at, smem_u32(out_stage) + TILE / 2, (nt0 + i) * 128 + 64, (it0 + t) * 128, bh);
          bulk_commit();
        }
      }
    }
    if (threadIdx.x == 0) bulk_wait0();                      // (shared memory goes away after this)
  }
  __syncthreads();
  if (abort_s) settle();
  tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(cols) : "memory");
  }
}

// ------------------------------------------------------------------ host side
typedef CUresult (*rem_encode_fn_t)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                    const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                    CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
static rem_encode_fn_t rem_encode() {
  static rem_encode_fn_t fn = nullptr;
  if (!fn) {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult qres;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &qres) != cudaSuccess ||
        qres != cudaDriverEntryPointSuccess)
      return nullptr;
    fn = reinterpret_cast<rem_encode_fn_t>(p);
  }
  return fn;
}
// bf16 map of `rank` dimensions (byte strides for dimensions 1..), box = 64 elements (128 bytes) x box_rows, 128-byte swizzle
static int rem_map(CUtensorMap* map, const void* ptr, int rank, const cuuint64_t* dims, const cuuint64_t* strides, int box_rows) {
  rem_encode_fn_t enc = rem_encode();
  if (!enc) return SVA_ERR_CUDA;
  cuuint64_t st[3] = {0, 0, 0};
  for (int i = 0; i < rank - 1; ++i) {
    st[i] = strides[i];
    if (dims[i + 1] == 1 && i > 0) st[i] = st[i - 1] * dims[i];      // a size-1 dimension may carry any stride: give it a legal one
    if (st[i] % 16 != 0 || st[i] == 0) return SVA_ERR_ALIGNMENT;
  }
  cuuint32_t box[4] = {64, (cuuint32_t)box_rows, 1, 1};
  cuuint32_t estr[4] = {1, 1, 1, 1};
  return enc(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, (cuuint32_t)rank, const_cast<void*>(ptr), dims, st, box, estr,
             CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
             CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS ? SVA_OK : SVA_ERR_CUDA;
}

// Bytes of the four buffers: C^T [B*H*Nb][128][128] bf16, A^T the same, W [R][Nbw] bf16, mu [R] fp32 (each 256-aligned).
static size_t al256(size_t x) { return (x + 255) & ~(size_t)255; }
size_t remainder1_bytes(const Dims& m) {
  const size_t mats = al256((size_t)m.R * rem::D * rem::D * 2);
  const int Nbw = (m.Nb + 63) / 64 * 64;
  return 2 * mats + al256((size_t)m.R * Nbw * 2) + al256((size_t)m.R * 4);
}

static int g_debug_rem = 0;
void rem_set_debug_mode(int v) { g_debug_rem = v; }
int rem_set_wait_limit(long long cycles) { return set_wait_limit(cycles); }

// Fills `buf` (remainder1_bytes) from K, V, the routing's score matrix and the CSR.  *at_out / *mu_out: where the
// attention kernel finds A_I^T ([R][128 e][128 c] bf16) and mu_I.
// natural: A_I itself ([R][128 c][128 e]) instead of its transpose -- for an attention kernel that takes its "V" tiles
// keys-major (V read where it lies): the covariance kernel then simply gets K and V in each other's place.
// k_mean, v_mean (both or neither): also the block means of K and V as rows, [B*H][Nbp][128] bf16, and the row counters at 0.
int launch_remainder1(const Dims& m, const sva_problem_t* p, const void* k, const void* v, const float* scores,
                      const int32_t* row_ptr, const int32_t* col_idx, void* buf, const __nv_bfloat16** at_out,
                      const float** mu_out, int32_t* status, cudaStream_t st, bool natural, __nv_bfloat16* k_mean, __nv_bfloat16* v_mean,
                      int Nbp, int32_t* row_counter) {
  if (m.d != rem::D || (m.block != 128 && m.block != 64)) return SVA_ERR_UNSUPPORTED;
  const size_t mats = al256((size_t)m.R * rem::D * rem::D * 2);
  const int Nbw = (m.Nb + 63) / 64 * 64;
  uint8_t* b = static_cast<uint8_t*>(buf);
  __nv_bfloat16* ct = reinterpret_cast<__nv_bfloat16*>(b);
  __nv_bfloat16* at = reinterpret_cast<__nv_bfloat16*>(b + mats);
  __nv_bfloat16* w = reinterpret_cast<__nv_bfloat16*>(b + 2 * mats);
  float* mu = reinterpret_cast<float*>(b + 2 * mats + al256((size_t)m.R * Nbw * 2));
  const Strides sk = make_strides(p->k_stride), sv = make_strides(p->v_stride);
  CUtensorMap tk, tv, tw, tc, tco, ta;
  int rc;
  {
    cuuint64_t dims[4] = {(cuuint64_t)m.d, (cuuint64_t)m.N, (cuuint64_t)m.H, (cuuint64_t)m.B};
    cuuint64_t s1[3] = {(cuuint64_t)sk.n * 2, (cuuint64_t)sk.h * 2, (cuuint64_t)sk.b * 2};
    cuuint64_t s2[3] = {(cuuint64_t)sv.n * 2, (cuuint64_t)sv.h * 2, (cuuint64_t)sv.b * 2};
    if (m.H == 1) { s1[1] = s1[0] * m.N; s2[1] = s2[0] * m.N; }
    if (m.B == 1) { s1[2] = s1[1] * m.H; s2[2] = s2[1] * m.H; }
    if ((rc = rem_map(&tk, k, 4, dims, s1, m.block)) != SVA_OK) return rc;
    if ((rc = rem_map(&tv, v, 4, dims, s2, m.block)) != SVA_OK) return rc;
  }
  {
    const int BH = m.B * m.H;
    cuuint64_t dw[3] = {(cuuint64_t)Nbw, (cuuint64_t)m.Nb, (cuuint64_t)BH};
    cuuint64_t sw[2] = {(cuuint64_t)Nbw * 2, (cuuint64_t)Nbw * 2 * m.Nb};
    if ((rc = rem_map(&tw, w, 3, dw, sw, 128)) != SVA_OK) return rc;
    cuuint64_t dc[3] = {(cuuint64_t)rem::D * rem::D, (cuuint64_t)m.Nb, (cuuint64_t)BH};
    cuuint64_t sc[2] = {(cuuint64_t)rem::D * rem::D * 2, (cuuint64_t)rem::D * rem::D * 2 * m.Nb};
    if ((rc = rem_map(&tc, ct, 3, dc, sc, 64)) != SVA_OK) return rc;
    if ((rc = rem_map(&ta, at, 3, dc, sc, 128)) != SVA_OK) return rc;
    cuuint64_t dr[3] = {(cuuint64_t)rem::D, (cuuint64_t)rem::D * m.Nb, (cuuint64_t)BH};             // C^T by rows, to be written
    cuuint64_t sr[2] = {(cuuint64_t)rem::D * 2, (cuuint64_t)rem::D * rem::D * 2 * m.Nb};
    if ((rc = rem_map(&tco, ct, 3, dr, sr, 128)) != SVA_OK) return rc;
  }
  const int smem_cov = 2 * rem::TILE + 1024, chunks = Nbw / 64;
  const agg::Plan ap = agg::plan(m.Nb, chunks);
  static DeviceOnce once;
  if ((rc = once.run([&] {
         return cudaFuncSetAttribute(cov_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_cov) == cudaSuccess &&
                cudaFuncSetAttribute(aggregate_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 226 * 1024) == cudaSuccess;
       })) != SVA_OK)
    return rc;
  if ((rc = launch_dep(cov_kernel, dim3(m.Nb, m.B * m.H), 128, smem_cov, st, natural ? tv : tk, natural ? tk : tv, tco, m.H, m.N, m.block,
                       m.Nb, natural ? v_mean : k_mean, natural ? k_mean : v_mean, Nbp, row_counter, g_debug_rem, status)) != SVA_OK)
    return rc;
  if ((rc = launch_dep(weights_kernel, (m.R + 7) / 8, 256, 0, st, scores, row_ptr, col_idx, m.R, m.Nb, Nbw, w, mu)) != SVA_OK) return rc;
  const int groups = ((m.Nb + 127) / 128 + ap.tiles - 1) / ap.tiles;
  if ((rc = launch_dep(aggregate_kernel, dim3(agg::runs(groups * m.B * m.H), groups, m.B * m.H), 192, ap.smem, st, tw, tc, ta, m.Nb, chunks, ap.tiles,
                       ap.resident, ap.stages, g_debug_rem, status)) != SVA_OK)
    return rc;
  *at_out = at;
  *mu_out = mu;
  return SVA_OK;
}

}  // namespace sva
