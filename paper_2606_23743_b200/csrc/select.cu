// Block routing: mean pooling of Q and K per block, scaled pooled scores, per-row top-k or
// cumulative-mass selection with ties to the lower block index, optional forced neighbour
// window, CSR assembly.  (Paper: "score-based routing" of the critical blocks; block-wise
// similarity metric of the sparse-attention section.)
//
// pool_kernel streams Q and K once from HBM: 128-bit loads, fp32 accumulation in a fixed order, a CTA per
// run of blocks of a head of a tensor.  block_scores_kernel computes a head's score matrix as a
// small fp32 GEMM (64 x 64 or 32 x 32 tiles from two shared-memory panels, fixed summation order).  With few blocks per head one kernel
// scores and selects (route_means_kernel); the smallest problems take one for all three (route_cluster_kernel).
// select_rows_kernel is one warp per query-block row: it reads the row's scores from that matrix (no shared
// memory) as order-preserving integer keys, finds the threshold of the rule by narrowing an interval of scores
// that holds it and emits the kept blocks in ascending order.  When the per-row count is known on the host (top-k with no window
// larger than k) rows go straight into the CSR; otherwise they are staged and csr_kernel builds it in one launch.
#include <mutex>
#include <type_traits>

#include "common.cuh"

namespace sva {

static constexpr int POOL_THREADS = 256;

// acc += the elements of a 16-byte vector (eight bf16 or sixteen e4m3 codes), in pairs
template <int ELEM_BYTES>
__device__ __forceinline__ void add_vector(const uint4& u, uint64_t (&acc)[8 / ELEM_BYTES]) {
  const uint32_t w[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    if constexpr (ELEM_BYTES == 2) {
      acc[e] = add2(acc[e], pack2(bf16lo(w[e]), bf16hi(w[e])));
    } else {
      const float2 lo2 = e4m3x2_to_float2(w[e] & 0xffffu), hi2 = e4m3x2_to_float2(w[e] >> 16);
      acc[2 * e] = add2(acc[2 * e], pack2(lo2.x, lo2.y));
      acc[2 * e + 1] = add2(acc[2 * e + 1], pack2(hi2.x, hi2.y));
    }
  }
}

// Block means of one head of one tensor (blockIdx.z: 0 = Q, 1 = K); a CTA pools `run` consecutive blocks.
// ELEM_BYTES = 2: bf16 input.  ELEM_BYTES = 1: e4m3 codes, multiplied by the block's scale.
// Bound by the HBM: one pass over Q and K.  A CTA's loads run one block ahead of its sums, across the reduction (two barriers); with a
// CTA per block nothing was in flight while it reduced.  VECS: 16-byte vectors of a block per thread, so that a step is a whole block
// whatever its size (with four per step a 128-token block took two steps, and 64-token blocks of e4m3 codes or of d = 64 masked
// half of the loads).
// Q and K of 24 heads x 32 760 tokens, d = 128 (403 MB): 75.8 us with a CTA per block, 70.8 with runs of four, two steps a block,
// 69.1 so (5.8 TB/s);
// another box, four vectors and runs of four -> a block at a time and runs of up to 128 KB: 24 x 32 760 66.9 -> 61.8 (6.5 TB/s), in
// 64-token blocks 68.6 -> 65.0, 16 heads x 8 192 14.6 -> 12.3, 20 x 17 550 33.6 -> 30.9, 64 x 47 616 236.5 -> 223.4; d = 64 in
// 64-token blocks, 16 x 8 192, 11.7 -> 8.0.
// e4m3 codes (201 MB, converted in pairs) are bound by the sums and the reduction, which half the bytes do not hide: 66.5 -> 58.6
// us with the run, 52.6 -> 46.4 (on a faster box) with pairs added in one instruction and partial sums laid out so that no two
// lanes of a warp meet in a bank, 41.2 with runs of eight; in 64-token blocks 87.4 -> 47.4.
template <int D, int ELEM_BYTES, int VECS>
__global__ void __launch_bounds__(POOL_THREADS)
pool_kernel(const uint8_t* __restrict__ q, const uint8_t* __restrict__ k, Strides sq, Strides sk,
            const float* __restrict__ q_scale, const float* __restrict__ k_scale, int H, int N,
            int block, int Nb, int run, float* __restrict__ qbar, float* __restrict__ kbar) {
  constexpr int EPV = 16 / ELEM_BYTES;          // elements per 16-byte vector
  constexpr int VPR = D / EPV;                  // vectors per token row
  constexpr int GROUPS = POOL_THREADS / VPR;    // token rows read concurrently; VECS * GROUPS = block
  __shared__ float part[EPV][POOL_THREADS + (EPV == 8 ? 4 : 2)];    // (a warp's writes and its reads touch every bank once)

  // (e4m3 codes: from the end, which the quantiser has just written and the L2 still holds)
  constexpr bool BACK = ELEM_BYTES == 1;
  const int zero = grid_dep_wait(), bh = (BACK ? gridDim.y - 1 - blockIdx.y : blockIdx.y) + zero, which = BACK ? 1 - blockIdx.z : blockIdx.z;
  const int b = bh / H, h = bh % H;
  const Strides s = which ? sk : sq;
  const uint8_t* base = (which ? k : q) + ((long long)b * s.b + (long long)h * s.h) * ELEM_BYTES;
  const int I0 = (BACK ? gridDim.x - 1 - blockIdx.x : blockIdx.x) * run, I1 = min(I0 + run, Nb);
  const int vec = threadIdx.x % VPR, grp = threadIdx.x / VPR;

  uint4 u[VECS];
  auto load = [&](int I) {
    const int lo = I * block, cnt = I < I1 ? min(block, N - lo) : 0;
#pragma unroll
    for (int j = 0; j < VECS; ++j) {
      const int t = grp + j * GROUPS;
      u[j] = make_uint4(0, 0, 0, 0);
      if (t < cnt) u[j] = __ldg(reinterpret_cast<const uint4*>(base + (long long)(lo + t) * s.n * ELEM_BYTES) + vec);
    }
  };
  load(I0);
  for (int I = I0; I < I1; ++I) {
    uint64_t acc[EPV / 2];
#pragma unroll
    for (int e = 0; e < EPV / 2; ++e) acc[e] = 0ull;
    uint4 c[VECS];
#pragma unroll
    for (int j = 0; j < VECS; ++j) c[j] = u[j];
    load(I + 1);
#pragma unroll
    for (int j = 0; j < VECS; ++j) add_vector<ELEM_BYTES>(c[j], acc);
#pragma unroll
    for (int e = 0; e < EPV / 2; ++e) unpack2(acc[e], part[2 * e][grp * VPR + vec], part[2 * e + 1][grp * VPR + vec]);
    __syncthreads();
    if (threadIdx.x < D) {
      float sum = 0.f;
#pragma unroll 8
      for (int g = 0; g < GROUPS; ++g) sum += part[threadIdx.x % EPV][g * VPR + threadIdx.x / EPV];   // fixed order
      float mean = sum / (float)min(block, N - I * block);
      if (ELEM_BYTES == 1) mean *= (which ? k_scale : q_scale)[(long long)bh * Nb + I];
      (which ? kbar : qbar)[((long long)bh * Nb + I) * D + threadIdx.x] = mean;
    }
    __syncthreads();
  }
}

struct SelParams {
  int Nb, k, use_window, win_t, win_s, bpf, cap, fixed_n;
  float tau;
};

__device__ __forceinline__ bool in_window(int I, int J, const SelParams& p) {
  int ti = I / p.bpf, si = I % p.bpf, tj = J / p.bpf, sj = J % p.bpf;
  return abs(ti - tj) <= p.win_t && abs(si - sj) <= p.win_s;
}

// Order-preserving map float -> uint32 (larger score <=> larger key, every real score maps to a
// non-zero key); +0 and -0 share a key; NaN maps to 0, which is never selected.
__device__ __forceinline__ uint32_t score_key(float v) {
  if (!(v == v)) return 0u;
  uint32_t u = __float_as_uint(v + 0.0f);
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
__device__ __forceinline__ float key_score(uint32_t key) {
  return __uint_as_float((key & 0x80000000u) ? (key ^ 0x80000000u) : ~key);
}

// Mass rule: the softmax weights of a row's candidates, in units of 2^-31 (0 where there is none).
template <int ITEMS>
__device__ __forceinline__ void mass_weights(const uint32_t (&key)[ITEMS], uint32_t (&wgt)[ITEMS]) {
  uint32_t km = 0u;
#pragma unroll
  for (int it = 0; it < ITEMS; ++it) km = max(km, key[it]);
  km = __reduce_max_sync(0xffffffffu, km);
  const float mx = key_score(km);
  float z = 0.f, ew[ITEMS];
#pragma unroll
  for (int it = 0; it < ITEMS; ++it) {
    ew[it] = 0.f;
    if (key[it]) { ew[it] = expf(key_score(key[it]) - mx); z += ew[it]; }
  }
#pragma unroll
  for (int o = 16; o; o >>= 1) z += __shfl_xor_sync(0xffffffffu, z, o);
  const float inv_z = 1.0f / z;
#pragma unroll
  for (int it = 0; it < ITEMS; ++it) wgt[it] = __float2uint_rn(ew[it] * inv_z * 2147483648.f);
}

// A row's kept blocks (bit it of `mask`: block it*32 + lane; n of them) in ascending order: straight into the CSR where every row has
// the same count, else staged with its count.
template <int ITEMS>
__device__ __forceinline__ void emit_row(const uint32_t mask, const int n, const int I, const int bh, const int lane, const SelParams& p,
                                         int32_t* __restrict__ row_ptr, int32_t* __restrict__ col_idx, int32_t* __restrict__ tmp_idx,
                                         int32_t* __restrict__ counts, const int R) {
  const int Nb = p.Nb;
  const int r = bh * Nb + I;
  int32_t* out;
  if (p.fixed_n) {
    out = col_idx + (long long)r * p.fixed_n;
    if (lane == 0) {
      row_ptr[r] = r * p.fixed_n;
      if (r == R - 1) row_ptr[R] = R * p.fixed_n;
    }
    // (NaN scores are no candidates: the row can come out short; what row_ptr covers is written all the same)
#pragma unroll 1
    for (int t = n + lane; t < p.fixed_n; t += 32) out[t] = 0;
  } else {
    out = tmp_idx + (long long)r * p.cap;
    if (lane == 0) counts[r] = n;
  }
  int base = 0;
#pragma unroll
  for (int it = 0; it < ITEMS; ++it) {
    if (it * 32 >= Nb) break;
    bool sel = mask >> it & 1u;
    uint32_t bal = __ballot_sync(0xffffffffu, sel);
    if (sel) out[base + __popc(bal & ((1u << lane) - 1u))] = it * 32 + lane;
    base += __popc(bal);
  }
}

// Selection and emission of one query-block row by one warp.  Lane j owns the key blocks
// J = it*32 + j, it < ITEMS, whose scores arrive as sortable keys (0 = no candidate).
// MASS: the cumulative-mass rule (mode 1).
template <int ITEMS, bool MASS>
__device__ __forceinline__ void select_and_emit(uint32_t (&key)[ITEMS], const int I, const int bh, const int lane,
                                                const SelParams& p, int32_t* __restrict__ row_ptr,
                                                int32_t* __restrict__ col_idx, int32_t* __restrict__ tmp_idx,
                                                int32_t* __restrict__ counts, const int R) {
  const int Nb = p.Nb;
  // ---- selection
  // The rule is sequential -- forced window first, then candidates by score (descending, ties to the
  // lower index) until k blocks are kept or, in mode 1, the kept softmax mass reaches tau -- but what it
  // keeps is "every candidate above a threshold key plus the first few of the candidates equal to it":
  // T = the largest key at which taking every candidate >= it ends the rule.  T is a candidate's key, so the
  // search narrows an interval [lo, hi) of keys that holds it (lo ends the rule, hi does not; each step one
  // compare per register, a warp reduction of the count and, in mode 1, of the mass) only until one distinct
  // key is left in it.  Steps halve the interval in SCORE space: the scores of a row spread over a few units,
  // so about log2(candidates) + 2 steps isolate one, where halving the 32 key bits takes all 32 (sign and
  // exponent bits separate nothing).  Every fourth step tightens the interval to the candidates in it, which
  // ends rows of equal scores and drops outliers; every eighth halves the key bits, which bounds the search for
  // any input.  Against 32 steps on the key bits: 12 288 rows of 512 scores,
  // top-k, 55 -> 36 us; 6 144 rows of 256, mass rule, 21.5 -> 16.7 us.
  // The masses are summed in fixed point (weights in units of 2^-31: a warp-wide integer add is
  // one instruction where a float sum is five shuffle rounds, and the result does not depend on the order),
  // so decisions agree with the round-by-round form except where the mass comes within about 1e-7 --
  // fp32 summation noise -- of tau.
  uint32_t mask = 0;            // bit it set <=> block it*32+lane is kept
  int n = 0;
  uint32_t cum = 0u;            // kept mass so far, units of 2^-31
  const uint32_t tau_q = __float2uint_rn(fminf(fmaxf(p.tau, 0.f), 1.f) * 2147483648.f);
  uint32_t wgt[ITEMS];          // mode 1: softmax weight of every candidate, units of 2^-31
#pragma unroll
  for (int it = 0; it < ITEMS; ++it) wgt[it] = 0u;
  if (MASS) {
    mass_weights<ITEMS>(key, wgt);
  }
  if (p.use_window) {
    uint32_t fm = 0u;
    int cnt = 0;
#pragma unroll
    for (int it = 0; it < ITEMS; ++it) {
      const int J = it * 32 + lane;
      if (J < Nb && in_window(I, J, p)) {
        mask |= 1u << it; ++cnt;
        fm += wgt[it];
        key[it] = 0u;                        // no longer a candidate
        wgt[it] = 0u;
      }
    }
    n = (int)__reduce_add_sync(0xffffffffu, (unsigned)cnt);
    if (MASS) cum = __reduce_add_sync(0xffffffffu, fm);
  }
  const int kk = min(p.k, Nb);
  if (n < kk && !(MASS && n >= 1 && cum >= tau_q)) {
    // count and mass of the candidates with key >= t (t >= 1)
    auto above = [&](uint32_t t, int& cnt, uint32_t& mass) {
      int c = 0;
      uint32_t g = 0u;
#pragma unroll
      for (int it = 0; it < ITEMS; ++it) {
        const bool ge = key[it] >= t;
        c += ge;
        if (MASS && ge) g += wgt[it];
      }
      cnt = (int)__reduce_add_sync(0xffffffffu, (unsigned)c);
      mass = MASS ? __reduce_add_sync(0xffffffffu, g) : 0u;
    };
    auto ends = [&](int c, uint32_t g) { return n + c >= kk || (MASS && c >= 1 && cum + g >= tau_q); };
    // smallest and largest candidate key in [lo, hi) (it holds at least one)
    auto range = [&](uint32_t lo, uint32_t hi, uint32_t& kmin, uint32_t& kmax) {
      uint32_t a = 0xffffffffu, b = 0u;
#pragma unroll
      for (int it = 0; it < ITEMS; ++it)
        if (key[it] >= lo && key[it] < hi) { a = min(a, key[it]); b = max(b, key[it]); }
      kmin = __reduce_min_sync(0xffffffffu, a);
      kmax = __reduce_max_sync(0xffffffffu, b);
    };
    uint32_t T = 0u;                         // 0: the rule never ends, take every candidate
    int cl, G = 0;                           // candidates >= lo; candidates >= hi, and their mass
    uint32_t ml, Mg = 0u;
    above(1u, cl, ml);
    if (!ends(cl, ml)) {
      G = cl;
      Mg = ml;
    } else {
      uint32_t lo, hi;
      range(1u, 0xffffffffu, lo, hi);        // (no score has the key 0xffffffff)
      ++hi;
#pragma unroll 1
      for (int step = 0; hi - lo > 1u && cl - G > 1; ++step) {
        uint32_t t;
        if ((step & 7) == 7) {
          t = lo + ((hi - lo) >> 1);
        } else {
          t = score_key(0.5f * key_score(lo) + 0.5f * key_score(hi - 1u));      // (NaN -- infinities of both signs -- gives 0)
          t = min(max(t, lo + 1u), hi - 1u);
        }
        int c;
        uint32_t g;
        above(t, c, g);
        if (ends(c, g)) { lo = t; cl = c; } else { hi = t; G = c; Mg = g; }
        if ((step & 3) == 3) {
          range(lo, hi, lo, hi);
          ++hi;
        }
      }
      if (hi - lo > 1u) range(lo, hi, lo, hi);        // one candidate left
      T = lo;
    }
    // everything above T, then ties at T in index order while the rule still runs
    int have = n + G;
    uint32_t acc = cum + Mg;
    int ties_wanted = 0, E = 0;              // ties: candidates equal to T
    if (T != 0u) {
      uint32_t wT = 0u;                      // weight of a candidate equal to T (they all have the same)
#pragma unroll
      for (int it = 0; it < ITEMS; ++it) {
        E += (key[it] == T);
        if (key[it] == T) wT = wgt[it];
      }
      E = (int)__reduce_add_sync(0xffffffffu, (unsigned)E);
      if (MASS) wT = __reduce_max_sync(0xffffffffu, wT);
      while (ties_wanted < E) {
        if (have >= kk) break;
        if (MASS && have >= 1 && acc >= tau_q) break;
        ++ties_wanted; ++have; acc += wT;
      }
    }
    if (ties_wanted == E) {                  // all of them (the common case: one candidate holds the threshold)
#pragma unroll
      for (int it = 0; it < ITEMS; ++it)
        if (key[it] >= max(T, 1u)) mask |= 1u << it;
    } else {
      int seen = 0;                          // ties met so far, in index order
#pragma unroll
      for (int it = 0; it < ITEMS; ++it) {
        const bool gt = key[it] > T, eq = key[it] == T;          // (T != 0 here: T = 0 has no ties)
        const uint32_t bal = __ballot_sync(0xffffffffu, eq);
        const bool take = gt || (eq && seen + __popc(bal & ((1u << lane) - 1u)) < ties_wanted);
        if (take) mask |= 1u << it;
        seen += __popc(bal);
      }
    }
    n = have;
  }

  emit_row<ITEMS>(mask, n, I, bh, lane, p, row_ptr, col_idx, tmp_idx, counts, R);
}

// The same rule for short rows: each candidate counts the candidates in front of it (larger score, or equal and a lower index) and, for the
// mass rule, adds up their mass; it is kept if the sequential rule would still run when its turn comes.  No search, so a row is Nb steps of
// two or three independent instructions.  Cycles of a CTA's selection phase, threshold search -> this: rows of 16 scores 2 550 ->
// 1 070, eight rows of 64 scores 4 400 -> 2 650.
// sk, sw: the row's keys and weights in shared memory (32 * ITEMS words each).
template <int ITEMS, bool MASS>
__device__ __forceinline__ void rank_and_emit(uint32_t (&key)[ITEMS], uint32_t* sk, uint32_t* sw, const int I, const int bh,
                                              const int lane, const SelParams& p, int32_t* __restrict__ row_ptr,
                                              int32_t* __restrict__ col_idx, int32_t* __restrict__ tmp_idx,
                                              int32_t* __restrict__ counts, const int R) {
  const int Nb = p.Nb;
  const uint32_t tau_q = __float2uint_rn(fminf(fmaxf(p.tau, 0.f), 1.f) * 2147483648.f);
  uint32_t mask = 0u, cum = 0u, wgt[ITEMS], ahead[ITEMS], before[ITEMS];
  int n = 0;
#pragma unroll
  for (int it = 0; it < ITEMS; ++it) wgt[it] = ahead[it] = before[it] = 0u;
  if (MASS) mass_weights<ITEMS>(key, wgt);
  if (p.use_window) {
    uint32_t fm = 0u;
#pragma unroll
    for (int it = 0; it < ITEMS; ++it) {
      const int J = it * 32 + lane;
      if (J < Nb && in_window(I, J, p)) {
        mask |= 1u << it;
        fm += wgt[it];
        key[it] = wgt[it] = 0u;              // no longer a candidate
      }
    }
    n = (int)__reduce_add_sync(0xffffffffu, (unsigned)__popc(mask));
    if (MASS) cum = __reduce_add_sync(0xffffffffu, fm);
  }
#pragma unroll
  for (int it = 0; it < ITEMS; ++it) {
    sk[it * 32 + lane] = key[it];
    if (MASS) sw[it * 32 + lane] = wgt[it];
  }
  __syncwarp();
#pragma unroll
  for (int jb = 0; jb < ITEMS; ++jb) {
    const int j1 = min(32, Nb - jb * 32);                          // (what lies beyond Nb has key 0: in front of nothing)
#pragma unroll 2
    for (int j = 0; j < j1; j += 4) {
      const uint4 k4 = *reinterpret_cast<const uint4*>(sk + jb * 32 + j);
      uint4 w4 = make_uint4(0u, 0u, 0u, 0u);
      if (MASS) w4 = *reinterpret_cast<const uint4*>(sw + jb * 32 + j);
      const uint32_t kj[4] = {k4.x, k4.y, k4.z, k4.w}, wj[4] = {w4.x, w4.y, w4.z, w4.w};
#pragma unroll
      for (int e = 0; e < 4; ++e)
#pragma unroll
        for (int it = 0; it < ITEMS; ++it) {
          // (equal scores: the lower index goes first; a block that is no candidate, key 0, is behind everything or irrelevant)
          const bool precedes = jb < it ? kj[e] >= key[it] : kj[e] > (jb == it && j + e < lane ? key[it] - 1u : key[it]);
          if (precedes) ++ahead[it];
          if (MASS && precedes) before[it] += wj[e];
        }
    }
  }
  const uint32_t kk = (uint32_t)min(p.k, Nb);
  uint32_t kept = 0u;
#pragma unroll
  for (int it = 0; it < ITEMS; ++it) {
    const uint32_t at = (uint32_t)n + ahead[it];                   // blocks kept when this one's turn comes
    if (key[it] != 0u && at < kk && !(MASS && at >= 1u && cum + before[it] >= tau_q)) kept |= 1u << it;
  }
  mask |= kept;
  n += (int)__reduce_add_sync(0xffffffffu, (unsigned)__popc(kept));
  emit_row<ITEMS>(mask, n, I, bh, lane, p, row_ptr, col_idx, tmp_idx, counts, R);
}

// Block scores of one head as a small fp32 GEMM: S[I][J] = scale * <qbar_I, kbar_J>.  A CTA computes a
// (PQ * TY) x (PK * 16) tile from two D-wide panels in shared memory (row stride D + 4 floats: 128-bit reads of
// eight consecutive rows touch every bank once); a thread owns a PQ x PK patch -- rows PQ*ty.., keys tx, tx+16, .. --
// and keeps two partial sums per entry (dimensions 0,2 mod 4 and 1,3 mod 4, each in ascending order; that
// order is part of the result: it is what makes the scores reproducible bit for bit).  The two sums are the halves
// of one packed f32x2 accumulator, so four dimensions of an entry are two instructions.
// A 128-bit shared-memory read delivers 512 bytes to a warp whatever it broadcasts -- four cycles of the port -- so the 4 x 4
// patch of 256 threads ran at 90 % of the port; 8 x 4 needs a quarter fewer reads per FMA.  Patches beyond that (8 x 8 of
// 64 x 128 tiles: 19.3 / 49.8 us) and scalar FMAs measured the same: what is left is the FMA pipe at about half its
// nominal rate and the panels' load.  24 heads of 256 / 512 blocks, d = 128: 18.9 / 57 -> 16.2 / 51 us.
template <int D, int PQ, int PK, int TY>
__global__ void __launch_bounds__(16 * TY)
block_scores_kernel(const float* __restrict__ qbar, const float* __restrict__ kbar, int Nb, float scale,
                    float* __restrict__ scores) {
  constexpr int LD = D + 4, TQ = PQ * TY, TK = PK * 16, THREADS = 16 * TY, V = D / 4;
  extern __shared__ __align__(16) float sc_smem[];
  float* qs = sc_smem;                     // [TQ][LD]
  float* ks = sc_smem + TQ * LD;           // [TK][LD]
  grid_dep_launch();
  const int bh = blockIdx.z + grid_dep_wait(), I0 = blockIdx.y * TQ, J0 = blockIdx.x * TK;
  auto fill = [&](float* dst, const float* src, int r0, auto rows_tag) {      // eight 16-byte vectors per thread in flight
    constexpr int PER = decltype(rows_tag)::value * V / THREADS, BATCH = PER < 8 ? PER : 8;
#pragma unroll
    for (int u0 = 0; u0 < PER; u0 += BATCH) {
      float4 a[BATCH];
#pragma unroll
      for (int u = 0; u < BATCH; ++u) {
        const int idx = threadIdx.x + THREADS * (u0 + u), row = idx / V, c4 = idx % V;
        a[u] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (r0 + row < Nb) a[u] = __ldg(reinterpret_cast<const float4*>(src + (long long)(r0 + row) * D) + c4);
      }
#pragma unroll
      for (int u = 0; u < BATCH; ++u) {
        const int idx = threadIdx.x + THREADS * (u0 + u), row = idx / V, c4 = idx % V;
        *reinterpret_cast<float4*>(dst + row * LD + 4 * c4) = a[u];
      }
    }
  };
  fill(qs, qbar + (long long)bh * Nb * D, I0, std::integral_constant<int, TQ>{});
  fill(ks, kbar + (long long)bh * Nb * D, J0, std::integral_constant<int, TK>{});
  __syncthreads();
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  uint64_t acc[PQ][PK];
#pragma unroll
  for (int i = 0; i < PQ; ++i)
#pragma unroll
    for (int j = 0; j < PK; ++j) acc[i][j] = pack2(0.f, 0.f);
#pragma unroll 2
  for (int c = 0; c < D; c += 4) {
    ulonglong2 qv[PQ], kv[PK];
#pragma unroll
    for (int i = 0; i < PQ; ++i) qv[i] = *reinterpret_cast<const ulonglong2*>(qs + (ty * PQ + i) * LD + c);
#pragma unroll
    for (int j = 0; j < PK; ++j) kv[j] = *reinterpret_cast<const ulonglong2*>(ks + (tx + 16 * j) * LD + c);
#pragma unroll
    for (int i = 0; i < PQ; ++i)
#pragma unroll
      for (int j = 0; j < PK; ++j) {
        acc[i][j] = fma2(qv[i].x, kv[j].x, acc[i][j]);
        acc[i][j] = fma2(qv[i].y, kv[j].y, acc[i][j]);
      }
  }
#pragma unroll
  for (int i = 0; i < PQ; ++i) {
    const int I = I0 + ty * PQ + i;
    if (I >= Nb) continue;
#pragma unroll
    for (int j = 0; j < PK; ++j) {
      const int J = J0 + tx + 16 * j;
      float s0, s1;
      unpack2(acc[i][j], s0, s1);
      if (J < Nb) scores[((long long)bh * Nb + I) * Nb + J] = (s0 + s1) * scale;
    }
  }
}

template <int D, int PQ, int PK, int TY>
static int launch_scores(const float* qbar, const float* kbar, int Nb, int heads, float scale, float* scores, cudaStream_t st) {
  auto kern = block_scores_kernel<D, PQ, PK, TY>;
  constexpr int TQ = PQ * TY, TK = PK * 16, smem = (TQ + TK) * (D + 4) * (int)sizeof(float);
  static DeviceOnce once;
  const int rc = once.run([&] { return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) == cudaSuccess; });
  if (rc != SVA_OK) return rc;
  return launch_dep(kern, dim3((Nb + TK - 1) / TK, (Nb + TQ - 1) / TQ, heads), 16 * TY, smem, st, qbar, kbar, Nb, scale, scores);
}

// Selection: one warp per query-block row, its Nb scores read straight from the score matrix (lane j owns
// the key blocks it*32 + j).  No shared memory and few registers, so the SMs hold enough warps to hide the
// serial chain of the threshold search.
static constexpr int SEL_WARPS = 8;
template <int ITEMS, bool MASS>
__global__ void __launch_bounds__(SEL_WARPS * 32)
select_rows_kernel(const float* __restrict__ scores, SelParams p, int32_t* __restrict__ row_ptr,
                   int32_t* __restrict__ col_idx, int32_t* __restrict__ tmp_idx, int32_t* __restrict__ counts, int R) {
  grid_dep_launch();
  const int lane = threadIdx.x & 31;
  const int r = blockIdx.x * SEL_WARPS + (threadIdx.x >> 5) + grid_dep_wait();
  if (r >= R) return;
  const int Nb = p.Nb, bh = r / Nb, I = r % Nb;
  const float* srow = scores + (long long)r * Nb;
  uint32_t key[ITEMS];
#pragma unroll
  for (int it = 0; it < ITEMS; ++it) {
    const int J = it * 32 + lane;
    key[it] = J < Nb ? score_key(__ldg(srow + J)) : 0u;
  }
  select_and_emit<ITEMS, MASS>(key, I, bh, lane, p, row_ptr, col_idx, tmp_idx, counts, R);
}

// The smallest problems: pooling, scores and selection of one head by one cluster of eight CTAs, one launch.  Each CTA pools
// its share of the head's blocks of Q and K (a team of 256 threads per block), writes a key mean into the shared memory of all eight,
// and then scores and selects its own query blocks.  Sums run in the orders of pool_kernel and block_scores_kernel, so lists and
// scores are the same bytes.
// Bound by latency: the launch, the cluster's barriers (about 0.5 us each), the pooling of a block per team (about 1 100 cycles of
// loads, sums and reduction), and the score and selection phase of a warp per row.  Microseconds of a routing call (top-k),
// pool_kernel and route_means_kernel / this one: 2 heads x 16 blocks of 64 x 64 7.3 / 5.3, of 128 x 128 7.35 / 6.3; 1 x 8
// 7.3 / 5.5.
static constexpr int RC_CTAS = 8, RC_TEAMS = 4, RC_TEAM = 256, RC_MAX_NB = 16;
static constexpr int RC_ROWS = RC_MAX_NB / RC_CTAS;                         // query blocks per CTA at most
static constexpr int RC_KEYS = 32;                                          // rows of the panel of key means, one per lane
static_assert(2 * RC_ROWS <= RC_TEAMS && RC_MAX_NB <= RC_KEYS, "a team per block of Q and K");
__device__ __forceinline__ uint32_t smem_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire;" ::: "memory"); }
// a float into the shared memory of CTA `rank` of the cluster, at this CTA's address `addr`
__device__ __forceinline__ void store_cluster(uint32_t addr, int rank, float v) {
  asm volatile("{\n.reg .b32 a;\nmapa.shared::cluster.u32 a, %0, %1;\nst.shared::cluster.f32 [a], %2;\n}" ::"r"(addr), "r"(rank), "f"(v) : "memory");
}
template <int D, int ELEM_BYTES>
struct RcSmem {
  static constexpr int VPR = D * ELEM_BYTES / 16, GROUPS = RC_TEAM / VPR, EPV = 16 / ELEM_BYTES, LD = D + 4;
  // partial sums [element of the vector][group][vector]: both the writes (a lane per vector) and the reads (a lane per column) of a
  // warp touch every bank once
  static constexpr int PART = GROUPS * VPR + (EPV == 8 ? 4 : 2);
  float part[RC_TEAMS][EPV * PART];
};
// Scores and selection of `mine` consecutive query blocks of a head, from I0 on, by a whole CTA (a warp per row at least): ks, qm are the
// head's key means and the blocks' means in shared memory ([..][D + 4]), keys and wgts room for 32 * ITEMS words per row.
template <int D, int RQ, int ITEMS, bool MASS>
__device__ __forceinline__ void score_and_select(const float* ks, const float* qm, uint32_t* keys, uint32_t* wgts, const int mine, const int I0,
                                                 const int bh, const float scale, const SelParams& p, float* __restrict__ scores,
                                                 int32_t* __restrict__ row_ptr, int32_t* __restrict__ col_idx,
                                                 int32_t* __restrict__ tmp_idx, int32_t* __restrict__ counts, const int R) {
  constexpr int LD = D + 4;
  const int Nb = p.Nb;
  // ---- scores as keys: a thread per RQ query blocks and ITEMS key blocks, sums as in block_scores_kernel
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (warp * RQ < mine) {
    uint64_t acc[RQ][ITEMS];
#pragma unroll
    for (int i = 0; i < RQ; ++i)
#pragma unroll
      for (int it = 0; it < ITEMS; ++it) acc[i][it] = pack2(0.f, 0.f);
    const float* qrow = qm + warp * RQ * LD;
    const float* krow = ks + lane * LD;
#pragma unroll 2
    for (int c = 0; c < D; c += 4) {
      ulonglong2 kv[ITEMS];
#pragma unroll
      for (int it = 0; it < ITEMS; ++it) kv[it] = *reinterpret_cast<const ulonglong2*>(krow + it * 32 * LD + c);
#pragma unroll
      for (int i = 0; i < RQ; ++i) {
        const ulonglong2 qv = *reinterpret_cast<const ulonglong2*>(qrow + i * LD + c);
#pragma unroll
        for (int it = 0; it < ITEMS; ++it) {
          acc[i][it] = fma2(qv.x, kv[it].x, acc[i][it]);
          acc[i][it] = fma2(qv.y, kv[it].y, acc[i][it]);
        }
      }
    }
#pragma unroll
    for (int i = 0; i < RQ; ++i) {
      const int li = warp * RQ + i;
      if (li >= mine) break;
#pragma unroll
      for (int it = 0; it < ITEMS; ++it) {
        const int J = it * 32 + lane;
        float s0, s1;
        unpack2(acc[i][it], s0, s1);
        const float v = (s0 + s1) * scale;
        keys[li * 32 * ITEMS + J] = J < Nb ? score_key(v) : 0u;
        if (scores && J < Nb) scores[((long long)bh * Nb + I0 + li) * Nb + J] = v;
      }
    }
  }
  __syncthreads();

  // ---- selection: a warp per row
  const int li = warp;
  if (li < mine) {
    uint32_t* sk = keys + li * 32 * ITEMS;
    uint32_t key[ITEMS];
#pragma unroll
    for (int it = 0; it < ITEMS; ++it) key[it] = sk[it * 32 + lane];
    rank_and_emit<ITEMS, MASS>(key, sk, wgts + li * 32 * ITEMS, I0 + li, bh, lane, p, row_ptr, col_idx, tmp_idx, counts, R);
  }
}
template <int D, int ELEM_BYTES, bool MASS>
__global__ void __launch_bounds__(RC_TEAMS * RC_TEAM)
route_cluster_kernel(const uint8_t* __restrict__ q, const uint8_t* __restrict__ k, Strides sq, Strides sk,
                     const float* __restrict__ q_scale, const float* __restrict__ k_scale, int H, int N, int block, float scale,
                     SelParams p, float* __restrict__ scores, int32_t* __restrict__ row_ptr, int32_t* __restrict__ col_idx,
                     int32_t* __restrict__ tmp_idx, int32_t* __restrict__ counts, int R) {
  using Sm = RcSmem<D, ELEM_BYTES>;
  constexpr int VPR = Sm::VPR, GROUPS = Sm::GROUPS, EPV = Sm::EPV, LD = Sm::LD, NV = 128 / GROUPS;     // NV: vectors per thread and block
  extern __shared__ __align__(16) uint8_t rc_smem[];
  Sm& sm = *reinterpret_cast<Sm*>(rc_smem);
  float* ks = reinterpret_cast<float*>(rc_smem + sizeof(Sm));          // [32][LD] key means of the head
  float* qm = ks + RC_KEYS * LD;                                       // [rows][LD] means of my query blocks
  uint32_t* keys = reinterpret_cast<uint32_t*>(qm + RC_ROWS * LD);      // [rows][32] scores as keys
  uint32_t* wgts = keys + RC_ROWS * RC_KEYS;                            // ... and their weights
  const int Nb = p.Nb, per = (Nb + RC_CTAS - 1) / RC_CTAS;
  cluster_arrive();                        // (the CTAs of the cluster have started: they may be written to)
  const int rank = blockIdx.x % RC_CTAS, bh = blockIdx.x / RC_CTAS + grid_dep_wait();
  const int b = bh / H, h = bh % H, I0 = rank * per, mine = max(0, min(per, Nb - I0));
  const int team = threadIdx.x / RC_TEAM, tt = threadIdx.x % RC_TEAM, vec = tt % VPR, grp = tt / VPR;

  // ---- pooling: teams 0 .. mine-1 take a block of Q each, the next ones a block of K
  const bool pools = team < 2 * mine;
  const int which = team >= mine, li = which ? team - mine : team, I = I0 + li;
  const int lo = I * block, cnt = pools ? min(block, N - lo) : 0;
  uint4 u[NV];
  {
    const Strides s = which ? sk : sq;
    const uint8_t* base = (which ? k : q) + ((long long)b * s.b + (long long)h * s.h + (long long)(lo + grp) * s.n) * ELEM_BYTES;
#pragma unroll
    for (int j = 0; j < NV; ++j) {
      u[j] = make_uint4(0, 0, 0, 0);
      if (grp + j * GROUPS < cnt) u[j] = __ldg(reinterpret_cast<const uint4*>(base + (long long)(j * GROUPS) * s.n * ELEM_BYTES) + vec);
    }
  }
  cluster_wait();
  if (pools) {
    uint64_t acc[EPV / 2];
#pragma unroll
    for (int e = 0; e < EPV / 2; ++e) acc[e] = 0ull;
#pragma unroll
    for (int j = 0; j < NV; ++j) add_vector<ELEM_BYTES>(u[j], acc);
    float* part = sm.part[team];
#pragma unroll
    for (int e = 0; e < EPV / 2; ++e)
      unpack2(acc[e], part[2 * e * Sm::PART + grp * VPR + vec], part[(2 * e + 1) * Sm::PART + grp * VPR + vec]);
    asm volatile("bar.sync %0, %1;" ::"r"(1 + team), "r"(RC_TEAM) : "memory");
    if (tt < D) {
      float sum = 0.f;
#pragma unroll 8
      for (int g = 0; g < GROUPS; ++g) sum += part[(tt % EPV) * Sm::PART + g * VPR + tt / EPV];       // fixed order
      float mean = sum / (float)cnt;
      if (ELEM_BYTES == 1) mean *= (which ? k_scale : q_scale)[(long long)bh * Nb + I];
      if (which) {
        const uint32_t dst = smem_addr(ks + I * LD + tt);
#pragma unroll
        for (int r = 0; r < RC_CTAS; ++r) store_cluster(dst, r, mean);
      } else {
        qm[li * LD + tt] = mean;
      }
    }
  }
  grid_dep_launch();
  cluster_arrive();
  cluster_wait();

  score_and_select<D, RC_ROWS, 1, MASS>(ks, qm, keys, wgts, mine, I0, bh, scale, p, scores, row_ptr, col_idx, tmp_idx, counts, R);
}

// The same tail for block means that are at hand (a pooling or prologue kernel has written them): scores and selection of eight query
// blocks of a head per CTA, one launch instead of two.  Up to 64 blocks per head, where the key means fit beside one another and a
// row's rank is counted.  Bound by latency: the means' way from the L2, then as above.  Routing from means, scores and selection
// kernels -> this one (us, top-k / mass rule with csr_kernel): 16 heads x 64 blocks 8.0 -> 4.9 / 15.2 -> 6.9, 24 x 64 12.3 ->
// 8.6 / 20.5 -> 11.2, 128 x 64 22.3 -> 15.0 / 27.8 -> 20.8, 2 x 16 6.3 -> 4.9 / 8.4 -> 6.9.
static constexpr int RT_ROWS = 8, RT_ITEMS = 2, RT_MAX_NB = 32 * RT_ITEMS;
// Counting ranks is Nb steps per row where the threshold search takes about log2(Nb) + 2, so with long rows it pays only while the
// two launches that it saves weigh more than the counting: up to 40 blocks always, beyond that up to a work (CTAs x steps) that 160
// heads of 64 blocks come to (187 with the mass rule, whose search carries the masses along).  From means, d = 128, us, scores and
// selection kernels / this one: top-k, 128 heads x 64 blocks 22.3 / 15.0, 160 x 64 19.4 / 18.3, 200 x 64 20.8 / 22.0, 1 024 x 64
// 76.6 / 99.2, 220 x 52 19.6 / 19.6, 1 200 x 52 78 / 89, 1 200 x 40 67 / 63; mass rule, 200 x 64 32.9 / 31.0, 300 x 64 40.6 / 44.5.
static bool route_by_rank(const Dims& m, int mode) {
  return m.Nb <= 40 || (m.Nb <= RT_MAX_NB && (long long)m.B * m.H * ((m.Nb + RT_ROWS - 1) / RT_ROWS) * m.Nb <= (mode == 1 ? 96000 : 82000));
}
template <int D, bool MASS>
__global__ void __launch_bounds__(RT_ROWS * 32)
route_means_kernel(const float* __restrict__ qbar, const float* __restrict__ kbar, float scale, SelParams p, float* __restrict__ scores,
                   int32_t* __restrict__ row_ptr, int32_t* __restrict__ col_idx, int32_t* __restrict__ tmp_idx,
                   int32_t* __restrict__ counts, int R) {
  constexpr int LD = D + 4, V = D / 4;
  extern __shared__ __align__(16) uint8_t rc_smem[];
  float* ks = reinterpret_cast<float*>(rc_smem);                       // [64][LD]
  float* qm = ks + RT_MAX_NB * LD;                                     // [8][LD]
  uint32_t* keys = reinterpret_cast<uint32_t*>(qm + RT_ROWS * LD);
  uint32_t* wgts = keys + RT_ROWS * RT_MAX_NB;
  grid_dep_launch();
  const int bh = blockIdx.y + grid_dep_wait(), I0 = blockIdx.x * RT_ROWS, mine = min(RT_ROWS, p.Nb - I0);
  const float4* ksrc = reinterpret_cast<const float4*>(kbar + (long long)bh * p.Nb * D);
  const float4* qsrc = reinterpret_cast<const float4*>(qbar + ((long long)bh * p.Nb + I0) * D);
  constexpr int PER = RT_MAX_NB * V / (RT_ROWS * 32);                  // 16-byte vectors per thread, all in flight
  float4 a[PER];
#pragma unroll
  for (int u = 0; u < PER; ++u) {
    const int x = threadIdx.x + u * RT_ROWS * 32;
    a[u] = x < p.Nb * V ? __ldg(ksrc + x) : make_float4(0.f, 0.f, 0.f, 0.f);
  }
  for (int x = threadIdx.x; x < mine * V; x += RT_ROWS * 32) *reinterpret_cast<float4*>(qm + x / V * LD + 4 * (x % V)) = __ldg(qsrc + x);
#pragma unroll
  for (int u = 0; u < PER; ++u) {
    const int x = threadIdx.x + u * RT_ROWS * 32;
    *reinterpret_cast<float4*>(ks + x / V * LD + 4 * (x % V)) = a[u];
  }
  __syncthreads();
  score_and_select<D, 2, RT_ITEMS, MASS>(ks, qm, keys, wgts, mine, I0, bh, scale, p, scores, row_ptr, col_idx, tmp_idx, counts, R);
}

// CSR assembly for rows of varying length, one launch: a CTA owns 32 consecutive rows (one warp each).  It
// first adds up the counts of all rows before its own (every thread a strided share, then a block
// reduction: at most R counts = a few KB from the L2 per CTA, which is cheaper than a scan kernel of its
// own plus its launch), then scans its 32 counts, writes row_ptr and copies the staged indices.
static constexpr int CSR_ROWS = 32;
__global__ void __launch_bounds__(CSR_ROWS * 32)
csr_kernel(const int32_t* __restrict__ tmp_idx, const int32_t* __restrict__ counts, int cap, int R,
           int32_t* __restrict__ row_ptr, int32_t* __restrict__ col_idx) {
  __shared__ int warp_sum[32];
  __shared__ int row_off[CSR_ROWS + 1];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  grid_dep_launch();
  const int zero = grid_dep_wait(), r0 = blockIdx.x * CSR_ROWS + zero;
  int part = 0;
  for (int i = threadIdx.x + zero; i < r0; i += CSR_ROWS * 32) part += __ldg(counts + i);
#pragma unroll
  for (int o = 16; o; o >>= 1) part += __shfl_xor_sync(0xffffffffu, part, o);
  if (lane == 0) warp_sum[warp] = part;
  __syncthreads();
  if (warp == 0) {
    int base = warp_sum[lane];
#pragma unroll
    for (int o = 16; o; o >>= 1) base += __shfl_xor_sync(0xffffffffu, base, o);   // rows before this CTA
    const int r = r0 + lane;
    const int c = r < R ? __ldg(counts + r) : 0;
    int incl = c;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += y;
    }
    row_off[lane] = base + incl - c;
    if (r < R) row_ptr[r] = base + incl - c;
    if (r == R - 1) row_ptr[R] = base + incl;
  }
  __syncthreads();
  const int r = r0 + warp;
  if (r >= R) return;
  const int n = __ldg(counts + r), dst = row_off[warp];
  for (int t = lane; t < n; t += 32) col_idx[dst + t] = tmp_idx[(long long)r * cap + t];
}

static size_t align256(size_t x) { return (x + 255) & ~(size_t)255; }

int select_row_cap(const Dims& m, const sva_select_t* s) {
  int kk = s->k < m.Nb ? s->k : m.Nb;
  int cap = kk;
  if (s->win_t >= 0 && s->win_s >= 0 && s->blocks_per_frame > 0) {
    long long w = (long long)(2 * s->win_t + 1) * (2 * s->win_s + 1);
    if (w > m.Nb) w = m.Nb;
    if (w > cap) cap = (int)w;
  }
  return cap;
}

// The row count is known on the host when the rule is top-k and the window cannot exceed k.
static int fixed_count(const Dims& m, const sva_select_t* s) {
  int kk = s->k < m.Nb ? s->k : m.Nb;
  if (s->mode != 0) return 0;
  return select_row_cap(m, s) == kk ? kk : 0;
}

size_t select_workspace_bytes(const Dims& m, const sva_select_t* s) {
  size_t pooled = align256((size_t)m.B * m.H * m.Nb * m.d * sizeof(float));
  size_t bytes = 2 * pooled;
  if (!fixed_count(m, s)) {
    bytes += align256((size_t)m.R * select_row_cap(m, s) * sizeof(int32_t));
    bytes += align256((size_t)m.R * sizeof(int32_t));
  }
  bytes += align256((size_t)m.R * m.Nb * sizeof(float));      // the score matrix (unused when the caller asks for it)
  return bytes;
}

template <int D>
static int launch_pool_d(const Dims& m, const sva_problem_t* p, const void* q, const void* k, const float* q_scale,
                         const float* k_scale, float* qbar, float* kbar, cudaStream_t st) {
  const int eb = m.fp8 ? 1 : 2, run = blocks_per_cta(2LL * m.R, m.block * D * eb);
  const dim3 grid((m.Nb + run - 1) / run, m.B * m.H, 2);
  // (blocks of 64 or 128 tokens: block * D * eb bytes over 256 threads of 16)
  constexpr int V2 = D / 32, V1 = D / 64;                         // vectors per thread of a 64-token block, bf16 and e4m3
  auto kern = m.block == 64 ? (m.fp8 ? pool_kernel<D, 1, V1> : pool_kernel<D, 2, V2>)
                            : (m.fp8 ? pool_kernel<D, 1, 2 * V1> : pool_kernel<D, 2, 2 * V2>);
  return launch_dep(kern, grid, POOL_THREADS, 0, st, (const uint8_t*)q, (const uint8_t*)k,
                    make_strides(p->q_stride), make_strides(p->k_stride), m.fp8 ? q_scale : nullptr, m.fp8 ? k_scale : nullptr,
                    m.H, m.N, m.block, m.Nb, run, qbar, kbar);
}

// Where the cluster kernel routes.  Up to 14 heads each of its CTAs has an SM to itself (15 or more clusters of eight SMs do not
// fit at once), and up to 16 blocks (RC_MAX_NB) a CTA pools in one round.  Beyond that pooling over all SMs and route_means_kernel
// are faster (us, them / a cluster): 12 heads x 20 blocks of 128 x 128 7.3 / 7.9, 12 x 44 9.8 / 12.2, 16 x 16 7.2 / 8.0 (with two
// CTAs per SM), 6 x 64 8.5 / 13.4.
// Where the device cannot hold such a cluster -- the largest cluster shrinks in a partition of too few SMs -- those two serve these
// sizes too.
static int g_debug_route = 0;
void route_set_debug_mode(int v) { g_debug_route = v; }
static bool route_in_cluster(const Dims& m) { return m.Nb <= RC_MAX_NB && m.B * m.H <= 14; }
template <int D, int ELEM_BYTES, bool MASS>
static int launch_route(const Dims& m, const sva_problem_t* p, const void* q, const void* k, const float* q_scale, const float* k_scale,
                        const SelParams& sp, float* scores, int32_t* row_ptr, int32_t* col_idx, int32_t* tmp_idx, int32_t* counts,
                        cudaStream_t st) {
  auto kern = route_cluster_kernel<D, ELEM_BYTES, MASS>;
  using Sm = RcSmem<D, ELEM_BYTES>;
  constexpr int smem = (int)sizeof(Sm) + 4 * ((RC_KEYS + RC_ROWS) * Sm::LD + 2 * RC_ROWS * RC_KEYS);
  const int ctas = g_debug_route & 64 ? 32 : RC_CTAS;                  // (test aid: more CTAs than any device takes)
  auto fits = [&] {
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = (unsigned)ctas;
    attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(ctas);
    cfg.blockDim = dim3(RC_TEAMS * RC_TEAM);
    cfg.dynamicSmemBytes = smem;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    int n = 0;
    const bool ok = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) == cudaSuccess &&
                    cudaOccupancyMaxActiveClusters(&n, kern, &cfg) == cudaSuccess && n > 0;
    if (!ok) (void)cudaGetLastError();
    return ok;
  };
  static DeviceOnce once;
  const int rc = ctas == RC_CTAS ? once.run(fits) : fits() ? (int)SVA_OK : (int)SVA_ERR_CUDA;
  if (rc != SVA_OK) return rc;
  return launch_dep_cluster(RC_CTAS, kern, m.B * m.H * RC_CTAS, RC_TEAMS * RC_TEAM, smem, st, (const uint8_t*)q, (const uint8_t*)k,
                            make_strides(p->q_stride), make_strides(p->k_stride), q_scale, k_scale, m.H, m.N, m.block, m.scale, sp,
                            scores, row_ptr, col_idx, tmp_idx, counts, m.R);
}

template <int D>
static int launch_select_d(const Dims& m, const sva_problem_t* p, const sva_select_t* s,
                           const void* q, const void* k, const float* q_scale,
                           const float* k_scale, int32_t* row_ptr, int32_t* col_idx,
                           float* block_scores, void* ws, cudaStream_t st,
                           const float* qbar_in = nullptr, const float* kbar_in = nullptr) {
  size_t pooled = align256((size_t)m.B * m.H * m.Nb * m.d * sizeof(float));
  char* w = static_cast<char*>(ws);
  // (block means supplied by the caller -- the fused prologue writes them -- are used where they are)
  float* qbar = qbar_in ? const_cast<float*>(qbar_in) : reinterpret_cast<float*>(w);
  float* kbar = kbar_in ? const_cast<float*>(kbar_in) : reinterpret_cast<float*>(w + pooled);
  const int cap = select_row_cap(m, s);
  const int fixed_n = fixed_count(m, s);
  int32_t* tmp_idx = nullptr;
  int32_t* counts = nullptr;
  if (!fixed_n) {
    tmp_idx = reinterpret_cast<int32_t*>(w + 2 * pooled);
    counts = reinterpret_cast<int32_t*>(w + 2 * pooled + align256((size_t)m.R * cap * sizeof(int32_t)));
  }
  int rc = SVA_OK;
  SelParams sp;
  sp.Nb = m.Nb; sp.k = s->k;
  sp.use_window = (s->win_t >= 0 && s->win_s >= 0 && s->blocks_per_frame > 0) ? 1 : 0;
  sp.win_t = s->win_t; sp.win_s = s->win_s; sp.bpf = sp.use_window ? s->blocks_per_frame : 1;
  sp.cap = cap; sp.fixed_n = fixed_n; sp.tau = s->mass;
  auto csr = [&]() {
    if (fixed_n) return (int)SVA_OK;
    return launch_dep(csr_kernel, (m.R + CSR_ROWS - 1) / CSR_ROWS, CSR_ROWS * 32, 0, st, tmp_idx, counts, cap, m.R, row_ptr, col_idx);
  };
  if (!qbar_in && route_in_cluster(m)) {
    auto route = [&](auto elem_tag, auto mass_tag) {
      return launch_route<D, decltype(elem_tag)::value, decltype(mass_tag)::value>(
          m, p, q, k, m.fp8 ? q_scale : nullptr, m.fp8 ? k_scale : nullptr, sp, block_scores, row_ptr, col_idx, tmp_idx, counts, st);
    };
    auto by_mass = [&](auto elem_tag) { return s->mode == 1 ? route(elem_tag, std::true_type{}) : route(elem_tag, std::false_type{}); };
    rc = m.fp8 ? by_mass(std::integral_constant<int, 1>{}) : by_mass(std::integral_constant<int, 2>{});
    if (rc == SVA_OK) return csr();                              // (else: no room for a cluster, nothing was launched)
  }
  if (!qbar_in && (rc = launch_pool_d<D>(m, p, q, k, q_scale, k_scale, qbar, kbar, st)) != SVA_OK) return rc;
  if (route_by_rank(m, s->mode)) {
    constexpr int smem = 4 * ((RT_MAX_NB + RT_ROWS) * (D + 4) + 2 * RT_ROWS * RT_MAX_NB);      // (below the 48 KB that need no attribute)
    static_assert(smem <= 48 * 1024, "");
    rc = launch_dep(s->mode == 1 ? route_means_kernel<D, true> : route_means_kernel<D, false>,
                    dim3((m.Nb + RT_ROWS - 1) / RT_ROWS, m.B * m.H), RT_ROWS * 32, smem, st, (const float*)qbar, (const float*)kbar,
                    m.scale, sp, block_scores, row_ptr, col_idx, tmp_idx, counts, m.R);
    return rc != SVA_OK ? rc : csr();
  }
  // scores: into the caller's matrix if it wants one, else into the workspace (after the staging arrays)
  float* scores = block_scores;
  if (!scores) {
    size_t off = 2 * pooled;
    if (!fixed_n) off += align256((size_t)m.R * cap * sizeof(int32_t)) + align256((size_t)m.R * sizeof(int32_t));
    scores = reinterpret_cast<float*>(w + off);
  }
  {
    // 64 x 64 tiles where they give most of the SMs a CTA, else 32 x 32: with few rows the time is one CTA's latency, and
    // that shrinks with its tile.  Routing from means, d = 128, top-k, us, 64 x 64 / 32 x 32: 1 head x 66 blocks 10.4 / 9.1,
    // 2 x 100 9.9 / 8.2, 6 x 128 10.8 / 10.0, 2 x 192 12.0 / 10.2.  Between 48 and 96 tiles of 64 x 64 neither is the better one
    // throughout, since the time also depends on where the selection's waiting CTAs have settled: 16 x 80 10.4 / 16.5, 20 x 66
    // 10.5 / 18.0, 6 x 129 16.4 / 12.4, 23 x 100 21.7 / 20.2, 8 x 192 21.3 / 22.5.
    const int heads = m.B * m.H, nt = (m.Nb + 63) / 64;
    rc = nt * nt * heads >= 96 ? launch_scores<D, 8, 4, 8>(qbar, kbar, m.Nb, heads, m.scale, scores, st)
                             : launch_scores<D, 2, 2, 16>(qbar, kbar, m.Nb, heads, m.scale, scores, st);
    if (rc != SVA_OK) return rc;
  }
  const int items = (m.Nb + 31) / 32;
  const int sg = (m.R + SEL_WARPS - 1) / SEL_WARPS;
  auto select = [&](auto items_tag) {
    constexpr int IT = decltype(items_tag)::value;
    return launch_dep(s->mode == 1 ? select_rows_kernel<IT, true> : select_rows_kernel<IT, false>, sg, SEL_WARPS * 32, 0, st, scores, sp,
                      row_ptr, col_idx, tmp_idx, counts, m.R);
  };
  if (items <= 4) rc = select(std::integral_constant<int, 4>{});
  else if (items <= 8) rc = select(std::integral_constant<int, 8>{});
  else if (items <= 12) rc = select(std::integral_constant<int, 12>{});
  else if (items <= 16) rc = select(std::integral_constant<int, 16>{});
  else rc = select(std::integral_constant<int, 32>{});
  return rc != SVA_OK ? rc : csr();
}

int launch_select(const Dims& m, const sva_problem_t* p, const sva_select_t* s, const void* q,
                  const void* k, const float* q_scale, const float* k_scale, int32_t* row_ptr,
                  int32_t* col_idx, float* block_scores, void* ws, size_t ws_bytes,
                  cudaStream_t st) {
  if (ws_bytes < select_workspace_bytes(m, s)) return SVA_ERR_WORKSPACE;
  if (m.Nb > 1024) return SVA_ERR_UNSUPPORTED;    // a lane holds at most 32 scores of a row, kept flags in one word per lane
  if (m.d == 128)
    return launch_select_d<128>(m, p, s, q, k, q_scale, k_scale, row_ptr, col_idx, block_scores, ws, st);
  if (m.d == 64)
    return launch_select_d<64>(m, p, s, q, k, q_scale, k_scale, row_ptr, col_idx, block_scores, ws, st);
  return SVA_ERR_UNSUPPORTED;
}

// Pooling alone: block means of Q and K into the caller's arrays ([B,H,Nb,d] fp32 each).
int launch_pool(const Dims& m, const sva_problem_t* p, const void* q, const void* k, const float* q_scale,
                const float* k_scale, float* qbar, float* kbar, cudaStream_t st) {
  if (m.d == 128) return launch_pool_d<128>(m, p, q, k, q_scale, k_scale, qbar, kbar, st);
  if (m.d == 64) return launch_pool_d<64>(m, p, q, k, q_scale, k_scale, qbar, kbar, st);
  return SVA_ERR_UNSUPPORTED;
}

// Routing from block means the caller already has (qbar, kbar: [B,H,Nb,d] fp32).
int launch_select_pooled(const Dims& m, const sva_problem_t* p, const sva_select_t* s, const float* qbar,
                         const float* kbar, int32_t* row_ptr, int32_t* col_idx, float* block_scores, void* ws,
                         size_t ws_bytes, cudaStream_t st) {
  if (ws_bytes < select_workspace_bytes(m, s)) return SVA_ERR_WORKSPACE;
  if (m.Nb > 1024) return SVA_ERR_UNSUPPORTED;
  if (m.d == 128)
    return launch_select_d<128>(m, p, s, nullptr, nullptr, nullptr, nullptr, row_ptr, col_idx, block_scores, ws, st, qbar, kbar);
  if (m.d == 64)
    return launch_select_d<64>(m, p, s, nullptr, nullptr, nullptr, nullptr, row_ptr, col_idx, block_scores, ws, st, qbar, kbar);
  return SVA_ERR_UNSUPPORTED;
}

// ---------------------------------------------------------------- no-allocation variant
// Scratch for callers that cannot call cudaMalloc: it lives in the library image, so every
// GPU that loads the library carries these bytes until the process exits.  In host code the
// array's name is only a stand-in for the symbol -- not a device address -- so the address
// is looked up once per device with cudaGetSymbolAddress and that pointer is what the kernels
// receive.
static __device__ __align__(256) unsigned char g_noalloc_scratch[SVA_NOALLOC_SCRATCH_BYTES];

static constexpr int MAX_DEVICES = 64;
static std::mutex g_noalloc_mutex;
static void* g_noalloc_addr[MAX_DEVICES];   // device address of g_noalloc_scratch, per device

int launch_select_noalloc(const Dims& m, const sva_problem_t* p, const sva_select_t* s,
                          const void* q, const void* k, const float* q_scale, const float* k_scale,
                          int32_t* row_ptr, int32_t* col_idx, float* block_scores, cudaStream_t st) {
  if (select_workspace_bytes(m, s) > (size_t)SVA_NOALLOC_SCRATCH_BYTES) return SVA_ERR_SCRATCH_LIMIT;
  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= MAX_DEVICES) return SVA_ERR_CUDA;
  void* scratch = nullptr;
  {
    std::lock_guard<std::mutex> lock(g_noalloc_mutex);
    if (!g_noalloc_addr[dev]) {
      // first call on this device (it is the current one): resolve the symbol
      void* addr = nullptr;
      if (cudaGetSymbolAddress(&addr, g_noalloc_scratch) != cudaSuccess || !addr) return SVA_ERR_CUDA;
      g_noalloc_addr[dev] = addr;
    }
    scratch = g_noalloc_addr[dev];
  }
  // Nothing in the scratch has to start at zero: pooled means, staged rows and counts are all
  // written by this call's kernels before they are read.
  return launch_select(m, p, s, q, k, q_scale, k_scale, row_ptr, col_idx, block_scores, scratch,
                       (size_t)SVA_NOALLOC_SCRATCH_BYTES, st);
}

}  // namespace sva
