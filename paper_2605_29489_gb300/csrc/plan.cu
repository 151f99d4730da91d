// Alg. 1 PlanGen on the device, as one persistent kernel.
//
// The grid's CTAs all stay resident and move through the phases below together, separated by
// grid-wide barriers.  Every phase gives warp w of CTA c a contiguous slice of the data, so
// order is preserved wherever it matters.
//
//  0  tensor-level fallback (only for catalogs with entries lacking statistics, nnz =
//     kNnzMissing): flag every (expert, tensor) pair holding one; then one warp per flagged
//     pair computes its unit's cost (the whole tensor's bytes) and score (|coef_i| times
//     the norm of the tensor's known blocks: an fp32 fma chain in block order, then sqrt).
//     The pair's unit is b0(t)*K + i; the tensor's other units are not candidates.
//  A  score: unit u = b*K + i is a candidate iff nnz > 0 (TIES: and key(maxabs) >= tau);
//     score = |coef_i| * norm (fp32), divided by the block's bytes in the score-per-byte
//     mode; sort key = ~bits(score), so ascending key order is decreasing score.  Each warp
//     counts the lowest digit of its slice's candidate keys.
//  C  stable LSD radix sort of (key, unit) pairs, four 8-bit digits; the first pass scatters
//     the candidates straight from the unit order, so equal scores stay in ascending unit
//     order; a later digit that is the same for every key is skipped.  A pass is two barriers:
//     every warp counts its slice's digits, and after the barrier every CTA adds up the
//     counts before its own and scatters.  (Up to kRankUnits units: each candidate's position
//     from comparisons with all of them instead, without a barrier.)
//  D  costs in that order: every position before the first prefix sum > B is selected.
//  E  after that first overflow only candidates with cost <= the remaining budget R0 can
//     ever be taken (R only shrinks): every CTA compacts those of its slice while the
//     positions before the overflow enter the mask, the set hash and the counts; then CTA 0
//     runs the greedy with skip over the compacted tail, in order, from shared memory.
//     (A taken fallback unit sets its expert's bit in a per-tensor word, which a last pass
//     ORs into every block of the tensor.)
//  F  CTA 0 computes the digest and writes the summary, also to the host's pinned copy.
//
// What bounds it is latency: a plan of 62 K units touches about 2 MB, in 11 phases.  Two
// launches of the same code: up to kClusterUnits units one thread-block cluster of up to 16 CTAs
// of 1024 threads, whose barrier is the hardware's (about 1 us with what the writes before it
// take, where the cooperative grid's in global memory takes 3 us) and whose CTAs read each
// other's digit counts from shared memory; above, a cooperative grid of one 256-thread CTA per
// SM, because a pass is then bound by the SMs' scattered stores.  Measured, first plan of an
// index / later plan, us: 2,048 units 34 / 15 in the cluster (45 / 15 with the radix sort), 80 / 20 in the grid; 62 K 65 / 22
// and 82 / 23; 384 K 184 / 40 and 114 / 32.  (Before, as 21 phases of the grid alone, with a
// compaction, a scan phase in every pass and one atomic ballot per taken tail candidate:
// 119 / 35 at 2,048 units, 116 / 43 at 62 K, 180 / 70 at 384 K, 1124 / 348 at 3.9 M where it now
// takes 750 / 160.)
#include "mp_internal.cuh"

namespace mp {
namespace {

constexpr uint32_t kMaxGrid = 256;       // upper bound of the cooperative grid (scratch sizing)
constexpr uint32_t kClusterMax = 16;     // CTAs of the cluster launch (non-portable size)
constexpr int kClusterThreads = 1024;    // threads per CTA of the cluster launch
constexpr int kGridThreads = 256;        // threads per CTA of the cooperative launch
constexpr uint64_t kClusterUnits = 1ull << 17;  // most units planned by one cluster
// Most units that are ordered by comparing each with every other (rank_units) instead of by four
// passes of the radix sort, whose barriers and round trips take 5 to 6 us each however few the
// units.  First plan, sort / compare: 400 units 38 / 31 us, 1,000 43 / 29, 2,048 45 / 34, 3,000
// 44 / 39, 4,000 44 / 51.
constexpr uint32_t kRankUnits = 3072;
constexpr uint32_t kBarrierLimit = 1u << 24;

// summary words (plan handle)
enum { S_CHAT = 0, S_NSEL = 1, S_NCAND = 2, S_SETHASH = 3, S_DIGEST = 4, S_TOUCHED = 5, S_ERR = 6 };
// scratch scalars
enum { X_BAR_COUNT = 0, X_BAR_GEN = 1, X_P = 2, X_PBP = 3, X_MISSING = 4, X_TAILMIN = 5, X_COUNT = 16 };

constexpr unsigned long long kNoP = ~0ull;

struct Scratch {
  uint2* kv_a;                  // [U] (key, unit) pairs of the sort: one scattered store each
  uint2* kv_b;                  // [U]
  uint32_t* tail_pos;           // [U] positions of the tail's candidates, compacted per CTA slice
  unsigned long long* tail_cost;  // [U] their costs
  uint32_t* hist;               // [kMaxGrid][256]
  unsigned long long* cta_a;    // [kMaxGrid]
  unsigned long long* cta_b;    // [kMaxGrid]
  unsigned long long* x;        // [X_COUNT]
  uint32_t* pair_flag;          // [K * n_tensors] (fallback only)
  uint32_t* pair_key;           // [K * n_tensors]
  unsigned long long* pair_cost;  // [K * n_tensors]
  uint32_t* sel_bits;           // [n_tensors] experts whose fallback unit of the tensor was taken
};

inline size_t align_up(size_t v) { return (v + 255) & ~(size_t)255; }

size_t carve(void* base, uint64_t U, uint64_t n_pairs, Scratch* s) {
  char* p = static_cast<char*>(base);
  size_t o = 0;
  auto take = [&](size_t bytes) { char* r = p + o; o += align_up(bytes); return r; };
  Scratch t;
  t.kv_a = (uint2*)take(U * 8);
  t.kv_b = (uint2*)take(U * 8);
  t.tail_pos = (uint32_t*)take(U * 4);
  t.tail_cost = (unsigned long long*)take(U * 8);
  t.hist = (uint32_t*)take((size_t)256 * kMaxGrid * 4);
  t.cta_a = (unsigned long long*)take(kMaxGrid * 8);
  t.cta_b = (unsigned long long*)take(kMaxGrid * 8);
  t.x = (unsigned long long*)take(X_COUNT * 8);
  t.pair_flag = (uint32_t*)take(n_pairs * 4);
  t.pair_key = (uint32_t*)take(n_pairs * 4);
  t.pair_cost = (unsigned long long*)take(n_pairs * 8);
  t.sel_bits = (uint32_t*)take(n_pairs * 4);  // n_tensors words used (n_pairs >= n_tensors)
  if (s) *s = t;
  return o;
}

__device__ __forceinline__ uint32_t ties_key(float d) {
  // bits(bf16_rne(|d|)) & 0x7FFF by integer rounding; |d| is finite and non-negative here
  uint32_t u = __float_as_uint(fabsf(d));
  return ((u + 0x7FFFu + ((u >> 16) & 1u)) >> 16) & 0x7FFFu;
}

__device__ __forceinline__ uint64_t splitmix64(uint64_t state) {
  uint64_t z = state + 0x9E3779B97F4A7C15ull;
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}

__device__ __forceinline__ unsigned ld_acquire(const unsigned long long* p) {
  unsigned long long v;
  asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return (unsigned)v;
}

// barrier of the cooperative grid: the last CTA to arrive bumps the generation; the others wait for it with
// a bounded number of polls.  Returns false (uniformly inside the CTA) if the wait expired: the CTA then
// returns, and as the host's copy of the summary is otherwise written at the very end only, the error
// word goes there too.
__device__ __forceinline__ bool grid_sync(const PlanLaunch& p, unsigned long long* x, unsigned& gen) {
  __shared__ int s_ok;
  __syncthreads();
  if (threadIdx.x == 0) {
    int ok = 1;
    const unsigned target = gen + 1;
    __threadfence();
    if (atomicAdd(&x[X_BAR_COUNT], 1ull) == (unsigned long long)(gridDim.x - 1)) {
      x[X_BAR_COUNT] = 0;
      __threadfence();
      atomicExch(&x[X_BAR_GEN], (unsigned long long)target);
    } else {
      const uint32_t limit = p.wait_limit ? p.wait_limit : kBarrierLimit;
      uint32_t k = 0;
      while (ld_acquire(&x[X_BAR_GEN]) != target) {
        if (++k > limit) {
          ok = 0;
          atomicOr((unsigned long long*)&p.summary[S_ERR], (unsigned long long)kErrTimeout);
          if (p.host_summary) *(volatile uint64_t*)&p.host_summary[S_ERR] = (uint64_t)kErrTimeout;
          break;
        }
        __nanosleep(32);
      }
    }
    __threadfence();
    gen = target;
    s_ok = ok;
  }
  __syncthreads();
  return s_ok != 0;
}

// barrier of the cluster: every thread arrives, and what any of them wrote before is visible
// to all of them after.  No limit is needed: the CTAs of a cluster run at the same time, and the hardware
// waits for the threads that have not exited, all of which come here or exit.
__device__ __forceinline__ void cluster_sync() {
  __syncwarp();
  asm volatile("barrier.cluster.arrive.release.aligned;\n barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// the barrier between phases; false (uniformly inside the CTA) when the wait expired
template <bool CL>
__device__ __forceinline__ bool phase_sync(const PlanLaunch& p, unsigned long long* x, unsigned& gen) {
  if constexpr (CL) {
    cluster_sync();
    return true;
  } else {
    return grid_sync(p, x, gen);
  }
}

// block-wide exclusive scan (PT threads) with total
template <int PT, typename T>
__device__ __forceinline__ T block_scan(T v, T& total) {
  __shared__ T s_w[PT / 32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  T x = v;
#pragma unroll
  for (int s = 1; s < 32; s <<= 1) {
    T y = __shfl_up_sync(0xFFFFFFFFu, x, s);
    if (lane >= s) x += y;
  }
  if (lane == 31) s_w[warp] = x;
  __syncthreads();
  if (warp == 0) {
    T t = lane < PT / 32 ? s_w[lane] : T(0);
#pragma unroll
    for (int s = 1; s < PT / 32; s <<= 1) {
      T y = __shfl_up_sync(0xFFFFFFFFu, t, s);
      if (lane >= s) t += y;
    }
    if (lane < PT / 32) s_w[lane] = t;
  }
  __syncthreads();
  const T before = warp > 0 ? s_w[warp - 1] : T(0);
  total = s_w[PT / 32 - 1];
  __syncthreads();
  return before + x - v;
}

template <int PT, typename T>
__device__ __forceinline__ T block_sum(T v) {
  T t;
  block_scan<PT, T>(v, t);
  return t;
}

// sums of a[0..c) and a[0..n), by every warp for itself
__device__ __forceinline__ unsigned long long warp_prefix(const unsigned long long* a, uint32_t c, uint32_t n,
                                                          unsigned long long& total) {
  unsigned long long t = 0, v = 0;
  for (uint32_t k = threadIdx.x & 31u; k < n; k += 32) {
    const unsigned long long x = a[k];
    t += x;
    v += k < c ? x : 0ull;
  }
#pragma unroll
  for (int sh = 16; sh > 0; sh >>= 1) {
    t += __shfl_xor_sync(0xFFFFFFFFu, t, sh);
    v += __shfl_xor_sync(0xFFFFFFFFu, v, sh);
  }
  total = t;
  return v;
}

struct Unit {
  bool cand;
  uint32_t key;
  bool missing;  // no statistics and no fallback
};

__device__ __forceinline__ Unit score_unit(const PlanLaunch& p, const Scratch& s, uint32_t u) {
  const uint32_t b = u / p.K;
  const uint32_t i = u - b * p.K;
  const uint64_t st = (uint64_t)i * p.n_blocks + b;
  if (p.fallback) {
    const uint32_t t = p.blk_tensor[b];
    const uint32_t pr = i * p.n_tensors + t;
    if (s.pair_flag[pr]) return Unit{b == p.t_blk0[t], s.pair_key[pr], false};
  }
  const uint32_t nz = p.nnz[st];
  bool cand = nz != 0u && nz != kNnzMissing;
  if (cand && p.op_kind == MP_OP_TIES)
    cand = ties_key(p.maxabs[st]) >= p.tau[(uint64_t)i * p.n_groups + p.blk_group[b]];
  float score = __fmul_rn(p.coef[i], p.norm[st]);
  // score per byte: one IEEE division by the block's byte cost (exact in fp32, <= 2^20)
  if (p.score_mode) score = __fdiv_rn(score, (float)(p.blk_len[b] * p.elem_size));
  return Unit{cand, ~__float_as_uint(score), !p.fallback && nz == kNnzMissing};
}

__device__ __forceinline__ unsigned long long unit_cost(const PlanLaunch& p, const Scratch& s, uint32_t u) {
  const uint32_t b = u / p.K;
  if (p.fallback) {
    const uint32_t pr = (u % p.K) * p.n_tensors + p.blk_tensor[b];
    if (s.pair_flag[pr]) return s.pair_cost[pr];
  }
  return (unsigned long long)p.blk_len[b] * p.elem_size;
}

// phase 0b for one flagged pair (i, t), by one warp: cost = the tensor's bytes, key from
// |coef_i| * sqrt(ss), ss the fp32 chain fma(n, n, ss) over the known blocks in block order.
// The lanes load a batch of kFbChunks chunks of 32 consecutive entries at once (one load
// latency per batch); every lane then runs the same chain over them in block order.
constexpr int kFbChunks = 8;

__device__ __forceinline__ void fallback_pair(const PlanLaunch& p, const Scratch& s, uint32_t pr, uint32_t lane) {
  const uint32_t i = pr / p.n_tensors, t = pr % p.n_tensors;
  const uint32_t b0 = p.t_blk0[t], b1 = p.t_blk0[t + 1];
  const float* nrm = p.norm + (uint64_t)i * p.n_blocks;
  const uint32_t* nz = p.nnz + (uint64_t)i * p.n_blocks;
  float ss = 0.0f;
  unsigned long long cost = 0;
  for (uint32_t bb = b0; bb < b1; bb += 32u * kFbChunks) {
    float n[kFbChunks];
    bool known[kFbChunks];
#pragma unroll
    for (int c = 0; c < kFbChunks; ++c) {
      const uint32_t b = bb + 32u * c + lane;
      n[c] = 0.0f;
      known[c] = false;
      if (b < b1) {
        n[c] = __ldg(nrm + b);
        known[c] = __ldg(nz + b) != kNnzMissing;
        cost += (unsigned long long)__ldg(p.blk_len + b) * p.elem_size;
      }
    }
#pragma unroll
    for (int c = 0; c < kFbChunks; ++c) {
      // an entry without statistics adds fma(0, 0, ss) = ss exactly (ss >= +0)
      const float nv = known[c] ? n[c] : 0.0f;
#pragma unroll
      for (int j = 0; j < 32; ++j) {
        const float nj = __shfl_sync(0xFFFFFFFFu, nv, j);
        ss = __fmaf_rn(nj, nj, ss);
      }
    }
  }
#pragma unroll
  for (int sh = 16; sh > 0; sh >>= 1) cost += __shfl_xor_sync(0xFFFFFFFFu, cost, sh);
  float score = __fmul_rn(p.coef[i], __fsqrt_rn(ss));
  if (p.score_mode) score = __fdiv_rn(score, __ull2float_rn(cost));
  if (lane == 0) {
    s.pair_key[pr] = ~__float_as_uint(score);
    s.pair_cost[pr] = cost;
  }
}

// elements of n that each warp of the grid takes: whole tiles of 32, so that few lanes idle
template <int PT>
__device__ __forceinline__ uint32_t slice_len(uint32_t n) {
  const uint32_t parts = gridDim.x * (PT / 32);
  const uint32_t tiles = n / 32u + (n % 32u ? 1u : 0u);
  return (tiles / parts + (tiles % parts ? 1u : 0u)) * 32u;
}

// the first element of slice k of n elements cut into slices of len
__device__ __forceinline__ uint32_t slice_begin(uint32_t n, uint32_t len, uint32_t k) {
  return (uint32_t)min((uint64_t)len * k, (uint64_t)n);
}

// what a thread has put into the mask: added up over the CTA by add_selected
struct Selected {
  unsigned long long hash = 0, n = 0, touched = 0;
};

__device__ __forceinline__ void select_unit(const PlanLaunch& p, const Scratch& s, uint32_t u, Selected& sel) {
  if (kChecked && (uint64_t)u >= p.n_blocks * p.K) {  // checked build: a unit id past U
    atomicOr((unsigned long long*)&p.summary[S_ERR], (unsigned long long)kErrBounds);
    return;
  }
  const uint32_t b = u / p.K, i = u - b * p.K;
  const uint32_t t = p.fallback ? p.blk_tensor[b] : 0u;
  if (p.fallback && s.pair_flag[i * p.n_tensors + t]) {
    atomicOr(&s.sel_bits[t], 1u << i);  // every block of t gets bit i in the last pass
  } else {
    sel.touched += atomicOr(&p.mask[b], 1u << i) == 0u ? 1ull : 0ull;
  }
  sel.hash += splitmix64(u);
  ++sel.n;
}

__device__ __forceinline__ unsigned long long warp_sum(unsigned long long v) {
#pragma unroll
  for (int sh = 16; sh > 0; sh >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, sh);
  return v;
}

// adds a CTA's selections to the summary (the last pass counts the touched blocks when
// fallback units put whole tensors into the mask)
template <int PT>
__device__ __forceinline__ void add_selected(const PlanLaunch& p, const Selected& sel) {
  __shared__ unsigned long long s_sel[3][PT / 32];
  const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
  const unsigned long long v[3] = {warp_sum(sel.hash), warp_sum(sel.n), warp_sum(sel.touched)};
  if (lane < 3) s_sel[lane][warp] = lane == 0 ? v[0] : (lane == 1 ? v[1] : v[2]);
  __syncthreads();
  if (warp >= 3) return;  // warp k adds up value k
  const unsigned long long t = warp_sum(lane < PT / 32 ? s_sel[warp][lane] : 0ull);
  if (lane != 0 || t == 0) return;
  if (warp == 0) atomicAdd((unsigned long long*)&p.summary[S_SETHASH], t);
  else if (warp == 1) atomicAdd((unsigned long long*)&p.summary[S_NSEL], t);
  else if (!p.fallback) atomicAdd((unsigned long long*)&p.summary[S_TOUCHED], t);
}

// inclusive scan over the warp
__device__ __forceinline__ unsigned long long warp_scan(unsigned long long v, uint32_t lane) {
#pragma unroll
  for (int sh = 1; sh < 32; sh <<= 1) {
    const unsigned long long o = __shfl_up_sync(0xFFFFFFFFu, v, sh);
    if ((int)lane >= sh) v += o;
  }
  return v;
}

// lanes of `who` whose digit d (8 bits) equals this lane's
__device__ __forceinline__ uint32_t same_digit(uint32_t d, uint32_t who) {
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    const bool bit = (d >> k) & 1u;
    const uint32_t v = __ballot_sync(0xFFFFFFFFu, bit);
    who &= bit ? v : ~v;
  }
  return who;
}

// the digit counts of CTA g of the cluster, in its shared memory
__device__ __forceinline__ uint32_t peer_count(const uint32_t* own, uint32_t g) {
  uint32_t a, v;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"((uint32_t)__cvta_generic_to_shared(own)), "r"(g));
  asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(v) : "r"(a) : "memory");
  return v;
}

// A and C for up to kRankUnits units: every CTA of the cluster scores all of them and compacts the
// candidates in its shared memory (mem, 32 KiB), and a candidate's position in the order is the
// number of candidates with a smaller key, or an equal one before it.  The CTAs share the
// candidates in runs of 32, a run's warps share the keys it is compared with.  Writes the order;
// Q is the number of candidates.  The caller's barrier follows.
template <int PT>
__device__ __forceinline__ void rank_units(const PlanLaunch& p, const Scratch& s, uint32_t U, uint32_t* mem,
                                           uint32_t& Q) {
  constexpr uint32_t W = PT / 32, R = kRankUnits / PT;
  static_assert(kRankUnits % PT == 0 && kRankUnits <= 65536, "runs of R units per thread, 16-bit unit numbers");
  static_assert(kRankUnits * 6 + PT * 4 <= W * 1024, "keys, units and positions fit the digit counters' memory");
  uint32_t* s_key = mem;                                             // [kRankUnits]
  uint16_t* s_unit = reinterpret_cast<uint16_t*>(mem + kRankUnits);  // [kRankUnits]
  uint32_t* s_pos = mem + kRankUnits + kRankUnits / 2;               // [PT] of this CTA's candidates
  const uint32_t tid = threadIdx.x, lane = tid & 31u, warp = tid >> 5, G = gridDim.x, c = blockIdx.x;
  const uint32_t r = (U + PT - 1) / PT, u0 = tid * r;  // this thread's units u0 .. u0 + r - 1
  uint32_t key[R], n = 0;
  bool cand[R], miss = false;
#pragma unroll
  for (uint32_t e = 0; e < R; ++e) {
    cand[e] = false;
    if (e < r && u0 + e < U) {
      const Unit x = score_unit(p, s, u0 + e);
      miss |= x.missing;
      key[e] = x.key;
      cand[e] = x.cand;
      n += x.cand ? 1u : 0u;
    }
  }
  uint32_t at = block_scan<PT, uint32_t>(n, Q);
#pragma unroll
  for (uint32_t e = 0; e < R; ++e)
    if (cand[e]) {
      s_key[at] = key[e];
      s_unit[at++] = (uint16_t)(u0 + e);
    }
  if (tid < 3 && Q + tid < kRankUnits) s_key[Q + tid] = 0xFFFFFFFFu;  // below no key: whole vectors of keys
  s_pos[tid] = 0u;
  if (c == 0 && miss) s.x[X_MISSING] = 1ull;  // cleared by this CTA before the scan
  __syncthreads();
  const uint32_t runs = (Q + 31u) / 32u, per = (runs + G - 1) / G, g0 = c * per;
  const uint32_t mine = g0 < runs ? min(per, runs - g0) : 0u;  // at most W (launch_plan)
  if (mine != 0u) {
    const uint32_t share = W / mine, g = warp / share, part = warp % share;
    if (g < mine) {
      const uint32_t i0 = (g0 + g) * 32u, i = i0 + lane;
      const uint32_t ki = i < Q ? s_key[i] : 0u;
      const uint32_t step = ((Q + share - 1) / share + 3u) & ~3u;
      const uint32_t j0 = min(part * step, Q), j1 = min(j0 + step, Q);
      uint32_t k = 0;
      const uint4* v = reinterpret_cast<const uint4*>(s_key);
#pragma unroll 4
      for (uint32_t j = j0; j < min(j1, i0); j += 4) {  // before the run: equal keys come first
        const uint4 q = v[j / 4u];
        k += (q.x <= ki) + (q.y <= ki) + (q.z <= ki) + (q.w <= ki);
      }
      for (uint32_t j = max(j0, i0); j < min(j1, i0 + 32u); ++j) k += s_key[j] < ki || (s_key[j] == ki && j < i);
#pragma unroll 4
      for (uint32_t j = max(j0, i0 + 32u); j < j1; j += 4) {
        const uint4 q = v[j / 4u];
        k += (q.x < ki) + (q.y < ki) + (q.z < ki) + (q.w < ki);
      }
      if (k) atomicAdd(&s_pos[g * 32u + lane], k);
    }
  }
  __syncthreads();
  if (tid < mine * 32u && g0 * 32u + tid < Q) {
    const uint32_t pos = s_pos[tid], u = s_unit[g0 * 32u + tid];
    if (kChecked && pos >= U) {  // checked build: a position past U
      atomicOr((unsigned long long*)&p.summary[S_ERR], (unsigned long long)kErrBounds);
      return;
    }
    p.order[pos] = u;
    if (p.cache_order_out) p.cache_order_out[pos] = u;
  }
}

template <int PT, bool CL>
__global__ void __launch_bounds__(PT, 1) plan_kernel(const PlanLaunch p, Scratch s) {
  constexpr int W = PT / 32;
  constexpr uint32_t kTailChunk = W * 128;  // tail costs held at once, in the digit counters' memory
  constexpr int kHold = 4;                  // tiles of a warp's slice whose keys stay in registers
  __shared__ __align__(16) uint32_t s_cnt[W][256];
  __shared__ uint32_t s_hist[256];
  __shared__ unsigned long long s_wsum[W];
  __shared__ uint32_t s_take[kTailChunk / 32];
  __shared__ uint32_t s_pre[kMaxGrid + 1];
  __shared__ unsigned long long s_bcast;
  unsigned long long* s_cost = reinterpret_cast<unsigned long long*>(&s_cnt[0][0]);
  const uint32_t tid = threadIdx.x, lane = tid & 31u, warp = tid >> 5;
  const uint32_t G = gridDim.x, c = blockIdx.x;
  const uint32_t gt = c * PT + tid, gn = G * PT;  // this thread of the grid's threads
  const uint32_t gw = c * W + warp;               // this warp of the grid's warps
  const uint32_t U = (uint32_t)((uint64_t)p.K * p.n_blocks);  // below 2^32 (launch_plan)
  const uint32_t lt = (1u << lane) - 1u;
  unsigned gen = 0;

  // ---- zero the outputs and the scalars (first used after a barrier) ----
  for (uint64_t k = gt; k < p.n_blocks; k += gn) p.mask[k] = 0u;
  if (c == 0 && tid < 8) p.summary[tid] = 0;
  if (c == 0 && tid == 0) {
    s.x[X_P] = kNoP;
    s.x[X_TAILMIN] = ~0ull;
    s.x[X_MISSING] = 0;
    if (p.cache_q_out) *p.cache_q_out = ~0ull;  // an invalid count until the sort is complete
  }
  // test hook: this CTA never comes to a barrier.  Its share of the mask is zero by now, as that of a CTA
  // which gives up is: a mask that was not finished selects some units or none, never an expert past K
  if (!CL && p.stall && c == 1) return;
  bool bad_order = false, miss = false;
  uint32_t Q = 0, len = 0, a = 0, b = 0;  // candidates; this warp's slice [a, b) of them
  auto own_slice = [&](uint32_t q) {
    Q = q;
    len = slice_len<PT>(q);
    a = slice_begin(q, len, gw);
    b = slice_begin(q, len, gw + 1);
  };
  if (p.cache_q_in) {
    // the candidates in traversal order from an earlier plan of this index and operator:
    // phases 0 to C depend on the operator and the catalog, not on the budget
    const unsigned long long q = *p.cache_q_in;
    bad_order = q > U;  // the plan that was to leave the order did not finish: report, plan nothing
    own_slice(bad_order ? 0u : (uint32_t)q);
    for (uint64_t j = a + lane; j < b; j += 32) p.order[j] = p.cache_order_in[j];
    __syncwarp();  // the warp reads its own slice of the order below
  } else {
    const uint32_t ul = slice_len<PT>(U), ua = slice_begin(U, ul, gw), ub = slice_begin(U, ul, gw + 1);
    if (p.fallback) {
      const uint32_t n_pairs = p.K * p.n_tensors;
      for (uint32_t k = gt; k < n_pairs; k += gn) s.pair_flag[k] = 0u;
      for (uint32_t k = gt; k < p.n_tensors; k += gn) s.sel_bits[k] = 0u;
      if (!phase_sync<CL>(p, s.x, gen)) return;
      // 0a: flag the pairs holding an entry without statistics (one atomic per pair and warp)
      for (uint64_t t0 = ua; t0 < ub; t0 += 32) {
        const uint64_t u = t0 + lane;
        uint32_t pr = 0xFFFFFFFFu;
        if (u < ub) {
          const uint32_t bb = (uint32_t)u / p.K, i = (uint32_t)u - bb * p.K;
          if (p.nnz[(uint64_t)i * p.n_blocks + bb] == kNnzMissing) pr = i * p.n_tensors + p.blk_tensor[bb];
        }
        const uint32_t peers = __match_any_sync(0xFFFFFFFFu, pr);
        if (pr != 0xFFFFFFFFu && lane == (uint32_t)(__ffs(peers) - 1)) atomicOr(&s.pair_flag[pr], 1u);
      }
      if (!phase_sync<CL>(p, s.x, gen)) return;
      // 0b: the flagged pairs' units, one warp each
      for (uint32_t pr = gw; pr < n_pairs; pr += G * W)
        if (s.pair_flag[pr]) fallback_pair(p, s, pr, lane);
      if (!phase_sync<CL>(p, s.x, gen)) return;
    }

    bool ranked = false;
    if constexpr (CL) {
      if (U <= kRankUnits) {
        rank_units<PT>(p, s, U, &s_cnt[0][0], Q);
        own_slice(Q);
        if (p.cache_q_out && gt == 0) *p.cache_q_out = Q;
        if (!phase_sync<CL>(p, s.x, gen)) return;
        ranked = true;
      }
    }
    // ---- A and C: candidates, then a stable LSD radix sort by 8-bit digits ----
    // Pass 0 takes the candidates of this warp's slice of the units, later passes its slice of
    // the pass before; the first kHold tiles' keys stay in registers from count to scatter.
    const uint2* in = nullptr;
    uint2* out = s.kv_a;
    bool ordered = false;  // the last pass has put the units into p.order
    for (uint32_t pass = 0; pass < 4 && !ranked; ++pass) {
      const uint32_t shift = 8u * pass;
      const uint64_t r0 = pass == 0 ? ua : a, r1 = pass == 0 ? ub : b;
      auto load = [&](uint64_t j, uint32_t& key, uint32_t& val) -> bool {  // false: no candidate
        if (j >= r1) return false;
        if (pass > 0) {
          const uint2 kv = in[j];
          key = kv.x;
          val = kv.y;
          return true;
        }
        const Unit x = score_unit(p, s, (uint32_t)j);
        // without the fallback an entry lacking statistics cannot be planned: it is reported
        miss |= x.missing;
        key = x.key;
        val = (uint32_t)j;
        return x.cand;
      };
      for (uint32_t k = lane; k < 256u; k += 32) s_cnt[warp][k] = 0u;
      __syncwarp();
      uint32_t hk[kHold], hv[kHold];
      uint32_t hvalid = 0u;
#pragma unroll
      for (int t = 0; t < kHold; ++t)
        if (load(r0 + 32u * t + lane, hk[t], hv[t])) hvalid |= 1u << t;
#pragma unroll
      for (int t = 0; t < kHold; ++t)
        if ((hvalid >> t) & 1u) atomicAdd(&s_cnt[warp][(hk[t] >> shift) & 255u], 1u);
#pragma unroll 4
      for (uint64_t j = r0 + 32u * kHold + lane; j < r1; j += 32) {
        uint32_t key, val;
        if (load(j, key, val)) atomicAdd(&s_cnt[warp][(key >> shift) & 255u], 1u);
      }
      __syncthreads();
      if (tid < 256u) {
        uint32_t n = 0;
#pragma unroll
        for (int w = 0; w < W; ++w) n += s_cnt[w][tid];
        if constexpr (CL) s_hist[tid] = n;
        else s.hist[(uint64_t)c * 256u + tid] = n;
      }
      if (!phase_sync<CL>(p, s.x, gen)) return;
      // digit starts, the counts of the CTAs before this one, then each warp's start
      uint32_t before = 0, tot = 0;
      if (tid < 256u) {
#pragma unroll 8
        for (uint32_t g = 0; g < G; ++g) {
          const uint32_t v = CL ? peer_count(&s_hist[tid], g) : s.hist[(uint64_t)g * 256u + tid];
          before += g < c ? v : 0u;
          tot += v;
        }
      }
      uint32_t total;
      const uint32_t start = block_scan<PT, uint32_t>(tot, total);
      if (pass == 0) {
        if (miss) s.x[X_MISSING] = 1ull;  // cleared before the barrier
        own_slice(total);
      }
      // one digit holds every key: nothing moves (uniform over the grid: the same totals)
      if (pass > 0 && (__syncthreads_or(tid < 256u && tot == Q) != 0 || Q == 0)) {
        if (!phase_sync<CL>(p, s.x, gen)) return;  // every CTA has read the counts
        continue;
      }
      if (tid < 256u) {
        uint32_t acc = start + before;
#pragma unroll
        for (int w = 0; w < W; ++w) {
          const uint32_t n = s_cnt[w][tid];
          s_cnt[w][tid] = acc;
          acc += n;
        }
      }
      __syncthreads();
      auto scatter = [&](bool valid, uint32_t key, uint32_t val) {
        const uint32_t d = (key >> shift) & 255u;
        const uint32_t peers = same_digit(d, __ballot_sync(0xFFFFFFFFu, valid));
        const uint32_t rank = __popc(peers & lt);
        const uint32_t pos = valid ? s_cnt[warp][d] + rank : 0u;
        __syncwarp();
        if (valid && rank == 0) s_cnt[warp][d] = pos + __popc(peers);
        __syncwarp();
        if (!valid) return;
        if (kChecked && pos >= U) {  // checked build: a slot past U
          atomicOr((unsigned long long*)&p.summary[S_ERR], (unsigned long long)kErrBounds);
          return;
        }
        if (pass < 3) out[pos] = make_uint2(key, val);
        else p.order[pos] = val;  // nobody reads the keys after the last pass
      };
#pragma unroll
      for (int t = 0; t < kHold; ++t)
        if (r0 + 32u * t < r1) scatter((hvalid >> t) & 1u, hk[t], hv[t]);  // uniform over the warp
      for (uint64_t t0 = r0 + 32u * kHold; t0 < r1; t0 += 32) {
        uint32_t key = 0u, val = 0u;
        const bool valid = load(t0 + lane, key, val);
        scatter(valid, key, val);
      }
      if (!phase_sync<CL>(p, s.x, gen)) return;
      ordered = pass == 3;
      in = out;
      out = in == s.kv_a ? s.kv_b : s.kv_a;
    }
    // the sorted units are in p.order unless the last pass was skipped (a uniform fact: every
    // CTA made the same skip decisions)
    if (!ordered && !ranked)
      for (uint64_t j = a + lane; j < b; j += 32) p.order[j] = in[j].y;
    if (p.cache_order_out && !ranked) {  // keep the order for later plans with the same operator
      for (uint64_t j = a + lane; j < b; j += 32) p.cache_order_out[j] = ordered ? p.order[j] : in[j].y;
      if (gt == 0) *p.cache_q_out = Q;
    }
    __syncwarp();  // the warp reads its own slice of the order below
  }
  const uint32_t* order = p.order;

  // ---- D: cost prefix in sorted order; the first position where it exceeds B ----
  {
    unsigned long long sum = 0;
#pragma unroll 4
    for (uint64_t j = a + lane; j < b; j += 32) sum += unit_cost(p, s, order[j]);
    sum = warp_sum(sum);
    if (lane == 0) s_wsum[warp] = sum;
    __syncthreads();
    if (warp == 0) {
      const unsigned long long t = warp_sum(lane < W ? s_wsum[lane] : 0ull);
      if (lane == 0) s.cta_b[c] = t;
    }
  }
  if (!phase_sync<CL>(p, s.x, gen)) return;
  unsigned long long total_cost;
  {
    unsigned long long own;
    unsigned long long run = warp_prefix(s.cta_b, c, G, total_cost) + warp_prefix(s_wsum, warp, W, own);
    // only the warp whose slice holds the crossing walks it (prefixes only grow: it is unique)
    if (run <= p.budget && run + s_wsum[warp] > p.budget) {
      for (uint64_t t0 = a; t0 < b; t0 += 32) {
        const uint64_t j = t0 + lane;
        const unsigned long long cj = j < b ? unit_cost(p, s, order[j]) : 0ull;
        const unsigned long long cum = run + warp_scan(cj, lane);
        const uint32_t over = __ballot_sync(0xFFFFFFFFu, cum > p.budget);
        if (over) {
          if ((int)lane == __ffs(over) - 1) {
            s.x[X_P] = j;
            s.x[X_PBP] = cum - cj;
          }
          break;
        }
        run = __shfl_sync(0xFFFFFFFFu, cum, 31);
      }
    }
  }
  if (!phase_sync<CL>(p, s.x, gen)) return;
  const unsigned long long P = s.x[X_P];
  const unsigned long long pbp = P == kNoP ? 0ull : s.x[X_PBP];
  const unsigned long long R0 = P == kNoP ? 0ull : p.budget - pbp;

  // ---- E: the positions before the overflow are selected; the tail after it is compacted ----
  {
    Selected sel;
    uint32_t cnt = 0;
    const uint32_t n_sel = P == kNoP ? Q : (uint32_t)P;
#pragma unroll 4
    for (uint64_t j = gt; j < n_sel; j += gn) select_unit(p, s, order[j], sel);  // over the whole grid
    add_selected<PT>(p, sel);
    if (P != kNoP) {
      if (b > P)
        for (uint64_t j = a + lane; j < b; j += 32) cnt += (j > P && unit_cost(p, s, order[j]) <= R0) ? 1u : 0u;
#pragma unroll
      for (int sh = 16; sh > 0; sh >>= 1) cnt += __shfl_xor_sync(0xFFFFFFFFu, cnt, sh);
      uint32_t n_cta;
      const uint32_t w0 = block_scan<PT, uint32_t>(lane == 0 ? cnt : 0u, n_cta);
      uint32_t o = slice_begin(Q, len, c * W) + __shfl_sync(0xFFFFFFFFu, w0, 0);
      unsigned long long cmin = ~0ull;
      if (cnt) {
        for (uint64_t t0 = a; t0 < b; t0 += 32) {
          const uint64_t j = t0 + lane;
          const unsigned long long cj = j < b && j > P ? unit_cost(p, s, order[j]) : ~0ull;
          const bool f = cj <= R0;
          const uint32_t m = __ballot_sync(0xFFFFFFFFu, f);
          if (f) {
            s.tail_pos[o + __popc(m & lt)] = (uint32_t)j;
            s.tail_cost[o + __popc(m & lt)] = cj;
            cmin = cj < cmin ? cj : cmin;
          }
          o += __popc(m);
        }
#pragma unroll
        for (int sh = 16; sh > 0; sh >>= 1) {
          const unsigned long long v = __shfl_xor_sync(0xFFFFFFFFu, cmin, sh);
          cmin = v < cmin ? v : cmin;
        }
        if (lane == 0) atomicMin(&s.x[X_TAILMIN], cmin);
      }
      if (tid == 0) s.cta_a[c] = n_cta;
    }
  }
  if (!phase_sync<CL>(p, s.x, gen)) return;
  unsigned long long tail_sum = 0;
  if (c == 0 && P != kNoP) {
    // greedy with skip over the compacted tail, in order, from shared memory; once R is
    // below the smallest tail cost nothing more can be taken
    Selected sel;
    uint32_t L;
    {
      const uint32_t v = tid < G ? (uint32_t)s.cta_a[tid] : 0u;
      const uint32_t e = block_scan<PT, uint32_t>(v, L);
      if (tid < G) s_pre[tid] = e;
      if (tid == 0) s_pre[G] = L;
      __syncthreads();
    }
    // slot of the k-th tail candidate: in the slice of the last CTA with s_pre <= k
    auto slot = [&](uint32_t k) -> uint32_t {
      uint32_t lo = 0, hi = G;  // s_pre[lo] <= k < s_pre[hi]
      while (hi - lo > 1) {
        const uint32_t mid = (lo + hi) >> 1;
        if (s_pre[mid] <= k) lo = mid;
        else hi = mid;
      }
      return slice_begin(Q, len, lo * W) + (k - s_pre[lo]);
    };
    const unsigned long long cmin = __ldcg(&s.x[X_TAILMIN]);
    unsigned long long R = R0;
    for (uint32_t k0 = 0; k0 < L && R >= cmin; k0 += kTailChunk) {
      const uint32_t n = min(kTailChunk, L - k0);
      unsigned long long sum = 0;
      for (uint32_t k = tid; k < n; k += PT) {
        const unsigned long long ck = __ldcg(s.tail_cost + slot(k0 + k));
        s_cost[k] = ck;
        sum += ck <= R ? ck : 0ull;
      }
      sum = block_sum<PT, unsigned long long>(sum);
      if (sum <= R) {  // everything that fits now fits together
        for (uint32_t k = tid; k < n; k += PT)
          if (s_cost[k] <= R) select_unit(p, s, order[__ldcg(s.tail_pos + slot(k0 + k))], sel);
        R -= sum;
        __syncthreads();  // the next chunk overwrites s_cost
        continue;
      }
      if (warp == 0) {
        for (uint32_t b0 = 0; b0 < n; b0 += 32) {
          const uint32_t k = b0 + lane;
          const unsigned long long ck = k < n ? s_cost[k] : ~0ull;
          uint32_t taken = 0u, rem = 0xFFFFFFFFu;
          // R only shrinks, so what does not fit now never will; of what fits now, everything
          // up to the first whose prefix exceeds R is taken, that one is skipped, and the
          // lanes after it are looked at again
          while (rem) {
            const bool e = ((rem >> lane) & 1u) && ck <= R;
            const uint32_t fit = __ballot_sync(0xFFFFFFFFu, e);
            if (fit == 0u) break;
            const unsigned long long v = e ? ck : 0ull, cum = warp_scan(v, lane);
            const uint32_t over = __ballot_sync(0xFFFFFFFFu, e && cum > R);
            if (over == 0u) {
              taken |= fit;
              R -= __shfl_sync(0xFFFFFFFFu, cum, 31);
              break;
            }
            const int f = __ffs(over) - 1;
            taken |= fit & ((1u << f) - 1u);
            R -= __shfl_sync(0xFFFFFFFFu, cum - v, f);
            rem &= f == 31 ? 0u : ~((2u << f) - 1u);
          }
          if (lane == 0) s_take[b0 / 32] = taken;
        }
        if (lane == 0) s_bcast = R;
      }
      __syncthreads();
      R = s_bcast;
      for (uint32_t k = tid; k < n; k += PT)
        if ((s_take[k / 32] >> (k & 31u)) & 1u) select_unit(p, s, order[__ldcg(s.tail_pos + slot(k0 + k))], sel);
      __syncthreads();  // the next chunk overwrites s_cost and s_take
    }
    tail_sum = R0 - R;
    add_selected<PT>(p, sel);
    __syncthreads();  // three warps have added to the summary that thread 0 reads
  }
  if (p.fallback) {
    // a taken fallback unit's expert bit goes into every block of its tensor
    if (!phase_sync<CL>(p, s.x, gen)) return;
    unsigned long long t = 0;
    for (uint64_t k = gt; k < p.n_blocks; k += gn) {
      uint32_t m = p.mask[k];
      const uint32_t sb = s.sel_bits[p.blk_tensor[k]];
      if (sb) {
        m |= sb;
        p.mask[k] = m;  // one thread per block in this pass
      }
      t += m != 0u ? 1ull : 0ull;
    }
    t = block_sum<PT, unsigned long long>(t);
    if (tid == 0 && t) atomicAdd((unsigned long long*)&p.summary[S_TOUCHED], t);
    if (!phase_sync<CL>(p, s.x, gen)) return;
  }
  if (gt != 0) return;
  // ---- F: the digest: FNV-1a 64 over the header (hashed by the host) and C_hat, n_sel, set_hash ----
  __threadfence();
  volatile unsigned long long* sum = (volatile unsigned long long*)p.summary;
  const unsigned long long chat = P == kNoP ? total_cost : pbp + tail_sum;
  const unsigned long long nsel = sum[S_NSEL], sh = sum[S_SETHASH];
  uint64_t h = p.digest_state;
  const unsigned long long tail[3] = {chat, nsel, sh};
  for (int w = 0; w < 3; ++w)
    for (int k = 0; k < 8; ++k) {
      h ^= (tail[w] >> (8 * k)) & 0xFFu;
      h *= 1099511628211ull;
    }
  const unsigned long long err = sum[S_ERR] | (unsigned long long)*p.index_err |
                                 (s.x[X_MISSING] ? (unsigned long long)kErrMissing : 0ull) |
                                 (bad_order ? (unsigned long long)kErrInternal : 0ull);
  const unsigned long long words[8] = {chat, nsel, Q, sh, h, sum[S_TOUCHED], err, 0ull};
  for (int k = 0; k < 8; ++k) {
    sum[k] = words[k];
    if (p.host_summary) p.host_summary[k] = words[k];
  }
}

}  // namespace

size_t plan_scratch_bytes(uint64_t n_units, uint64_t n_pairs) { return carve(nullptr, n_units, n_pairs, nullptr); }

uint64_t plan_digest_state(const uint8_t* header, size_t n) {
  uint64_t h = 14695981039346656037ull;
  for (size_t k = 0; k < n; ++k) {
    h ^= header[k];
    h *= 1099511628211ull;
  }
  return h;
}

cudaError_t launch_plan(const PlanLaunch& p, void* scratch, cudaStream_t st) {
  const uint64_t U = (uint64_t)p.K * p.n_blocks;
  if (U > 0xFFFFFFFFull) return cudaErrorInvalidValue;
  const uint64_t n_pairs = p.fallback ? (uint64_t)p.K * p.n_tensors : 0ull;
  if (p.fallback && (!p.blk_tensor || !p.t_blk0 || n_pairs == 0)) return cudaErrorInvalidValue;
  Scratch s;
  carve(scratch, U, n_pairs, &s);
  cudaError_t e;
  bool cluster = U <= kClusterUnits;
  if (cluster) {
    // half a unit per thread, then more, in one cluster; where the units are compared with one
    // another, 2^16 comparisons per CTA, then more
    uint32_t grid = 1;
    while (grid < kClusterMax && (grid * 512ull < U || (U <= kRankUnits && U * U > (uint64_t)grid << 16))) grid *= 2;
    auto k = plan_kernel<kClusterThreads, true>;
    if ((e = cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1)) != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(kClusterThreads);
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = grid;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    // Up to 16 whole SMs of one GPC, more than a partition of the device or a limit on its SMs may leave
    // this process: without room for the cluster the cooperative grid below plans any number of units.
    int room = 0;
    if ((e = cudaOccupancyMaxActiveClusters(&room, k, &cfg)) != cudaSuccess) {
      cudaGetLastError();
      room = 0;
    }
    cluster = room > 0 && !cluster_refused();
    if (cluster) {
      if ((e = cudaLaunchKernelEx(&cfg, k, p, s)) != cudaSuccess) return e;
      count_launches(1);
      return cudaGetLastError();
    }
  }
  int dev = 0, sms = 0, per_sm = 0;
  auto kern = plan_kernel<kGridThreads, false>;
  if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
  if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
  if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kGridThreads, 0)) != cudaSuccess) return e;
  // at most one CTA per SM, all co-resident
  if (per_sm < 1) return cudaErrorInvalidConfiguration;
  uint64_t grid = (uint64_t)sms;
  if (grid > kMaxGrid) grid = kMaxGrid;
  static_assert(kMaxGrid <= (uint32_t)kGridThreads && kClusterMax <= (uint32_t)kClusterThreads,
                "one thread per CTA where the CTAs' counts are added up");
  if ((e = launch_fill(s.x, 0, X_COUNT * sizeof(unsigned long long), st)) != cudaSuccess) return e;
  PlanLaunch pc = p;
  void* args[] = {&pc, &s};
  if ((e = cudaLaunchCooperativeKernel((const void*)kern, dim3((unsigned)grid), dim3(kGridThreads), args, 0, st)) !=
      cudaSuccess)
    return e;
  count_launches(1);
  return cudaGetLastError();
}

}  // namespace mp
