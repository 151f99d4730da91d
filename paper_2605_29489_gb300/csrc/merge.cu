// Alg. 2 ExecuteMerge on the device: M_A[t,b] = M_0[t,b] + Psi_op(A_{.,t,b}, Delta_{.,t,b})
// (Eq. 4) for every block, reading only the experts the access mask selects.
//
// Pipeline (persistent CTAs, 2 to 4 per SM, 128 or 256 consumer threads + 1 producer warp):
//  * work unit = one chunk of a block (8 KiB for AVG/TA, 4 KiB for TIES/DARE); chunks are
//    handed out dynamically through a global counter, GRAB at a time;
//  * the producer warp takes a grab: its lanes load the chunks' block metadata (and, for
//    TIES, every expert's trim threshold) in parallel, and the counter value of the next grab is
//    requested before this one is issued, so that no fill waits on a global-memory round trip;
//  * it then walks each chunk's fills — the base chunk, then every selected expert's
//    chunk in ascending expert order — and streams each fill into the next slot of a ring
//    of NS shared-memory slots with one cp.async.bulk (TMA 1-D bulk copy), completing on
//    a "full" mbarrier (AVG/TA one per slot, the others one per group of slots); it writes the
//    metadata (chunk, offset, length, mask, TIES threshold) before arming the barrier;
//  * consumers take the fills in the same order: the base fill loads M_0 into registers,
//    each expert fill folds Delta_i into fp32 accumulators, the last fill of a chunk
//    writes the output with 16-byte streaming stores; every consumer thread arrives on the
//    "empty" mbarrier as soon as it has read the slot or the group;
//  * the bytes in flight are the ring (NS slots per CTA), independent of registers and of
//    how many experts a block selects.
// Per element, in the fixed ascending expert order:
//   AVG/TA: acc = fma(alpha_i, delta_i, acc)                          out = M_0 + acc
//   DARE:   delta_i kept by a Philox word >= T, scaled by sigma; then as AVG
//   TIES:   trimmed by tau_i; S, P, N, counts;  m = P/c+ | N/c- | 0;   out = fma(lambda, m, M_0)
//   renormalised AVG (App. A.1): as AVG with alpha_i / (sum of alpha over the experts that are
//           selected or have an exactly zero delta block, known from the catalog)
//   DARE-TIES: DARE's keep and rescale, then TIES's election and mean without trimming
// An omitted expert contributes exactly zero to every accumulator, so skipping it equals
// reading a zero-completed tuple (App. A.1) and it is never dereferenced; a chunk that
// selects no expert is M_0 plus the zero the operator adds, or, in the touched-only mode
// (Alg. 2 WriteBlockOrReference), not produced at all: the output keeps its contents there.
// Every mbarrier wait is bounded: on expiry the CTA records kErrTimeout, stops, waits
// (bounded) for its own copies in flight and returns.
#include <cuda_bf16.h>

#include <type_traits>

#include "mp_internal.cuh"
#include "philox.cuh"
#include "small_div.cuh"
#include "tma.cuh"

namespace mp {
namespace {

constexpr uint32_t kEnd = 0xFFFFFFFFu;

enum { OP_ADD = 0, OP_TIES = 1, OP_DARE = 2, OP_RENORM = 3, OP_DTIES = 4 };

// TIES and DARE-TIES share the sign election and disjoint mean (DARE and DARE-TIES share
// the random keep mask)
template <int OPC>
constexpr bool kTiesLike = OPC == OP_TIES || OPC == OP_DTIES;

// slot geometry of the streaming kernel (AVG/TA and the renormalised AVG), which is bound by
// HBM: two CTAs per SM with a 96 KiB ring each (two 16-byte vectors per consumer thread and fill)
struct Geo {
  static constexpr int kConsumers = 256;
  static constexpr int kThreads = kConsumers + 32;  // + one producer warp
  static constexpr int kCtasPerSm = 2;
  static constexpr uint32_t kSlotBytes = 8192u;  // one chunk of one checkpoint
  static constexpr int kSlots = 12;
  static constexpr uint32_t kGrab = 8;  // most chunks taken per counter increment (<= 32)
};

struct SlotMeta {
  uint64_t off;   // element offset of the chunk in the flat buffers
  uint32_t q;     // chunk id, or kEnd
  uint32_t n;     // elements in the chunk
  uint32_t m;     // the block's access mask
  uint32_t aux;   // renormalised AVG: the experts counted in the normaliser (selected or with a
                  // zero delta block)
};

// block metadata of one chunk of a grab, staged by the producer warp
struct ChunkMeta {
  uint64_t off;  // element offset of the chunk
  uint32_t n;    // elements (0: nothing to do)
  uint32_t m;    // access mask
};

template <int NS, uint32_t SB, uint32_t G>
struct __align__(128) Smem {
  uint8_t slot[NS][SB];
  SlotMeta meta[NS];
  ChunkMeta chunk[G];
  uint32_t zmask[G];       // renormalised AVG: experts whose delta block is exactly zero
  uint64_t full[NS];
  uint64_t empty[NS];
  unsigned long long realized[kMaxK];
  int abort, last;
};

// packed fp32x2 arithmetic (two independent IEEE round-to-nearest operations per
// instruction): (d0, d1) = (a0 op b0, a1 op b1)
__device__ __forceinline__ void f2_sub(float a0, float a1, float b0, float b1, float& d0, float& d1) {
  asm("{\n .reg .b64 ra, rb, rd;\n mov.b64 ra, {%2, %3};\n mov.b64 rb, {%4, %5};\n sub.rn.f32x2 rd, ra, rb;\n"
      " mov.b64 {%0, %1}, rd;\n}"
      : "=f"(d0), "=f"(d1)
      : "f"(a0), "f"(a1), "f"(b0), "f"(b1));
}

__device__ __forceinline__ void f2_mul(float a0, float a1, float b0, float b1, float& d0, float& d1) {
  asm("{\n .reg .b64 ra, rb, rd;\n mov.b64 ra, {%2, %3};\n mov.b64 rb, {%4, %5};\n mul.rn.f32x2 rd, ra, rb;\n"
      " mov.b64 {%0, %1}, rd;\n}"
      : "=f"(d0), "=f"(d1)
      : "f"(a0), "f"(a1), "f"(b0), "f"(b1));
}

__device__ __forceinline__ void f2_add(float a0, float a1, float b0, float b1, float& d0, float& d1) {
  asm("{\n .reg .b64 ra, rb, rd;\n mov.b64 ra, {%2, %3};\n mov.b64 rb, {%4, %5};\n add.rn.f32x2 rd, ra, rb;\n"
      " mov.b64 {%0, %1}, rd;\n}"
      : "=f"(d0), "=f"(d1)
      : "f"(a0), "f"(a1), "f"(b0), "f"(b1));
}

// (d0, d1) = (a0 * b0 + c0, a1 * b1 + c1), each a single fused rounding
__device__ __forceinline__ void f2_fma(float a0, float a1, float b0, float b1, float c0, float c1, float& d0,
                                       float& d1) {
  asm("{\n .reg .b64 ra, rb, rc, rd;\n mov.b64 ra, {%2, %3};\n mov.b64 rb, {%4, %5};\n mov.b64 rc, {%6, %7};\n"
      " fma.rn.f32x2 rd, ra, rb, rc;\n mov.b64 {%0, %1}, rd;\n}"
      : "=f"(d0), "=f"(d1)
      : "f"(a0), "f"(a1), "f"(b0), "f"(b1), "f"(c0), "f"(c1));
}

// The TIES trim compares the 15-bit key bits(bf16_rne(|d|)) & 0x7FFF with tau.  For
// |d| >= 0 the key reaches tau >= 1 exactly when bits(|d|) >= (tau << 16) - 0x8000 +
// (tau & 1): the halfway point below tau rounds up to tau only when tau is even.  tau = 0
// keeps everything; tau = 0x8000 ("keep nothing") gives 0x7FFF8000, a NaN pattern, so a
// float compare against it is never true.
__host__ __device__ __forceinline__ uint32_t ties_bits_threshold(uint32_t tau) {
  return tau == 0u ? 0u : (tau << 16) - 0x8000u + (tau & 1u);
}

// bf16 -> fp32: the upper element by a mask, the lower one moved up by a multiply (which runs
// on the FMA pipe and leaves the ALU pipe to the compares)
template <bool BF16>
__device__ __forceinline__ void unpack(const uint4 r, float* x) {
  if constexpr (BF16) {
    x[0] = __uint_as_float(r.x * 65536u);
    x[1] = __uint_as_float(r.x & 0xFFFF0000u);
    x[2] = __uint_as_float(r.y * 65536u);
    x[3] = __uint_as_float(r.y & 0xFFFF0000u);
    x[4] = __uint_as_float(r.z * 65536u);
    x[5] = __uint_as_float(r.z & 0xFFFF0000u);
    x[6] = __uint_as_float(r.w * 65536u);
    x[7] = __uint_as_float(r.w & 0xFFFF0000u);
  } else {
    x[0] = __uint_as_float(r.x);
    x[1] = __uint_as_float(r.y);
    x[2] = __uint_as_float(r.z);
    x[3] = __uint_as_float(r.w);
  }
}

// vector v of a fill: from the slot when inside the bulk-copied bytes, else (the ragged
// tail of a tensor, < 16 bytes) straight from global memory; zeros past the chunk
template <bool BF16>
__device__ __forceinline__ void read_vec(const uint8_t* slot, const void* gsrc, uint64_t off, uint32_t k0,
                                         uint32_t n, uint32_t n_tma, float* x) {
  constexpr uint32_t V = BF16 ? 8u : 4u;
  if (k0 + V <= n_tma) {
    unpack<BF16>(*reinterpret_cast<const uint4*>(slot + k0 * (BF16 ? 2u : 4u)), x);
    return;
  }
#pragma unroll
  for (uint32_t e = 0; e < V; ++e) {
    float v = 0.0f;
    if (k0 + e < n) {
      if constexpr (BF16) v = __uint_as_float((uint32_t)(static_cast<const uint16_t*>(gsrc)[off + k0 + e]) << 16);
      else v = static_cast<const float*>(gsrc)[off + k0 + e];
    }
    x[e] = v;
  }
}

// the raw 16-byte vector at element k0 of a fill, as read_vec reads it (zeros past the chunk)
template <bool BF16>
__device__ __forceinline__ uint4 read_raw(const uint8_t* slot, const void* gsrc, uint64_t off, uint32_t k0,
                                          uint32_t n, uint32_t n_tma) {
  constexpr uint32_t V = BF16 ? 8u : 4u;
  if (k0 + V <= n_tma) return *reinterpret_cast<const uint4*>(slot + k0 * (BF16 ? 2u : 4u));
  uint32_t w[4] = {0u, 0u, 0u, 0u};
#pragma unroll
  for (uint32_t e = 0; e < V; ++e) {
    if (k0 + e < n) {
      if constexpr (BF16) w[e >> 1] |= (uint32_t)(static_cast<const uint16_t*>(gsrc)[off + k0 + e]) << (16u * (e & 1u));
      else w[e] = static_cast<const uint32_t*>(gsrc)[off + k0 + e];
    }
  }
  return make_uint4(w[0], w[1], w[2], w[3]);
}

// the deltas of elements 2k and 2k + 1 of a raw vector against the base elements a and b (k is a
// compile-time index), each one IEEE fp32 subtraction.  bf16 elements are converted by the
// mixed-precision subtract itself (128 lanes per clock and SM): two instructions per pair where
// moving both up to fp32 and a packed subtract take three, two of them at half rate (DARE with 4
// experts 1.436 -> 1.385 ms, TIES with 8 experts 0.851 -> 0.819 ms).
template <bool BF16, int k>
__device__ __forceinline__ void delta_pair(const uint4 r, float a, float b, float& d0, float& d1) {
  if constexpr (BF16) {
    const uint32_t w = k == 0 ? r.x : (k == 1 ? r.y : (k == 2 ? r.z : r.w));
    asm("{\n .reg .b16 l, h;\n mov.b32 {l, h}, %2;\n sub.rn.f32.bf16 %0, l, %3;\n sub.rn.f32.bf16 %1, h, %4;\n}"
        : "=f"(d0), "=f"(d1)
        : "r"(w), "f"(a), "f"(b));
  } else {
    f2_sub(__uint_as_float(k == 0 ? r.x : r.z), __uint_as_float(k == 0 ? r.y : r.w), a, b, d0, d1);
  }
}

// fold(v, d0, d1) for the deltas of elements v and v + 1 of a raw vector, v = 0, 2, ...
template <bool BF16, typename Fold>
__device__ __forceinline__ void delta_pairs(const uint4 r, const float* x0, Fold fold) {
  float d0, d1;
  delta_pair<BF16, 0>(r, x0[0], x0[1], d0, d1);
  fold(0, d0, d1);
  delta_pair<BF16, 1>(r, x0[2], x0[3], d0, d1);
  fold(2, d0, d1);
  if constexpr (BF16) {
    delta_pair<BF16, 2>(r, x0[4], x0[5], d0, d1);
    fold(4, d0, d1);
    delta_pair<BF16, 3>(r, x0[6], x0[7], d0, d1);
    fold(6, d0, d1);
  }
}

// elements e and e + 1 of an output vector into its words: bf16 two per conversion, each rounded
// to nearest-even, element e in the low half
template <bool BF16>
__device__ __forceinline__ void put_pair(uint32_t (&w)[4], int e, float y0, float y1) {
  if constexpr (BF16) {
    const __nv_bfloat162 h2 = __floats2bfloat162_rn(y0, y1);
    w[e >> 1] = *reinterpret_cast<const uint32_t*>(&h2);
  } else {
    w[e] = __float_as_uint(y0);
    w[e + 1] = __float_as_uint(y1);
  }
}

// the tail is unrolled over the vector with a predicate, so that w stays in registers (a loop
// bounded by navail would index it at run time, through local memory)
template <bool BF16>
__device__ __forceinline__ void store_words(void* ptr, uint64_t elem, uint32_t navail, const uint32_t (&w)[4]) {
  constexpr uint32_t V = BF16 ? 8u : 4u, ES = BF16 ? 2u : 4u;
  if (navail >= V) {
    __stcs(reinterpret_cast<uint4*>(static_cast<char*>(ptr) + elem * ES), make_uint4(w[0], w[1], w[2], w[3]));
    return;
  }
#pragma unroll
  for (uint32_t e = 0; e < V; ++e) {
    if (e >= navail) break;
    if constexpr (BF16) static_cast<uint16_t*>(ptr)[elem + e] = (uint16_t)(w[e >> 1] >> (16u * (e & 1u)));
    else static_cast<uint32_t*>(ptr)[elem + e] = w[e];
  }
}

// Checked build: a chunk's block must lie in the launch's block range before the block table
// is read for it, and the chunk (its elements, buffers, alignment, experts and TIES trim
// group) must pass chunk_in_bounds before anything is copied; a failure is recorded in the
// call's error word and the chunk is skipped.  Both are constant true in the default build.
__device__ __forceinline__ bool checked_block(const MergeLaunch& p, uint64_t b) {
  if constexpr (!kChecked) return true;
  if (b >= p.b_begin && b < p.b_end && b < p.n_blocks) return true;
  atomicOr(p.err, kErrBounds);
  return false;
}

template <bool TIES>
__device__ __forceinline__ bool checked_chunk(const MergeLaunch& p, uint64_t b, const ChunkMeta& cm, uint32_t grp,
                                              uint32_t es) {
  if constexpr (!kChecked) return true;
  if (cm.n == 0u) return true;
  if ((!TIES || grp < p.n_groups) &&
      chunk_in_bounds(b, p.b_begin, p.b_end, p.blk_off[b], p.blk_len[b], cm.off, cm.n, cm.m, p.K, es,
                      p.expert_origin, p.ext))
    return true;
  atomicOr(p.err, kErrBounds);
  return false;
}

// DARE keep words: element j of expert i keeps its delta iff 16-bit word j mod 8 of the
// Philox4x32-10 output for counter (j / 8, i, tag) is >= T.  A bf16 vector is exactly the 8 words
// of one call (chunk and tensor offsets are multiples of 8 elements); an fp32 vector is half of
// one.  The experts' share of the first two rounds comes with each group of fills (dare_expert,
// made by the producer; consumers that made it themselves for groups past 2^32 tested for them in
// every call: 10 instructions per vector and expert, 5 % of the DARE merge).
constexpr uint32_t kDareTag = 0x44415245u;

struct DareVec {
  PhiloxGroup grp;
  bool upper;  // fp32: the vector is the upper half of its group
};

__device__ __forceinline__ DareVec dare_vec(uint64_t j0, const MergeLaunch& p) {
  return DareVec{philox_group((uint32_t)(j0 >> 3), kDareTag, p.dare_rk), (j0 & 4u) != 0u};
}

__device__ __forceinline__ uint4 dare_expert(const MergeLaunch& p, uint32_t g_hi, uint32_t i) {
  const PhiloxExpert e = philox_expert(g_hi, i, p.dare_rk);
  return make_uint4(e.x0, e.x2, e.x3, __float_as_uint(p.alpha[i]));
}

// word j mod 8 of element j in the upper half of a 32-bit register: the upper word as it
// stands, the lower one moved up by a multiply (FMA pipe; the ALU pipe is the busy one); it is
// kept iff that register >= T << 16
template <bool BF16>
__device__ __forceinline__ void dare_keep_words(const MergeLaunch& p, const DareVec& v, const uint4 pe,
                                                uint32_t (&kw)[BF16 ? 8 : 4]) {
  constexpr int V = BF16 ? 8 : 4;
  const Philox4 r = philox_finish(v.grp, PhiloxExpert{pe.x, pe.y, pe.z}, p.dare_rk);
#pragma unroll
  for (int k = 0; k < V; ++k) {
    const uint32_t wd = BF16 ? r.w[k >> 1] : (v.upper ? r.w[2 + (k >> 1)] : r.w[k >> 1]);
    kw[k] = (k & 1) ? wd : wd * 65536u;
  }
}

// The end of a merge kernel, reached by every warp of the CTA (a named barrier: the producer
// warp and the consumers come from different places): when all of them are done, so are the
// CTA's realized counts and error bits, and the last CTA of the launch writes the manifest to
// the host's pinned copy.  It replaces two copy kernels after every merge.
template <int THREADS>
__device__ __forceinline__ void merge_end(const MergeLaunch& p, volatile int* s_last) {
  if (!p.back_host) return;
  __syncwarp();
  asm volatile("bar.sync 1, %0;" ::"n"(THREADS) : "memory");
  if (threadIdx.x == 0) {
    __threadfence();
    *s_last = atomicAdd(p.done, 1ull) == (unsigned long long)(gridDim.x - 1) ? 1 : 0;
  }
  asm volatile("bar.sync 1, %0;" ::"n"(THREADS) : "memory");
  if (!*s_last) return;
  __threadfence();
  const uint32_t n = (uint32_t)kCounterSlots * p.K;
  for (uint32_t k = threadIdx.x; k < n + 8u + (uint32_t)kBackTail; k += THREADS)
    p.back_host[k] = k >= n && k < n + 8u ? (unsigned long long)p.back_summary[k - n] : __ldcg(p.realized + k);
}

template <bool BF16, int OPC>
__global__ void __launch_bounds__(Geo::kThreads, Geo::kCtasPerSm)
    merge_tma_kernel(const MergeLaunch p, uint32_t cpb, uint32_t grab, uint64_t n_chunks, unsigned long long* work) {
  kernel_begin();
  static_assert(OPC == OP_ADD || OPC == OP_RENORM, "streaming consumers: AVG/TA and the renormalised AVG");
  constexpr int kConsumers = Geo::kConsumers;
  constexpr uint32_t ES = BF16 ? 2u : 4u;
  constexpr uint32_t SB = Geo::kSlotBytes;
  constexpr int kSlots = Geo::kSlots;
  constexpr uint32_t G = Geo::kGrab;
  constexpr uint32_t CH = SB / ES;  // elements per chunk
  constexpr int V = BF16 ? 8 : 4;
  constexpr int VPT = (int)(CH / (kConsumers * V));  // vectors per consumer thread per chunk
  static_assert(CH == (uint32_t)(kConsumers * VPT * V), "chunk geometry");
  extern __shared__ __align__(128) uint8_t smem_raw[];
  Smem<kSlots, SB, G>& S = *reinterpret_cast<Smem<kSlots, SB, G>*>(smem_raw);
  const uint32_t tid = threadIdx.x, warp = tid >> 5, lane = tid & 31u;
  volatile int* abort_flag = &S.abort;
  const uint32_t wl = wait_limit_of(p.wait_limit);

  if (tid == 0) {
    for (int s = 0; s < kSlots; ++s) {
      mbar_init(&S.full[s], 1);
      mbar_init(&S.empty[s], kConsumers);  // every consumer thread arrives
    }
    S.abort = 0;
    mbar_fence_init();
  }
  if (tid < (uint32_t)kMaxK) S.realized[tid] = 0;
  __syncthreads();

  if (warp == kConsumers / 32) {
    // ---------------- producer ----------------
    uint32_t fill = 0;
    bool ok = true;
    // lane 0 arms slot `fill` with the given chunk data and starts its bulk copy
    auto produce = [&](uint32_t q, uint64_t off, uint32_t n, uint32_t m, uint32_t aux,
                       const char* src_row, uint32_t bytes) -> bool {
      const uint32_t s = fill % kSlots, r = fill / kSlots;
      if (fill == 0 && p.stall) {  // test hook: slot 0 is never armed, so its wait runs out
        ++fill;
        return true;
      }
      if (r > 0 && !mbar_wait<true>(&S.empty[s], (r - 1) & 1u, abort_flag, wl)) return false;
      if (r > 0) fence_proxy_async_smem();
      S.meta[s].off = off;
      S.meta[s].q = q;
      S.meta[s].n = n;
      S.meta[s].m = m;
      S.meta[s].aux = aux;
      mbar_arrive_expect_tx(&S.full[s], bytes);
      if (bytes) tma_load_1d(S.slot[s], src_row, bytes, &S.full[s]);
      ++fill;
      return true;
    };
    unsigned long long q_next = 0;
    if (lane == 0) q_next = atomicAdd(work, (unsigned long long)grab);
    for (;;) {
      const unsigned long long q0 = __shfl_sync(0xFFFFFFFFu, q_next, 0);
      if (q0 >= n_chunks || !ok) break;
      if (lane == 0) q_next = atomicAdd(work, (unsigned long long)grab);  // used by the next grab
      // lanes c < grab: metadata of chunk q0 + c
      uint64_t bq = 0;  // block of chunk q0 + lane
      if (lane < grab) {
        const unsigned long long q = q0 + lane;
        ChunkMeta cm{0, 0, 0};
        if (q < n_chunks && checked_block(p, p.b_begin + q / cpb)) {
          const uint64_t b = p.b_begin + q / cpb;
          bq = b;
          const uint32_t start = (uint32_t)(q % cpb) * CH;
          const uint32_t len = p.blk_len[b];
          cm.off = p.blk_off[b] + start;
          cm.m = p.mask[b];
          cm.n = start < len ? min(CH, len - start) : 0u;
          if (p.touched_only && cm.m == 0u) cm.n = 0u;  // left as it is: a reference to M_0
          if (!checked_chunk<false>(p, b, cm, 0u, ES)) cm.n = 0u;
        }
        S.chunk[lane] = cm;
      }
      if constexpr (OPC == OP_RENORM) {
        // lane i < K: is expert i's delta block exactly zero (catalog nnz = 0)?  Such an
        // expert is counted in the normaliser without being read.
#pragma unroll
        for (uint32_t c = 0; c < G; ++c) {
          const uint64_t b = __shfl_sync(0xFFFFFFFFu, bq, c);
          const bool z = lane < p.K && p.nnz[(uint64_t)lane * p.n_blocks + b] == 0u;
          const uint32_t zb = __ballot_sync(0xFFFFFFFFu, z);
          if (lane == 0) S.zmask[c] = zb;
        }
      }
      __syncwarp();
      if (lane == 0) {
        const uint32_t nq = (uint32_t)min((unsigned long long)grab, n_chunks - q0);
        for (uint32_t c = 0; c < nq && ok; ++c) {
          const ChunkMeta cm = S.chunk[c];
          if (cm.n == 0) continue;
          const uint32_t q = (uint32_t)(q0 + c);
          const uint32_t bytes = (cm.n * ES) & ~15u;
          const uint32_t aux0 = OPC == OP_RENORM ? (cm.m | S.zmask[c]) : 0u;
          ok = produce(q, cm.off, cm.n, cm.m, aux0, static_cast<const char*>(p.base) + cm.off * ES, bytes);
          for (uint32_t mm = cm.m; ok && mm; mm &= mm - 1) {
            const uint32_t i = __ffs(mm) - 1;
            ok = produce(q, cm.off, cm.n, cm.m, 0u,
                         static_cast<const char*>(p.experts.p[i]) + (cm.off - p.expert_origin) * ES, bytes);
            S.realized[i] += (unsigned long long)cm.n * ES;
          }
        }
      }
      ok = __shfl_sync(0xFFFFFFFFu, ok, 0);
      __syncwarp();
    }
    if (lane == 0) {
      if (ok) ok = produce(kEnd, 0, 0, 0, 0u, nullptr, 0);
      if (!ok) {
        atomicOr(p.err, kErrTimeout);
        S.abort = 1;
      }
      // drain: the last fill of every slot must have landed before the CTA may exit
      for (uint32_t s = 0; s < (uint32_t)kSlots && s < fill; ++s) {
        const uint32_t last = fill - 1 - ((fill - 1 + kSlots - s) % kSlots);
        if (last == 0 && p.stall) continue;  // never armed: nothing in flight
        mbar_wait_drain(&S.full[s], (last / kSlots) & 1u);
      }
      for (uint32_t i = 0; i < p.K; ++i)
        if (S.realized[i])
          atomicAdd(p.realized + (uint64_t)(blockIdx.x % kCounterSlots) * p.K + i, S.realized[i]);
    }
    merge_end<kConsumers + 32>(p, &S.last);
    return;
  }

  // ---------------- consumers ----------------
  float x0[VPT][V], acc[VPT][V];
  uint64_t off = 0;
  uint32_t n = 0, n_tma = 0, remaining = 0;
  uint32_t m_chunk = 0, m_rest = 0;  // the chunk's access mask; its experts still to come
  float s_sel = 0.0f;  // renormalised AVG: sum of the counted experts' alpha (ascending)
  for (uint32_t fill = 0;; ++fill) {
    const uint32_t s = fill % kSlots, r = fill / kSlots;
    if (!warp_wait<true>(&S.full[s], r & 1u, abort_flag, wl)) {
      atomicOr(p.err, kErrTimeout);
      S.abort = 1;
      break;
    }
    const uint8_t* slot = S.slot[s];
    // fills come as the base chunk, then its selected experts in ascending order: only a
    // base fill needs the slot's metadata; an expert fill's expert is the next set bit
    if (remaining == 0) {
      const SlotMeta mt = S.meta[s];
      if (mt.q == kEnd) break;
      off = mt.off;
      n = mt.n;
      n_tma = ((n * ES) & ~15u) / ES;
      m_chunk = m_rest = mt.m;
      remaining = __popc(mt.m);
      if constexpr (OPC == OP_RENORM) {
        s_sel = 0.0f;
        for (uint32_t mm = mt.aux; mm; mm &= mm - 1) s_sel = __fadd_rn(s_sel, p.alpha[__ffs(mm) - 1]);
      }
#pragma unroll
      for (int u = 0; u < VPT; ++u) {
        const uint32_t k0 = (tid + (uint32_t)u * kConsumers) * V;
        read_vec<BF16>(slot, p.base, off, k0, n, n_tma, x0[u]);
        if (remaining) {
#pragma unroll
          for (int e = 0; e < V; ++e) acc[u][e] = 0.0f;
        }
      }
    } else {
      const uint32_t i = __ffs(m_rest) - 1;
      m_rest &= m_rest - 1;
      const void* src = p.experts.p[i];
      // renormalised AVG: beta_i = alpha_i / (sum of the selected alpha), one IEEE division
      const float a = OPC == OP_RENORM ? __fdiv_rn(p.alpha[i], s_sel) : p.alpha[i];
#pragma unroll
      for (int u = 0; u < VPT; ++u) {
        const uint32_t k0 = (tid + (uint32_t)u * kConsumers) * V;
        const uint4 re = read_raw<BF16>(slot, src, off - p.expert_origin, k0, n, n_tma);
        delta_pairs<BF16>(re, x0[u], [&](int e, float d0, float d1) {
          f2_fma(a, a, d0, d1, acc[u][e], acc[u][e + 1], acc[u][e], acc[u][e + 1]);
        });
      }
      --remaining;
    }
    mbar_arrive(&S.empty[s]);  // every consumer thread: its own reads of the slot are done
    if (remaining == 0) {
#pragma unroll
      for (int u = 0; u < VPT; ++u) {
        const uint32_t k0 = (tid + (uint32_t)u * kConsumers) * V;
        if (k0 >= n) continue;
        // no expert selected: every accumulator would be +0, the output is M_0 plus that
        uint32_t w[4];
#pragma unroll
        for (int e = 0; e < V; e += 2)
          put_pair<BF16>(w, e, __fadd_rn(x0[u][e], m_chunk == 0 ? 0.0f : acc[u][e]),
                         __fadd_rn(x0[u][e + 1], m_chunk == 0 ? 0.0f : acc[u][e + 1]));
        store_words<BF16>(p.out, off + k0, n - k0, w);
      }
    }
  }
  merge_end<kConsumers + 32>(p, &S.last);
}

// ---------------- TIES, DARE and DARE-TIES: groups of fills ----------------
//
// The same TMA ring, but fills are published in groups: a chunk's base fill and its first GF
// selected experts' fills, then GF more at a time, each group in consecutive ring slots with
// one "full" mbarrier that counts the bytes of its fills and one "empty" mbarrier that counts
// the consumers' releases.  A consumer thread waits once per group, folds the group's experts
// into its vector in the fixed ascending order, and releases the group; after a chunk's last
// group it finalises.  The per-fill waits, arrivals and metadata reads of the streaming kernel
// above disappear, and whatever a chunk selects the ring holds two groups or more, so that one
// is brought in while another is folded.
constexpr uint32_t kTcMaxK = 32;

// Ring slots, experts per group and CTAs per SM by expert count: K <= 4 takes a chunk of up to 5
// fills as one group, two of them in 11 slots, at four CTAs per SM (three for DARE-TIES, whose
// state needs more registers); K <= 8 one group of up to 9 fills, two in 18 slots (17 where the
// mask words fill the entries), at three; larger K groups of up to 8 experts in 17 slots at
// three, whose consumers keep a chunk's state from group to group.  A fill is 4 KiB: 256 consumer
// threads take one vector each, but for TIES and DARE with K <= 4 128 threads take two (a group's
// wait, release and metadata reads are then shared by two vectors, and 96 registers a thread hold
// both: TIES 1.006 -> 0.969 ms on four Llama layers at the full budget, DARE 1.304 -> 1.248).
//
// Merge times, ms, of the streaming kernel (K > 8 TIES, K > 16), of whole chunks in the ring, and
// here: Qwen2.5-0.5B TIES K = 16 at f = 0.25 1.313 / 1.235 / 0.945, at f = 1 1.614 / 1.480 / 1.099;
// K = 32 (8 layers) TIES 1.258 / - / 0.835, DARE 1.526 / - / 1.108, DARE-TIES 1.843 / - / 1.596;
// Qwen2.5-1.5B (8 layers) K = 16 DARE - / 1.414 / 1.315; TIES K = 8 - / 0.819 / 0.712; four Llama
// layers TIES K = 4 - / 0.978 / 0.926 at f = 1, - / 0.654 / 0.621 at f = 0.1.  Groups of 5 gave
// 1.141 ms for TIES K = 16 at f = 1 (1.109 with 8 then), 7 1.119, 16 (one chunk) 1.240.  Measured
// and not taken, on DARE with 16 experts: two vectors per thread 1.430 ms, four CTAs per SM with
// groups of 6 in 13 slots 1.344, both 1.328; earlier, 2 KiB fills at six CTAs per SM 1.55 against
// 1.41, 3 KiB fills at four 1.46.
template <int OPC, int KC>
struct TcGeo {
  static constexpr int kSlots = KC <= 4 ? 11 : (KC <= 8 && OPC == OP_TIES ? 18 : 17);
  static constexpr int kGroup = KC <= 4 ? 4 : 8;  // expert fills per group
  static constexpr int kCtasPerSm = KC <= 4 && OPC != OP_DTIES ? 4 : 3;
  static constexpr int kVpt = KC <= 4 && OPC != OP_DTIES ? 2 : 1;  // vectors per consumer thread and fill
  static constexpr int kConsumers = 256 / kVpt;
  static constexpr int kThreads = kConsumers + 32;
  static constexpr uint32_t kSlotBytes = kConsumers * kVpt * 16u;
  static constexpr uint32_t kGrab = 8;
};

enum : uint32_t { kFirst = 1u, kLast = 2u, kFast = 4u, kNone = 8u, kEndGroup = 16u };

template <int GF, bool TIES>
struct TcEntry {
  uint64_t off;    // element offset of the chunk
  uint32_t n;      // elements in the chunk
  uint32_t flags;  // kFirst: the group begins with the base fill; kLast: it ends its chunk; kFast:
                   // every selected threshold is >= 2^-100 (no numerator needs the IEEE division);
                   // kNone: the chunk selects no expert
  uint32_t s0;     // ring slot of the group's first fill; fill j sits in slot s0 + j (mod NS)
  uint32_t nexp;   // expert fills
  uint8_t ex[GF < 8 ? 8 : GF];    // their experts in fill order
  float thr[TIES ? GF : 1];       // TIES: their trim thresholds
  alignas(16) uint4 pe[TIES ? 1 : GF];  // DARE, DARE-TIES: dare_expert of each
};

template <int NS, uint32_t SB, uint32_t G, int KC, int GF, bool TIES>
struct __align__(128) TcSmem {
  uint8_t slot[NS][SB];
  TcEntry<GF, TIES> ce[NS];
  uint32_t thr[TIES ? G : 1][KC];  // producer only, TIES: bits threshold of (chunk of the grab, expert)
  uint64_t full[NS];
  uint64_t empty[NS];
  // -c and RN(1/c) for the counts c = 0..32 (entry 0: -1, 1); apart, so that two elements' entries
  // load into the register pairs that the packed operations take
  float nneg[kTcMaxK + 1], nrcp[kTcMaxK + 1];
  int abort, last;
};

// DARE-TIES: a rescaled delta d whose keep word passes goes to P and c+ or to N and c- by its sign
// (C = 2^23 + c+ + 256 c-).  Predicated adds, which the FMA pipe takes, instead of keep factors as
// floats from two more compares and packed multiply-adds: the ALU pipe was the busy one (67 %).
// Qwen2.5-1.5B (8 layers) K = 16 2.152 -> 1.930 ms, K = 4 2.116 -> 1.905, K = 8 2.126 -> 1.943,
// Qwen2.5-0.5B (8 layers) K = 32 1.598 -> 1.424, fp32 K = 8 1.175 -> 1.125.  TIES, which tests two
// thresholds and no keep word, lost by the same (K = 16 0.939 -> 0.986).
__device__ __forceinline__ void keep_signed(uint32_t kw, uint32_t T16, float d, float& P, float& N, float& C) {
  asm("{\n .reg .pred q, a, b;\n setp.ge.u32 q, %3, %4;\n setp.gt.and.f32 a, %5, 0f00000000, q;\n"
      " setp.lt.and.f32 b, %5, 0f00000000, q;\n @a add.rn.f32 %0, %0, %5;\n @b add.rn.f32 %1, %1, %5;\n"
      " @a add.rn.f32 %2, %2, 0f3F800000;\n @b add.rn.f32 %2, %2, 0f43800000;\n}"
      : "+f"(P), "+f"(N), "+f"(C)
      : "r"(kw), "r"(T16), "f"(d));
}

template <bool BF16, int OPC, int KC>
__global__ void __launch_bounds__(TcGeo<OPC, KC>::kThreads, TcGeo<OPC, KC>::kCtasPerSm)
    merge_chunk_kernel(const MergeLaunch p, uint32_t cpb, uint32_t grab, uint64_t n_chunks, unsigned long long* work) {
  kernel_begin();
  static_assert(OPC == OP_TIES || OPC == OP_DARE || OPC == OP_DTIES, "groups of fills: TIES, DARE, DARE-TIES");
  // the packed counts C = 2^23 + c+ + 2^8 c-, a byte each, which one byte selection extracts (with
  // CB = 4 or 6 a shift, a select and a mask; that and the split table above: four Llama layers
  // TIES K = 4 0.924 -> 0.910 ms, Qwen2.5-1.5B (8 layers) DARE-TIES K = 16 2.181 -> 2.152, K = 4
  // 2.142 -> 2.116, K = 8 2.159 -> 2.126)
  constexpr uint32_t CB = 8u;
  constexpr int GF = TcGeo<OPC, KC>::kGroup;
  constexpr int NS = TcGeo<OPC, KC>::kSlots;
  constexpr int kConsumers = TcGeo<OPC, KC>::kConsumers;
  constexpr uint32_t G = TcGeo<OPC, KC>::kGrab;
  constexpr uint32_t ES = BF16 ? 2u : 4u;
  constexpr uint32_t SB = TcGeo<OPC, KC>::kSlotBytes;
  constexpr uint32_t CH = SB / ES;  // elements per chunk
  constexpr int V = BF16 ? 8 : 4;
  constexpr int VPT = TcGeo<OPC, KC>::kVpt;
  static_assert(CH == (uint32_t)(kConsumers * VPT * V), "whole vectors per consumer thread and chunk");
  static_assert(NS >= 2 * GF + 1, "a group is brought in while another is folded");
  extern __shared__ __align__(128) uint8_t smem_raw[];
  using Sm = TcSmem<NS, SB, G, KC, GF, OPC == OP_TIES>;
  Sm& S = *reinterpret_cast<Sm*>(smem_raw);
  const uint32_t tid = threadIdx.x, warp = tid >> 5, lane = tid & 31u;
  volatile int* abort_flag = &S.abort;
  const uint32_t wl = wait_limit_of(p.wait_limit);

  if (tid == 0) {
    for (int s = 0; s < NS; ++s) {
      mbar_init(&S.full[s], 1);
      mbar_init(&S.empty[s], kConsumers);  // every consumer thread arrives once per group
    }
    S.abort = 0;
    mbar_fence_init();
  }
  if (tid <= kTcMaxK) {
    const float c = tid == 0 ? 1.0f : (float)tid;
    S.nneg[tid] = -c;
    S.nrcp[tid] = __fdiv_rn(1.0f, c);
  }
  __syncthreads();

  if (warp == kConsumers / 32) {
    // ---------------- producer: lane i serves expert i ----------------
    // The whole warp walks the chunks together.  A single lane that wrote each fill's metadata and
    // issued its copy in a loop was what bounded these merges: TIES with 16 experts took 1.27 ms
    // with it and 1.00 without, with 32 experts 1.14 and 0.88, DARE with 16 1.43 and 1.33 (groups
    // of 7 on both sides).  Lane i keeps expert i's
    // trim thresholds, mask words and realized bytes in registers; every lane waits for the ring
    // itself, so that each has acquired the slots its copies refill.
    uint32_t fill = 0;  // ring slots used so far (monotonic)
    uint32_t seq = 0;   // groups published
    uint32_t head = 0;  // oldest published group not yet seen released
    uint32_t used = 0;  // slots held by groups head .. seq - 1
    // Lane e: the fills held by the group of entry e, read by a shuffle.  (In shared memory a lane that
    // lagged behind in reserve() could read the count that lane 0 had written for the next group of the
    // same entry: with all entries outstanding, as in a run of chunks that select no expert, the entry
    // just freed is the one published next.)
    static_assert(NS <= 32, "one lane per entry");
    uint32_t nf = 0;
    bool ok = true;
    // wait until entry seq % NS is free and nfill slots are free; groups are released in order,
    // so the oldest one is the next to free its slots
    auto reserve = [&](uint32_t nfill) -> bool {
      while (seq - head >= (uint32_t)NS || used + nfill > (uint32_t)NS) {
        const uint32_t he = head % NS;
        if (!warp_wait(&S.empty[he], (head / NS) & 1u, abort_flag, wl)) return false;
        used -= __shfl_sync(0xFFFFFFFFu, nf, (int)he);
        ++head;
      }
      return true;
    };
    const bool mine = lane < p.K;  // this lane serves an expert
    const char* src = mine ? static_cast<const char*>(p.experts.p[lane]) : nullptr;
    unsigned long long realized = 0;
    uint4 pe = make_uint4(0u, 0u, 0u, 0u);
    uint32_t pe_hi = 0xFFFFFFFFu;  // the upper word of the group number that pe is for
    unsigned long long q_next = 0;
    if (lane == 0) q_next = atomicAdd(work, (unsigned long long)grab);
    for (;;) {
      const unsigned long long q0 = __shfl_sync(0xFFFFFFFFu, q_next, 0);
      if (q0 >= n_chunks || !ok) break;
      if (lane == 0) q_next = atomicAdd(work, (unsigned long long)grab);  // used by the next grab
      // lane c < grab: metadata of chunk q0 + c
      uint32_t grp = 0;
      ChunkMeta cl{0, 0, 0};
      if (lane < grab) {
        const unsigned long long q = q0 + lane;
        if (q < n_chunks && checked_block(p, p.b_begin + q / cpb)) {
          const uint64_t b = p.b_begin + q / cpb;
          const uint32_t start = (uint32_t)(q % cpb) * CH;
          const uint32_t len = p.blk_len[b];
          cl.off = p.blk_off[b] + start;
          cl.m = p.mask[b];
          cl.n = start < len ? min(CH, len - start) : 0u;
          if (p.touched_only && cl.m == 0u) cl.n = 0u;  // left as it is: a reference to M_0
          if (OPC == OP_TIES) grp = p.blk_group[b];
          if (!checked_chunk<OPC == OP_TIES>(p, b, cl, grp, ES)) cl.n = 0u, grp = 0u;
        }
      }
      // TIES: this lane's expert's trim threshold for every chunk of the grab, at least the smallest
      // subnormal (a zero delta is never kept: it would add nothing); each lane reads its own back
      if constexpr (OPC == OP_TIES) {
#pragma unroll
        for (uint32_t c = 0; c < G; ++c) {
          const uint32_t g = __shfl_sync(0xFFFFFFFFu, grp, c);  // past the grab 0, a group like any
          if (mine) S.thr[c][lane] = max(ties_bits_threshold(p.tau[(uint64_t)lane * p.n_groups + g]), 1u);
        }
      }
      // not unrolled, and without the loops that a class cannot take: the producer's code competes
      // with the consumers' for the instruction cache (0.701 -> 0.623 ms at f = 0.1, with empty
      // chunks apart in the consumers)
#pragma unroll 1
      for (uint32_t c = 0; c < grab; ++c) {
        uint64_t off = __shfl_sync(0xFFFFFFFFu, cl.off, c);
        uint32_t left = __shfl_sync(0xFFFFFFFFu, cl.n, c);  // elements of the chunk still to be published
        const uint32_t m = __shfl_sync(0xFFFFFFFFu, cl.m, c);
        if (left == 0u || !ok) continue;
        const bool sel = (m >> lane) & 1u;
        const uint32_t rank = __popc(m & ((1u << lane) - 1u)), nsel = __popc(m);
        uint32_t fast = 0u, thr = 0u;  // DARE-TIES: rescaled deltas may be tiny
        if constexpr (OPC == OP_TIES) {
          if (sel) thr = S.thr[c][lane];
          fast = __any_sync(0xFFFFFFFFu, sel && thr < 0x0D800000u) ? 0u : kFast;  // bits of 2^-100
        }
        do {
          uint32_t n = left;
          if constexpr (OPC != OP_TIES) {
            // an entry's share of the mask generator holds one upper word of the group number: a
            // chunk that crosses a multiple of 2^35 elements goes as two
            const uint32_t g_hi = (uint32_t)(off >> 35);
            n = (uint32_t)min((uint64_t)left, ((uint64_t)g_hi + 1u << 35) - off);
            if (g_hi != pe_hi && mine) pe = dare_expert(p, g_hi, lane);
            pe_hi = g_hi;
          }
          left -= n;
          const uint32_t bytes = (n * ES) & ~15u;
          uint32_t done = 0u, first = 1u;
          do {
            const uint32_t nexp = min(nsel - done, (uint32_t)GF), nfill = nexp + first;
            if (!(ok = reserve(nfill))) break;
            if (fill >= (uint32_t)NS) fence_proxy_async_smem();  // slots the consumers have read are refilled
            const uint32_t e = seq % NS;
            const bool here = sel && rank >= done && rank < done + nexp;  // this lane's fill is in the group
            auto& ce = S.ce[e];
            if (here) {
              ce.ex[rank - done] = (uint8_t)lane;
              if constexpr (OPC == OP_TIES) ce.thr[rank - done] = __uint_as_float(thr);
              else ce.pe[rank - done] = pe;
            }
            if (lane == 0) {
              ce.off = off;
              ce.n = n;
              ce.flags = (first ? kFirst : 0u) | (done + nexp == nsel ? kLast : 0u) | (nsel ? 0u : kNone) | fast;
              ce.s0 = fill % NS;
              ce.nexp = nexp;
            }
            if (lane == e) nf = nfill;
            __syncwarp();  // the entry is written before it is published
            // test hook: the first group is never armed, so the consumers' wait for it runs out
            const bool arm = !(seq == 0 && p.stall);
            if (lane == 0 && arm) {
              mbar_arrive_expect_tx(&S.full[e], nfill * bytes);
              if (first && bytes)
                tma_load_1d(S.slot[fill % NS], static_cast<const char*>(p.base) + off * ES, bytes, &S.full[e]);
            }
            __syncwarp();  // armed before any lane's copy can complete
            if (here) {
              if (bytes && arm)
                tma_load_1d(S.slot[(fill + first + rank - done) % NS], src + (off - p.expert_origin) * ES, bytes, &S.full[e]);
              realized += (unsigned long long)n * ES;
            }
            fill += nfill;
            used += nfill;
            ++seq;
            done += nexp;
            first = 0u;
          } while (GF < KC && done < nsel);
          off += n;
        } while (OPC != OP_TIES && left && ok);
      }
    }
    if (ok && (ok = reserve(0u))) {
      const uint32_t e = seq % NS;
      if (lane == 0) {
        S.ce[e].flags = kEndGroup;
        if (!(seq == 0 && p.stall)) mbar_arrive_expect_tx(&S.full[e], 0u);
      }
      ++seq;
    }
    if (!ok && lane == 0) {
      atomicOr(p.err, kErrTimeout);
      S.abort = 1;
    }
    // drain: the last group of every entry must have landed before the CTA may exit
    for (uint32_t e = 0; e < (uint32_t)NS && e < seq; ++e) {
      const uint32_t last = seq - 1 - ((seq - 1 + NS - e) % NS);
      if (last == 0 && p.stall) continue;  // never armed: nothing in flight
      mbar_wait_drain(&S.full[e], (last / NS) & 1u);
    }
    if (realized) atomicAdd(p.realized + (uint64_t)(blockIdx.x % kCounterSlots) * p.K + lane, realized);
    merge_end<kConsumers + 32>(p, &S.last);
    return;
  }
  // ---------------- consumers: thread t owns vectors t, t + kConsumers, ... of every chunk ----------------
  float x0[VPT][V];
  // DARE: acc = fma(alpha_i, v_i, acc) over the selected experts whose keep word passes, in
  // ascending order, with v_i = delta_i * sigma (a dropped entry is omitted).
  // TIES: P and N, the sums of the kept positive and negative deltas, and both counts in one
  // float C = 2^23 + c+ + 2^CB c- (exact: every value is an integer below 2^24, so the low bits
  // of C hold c+ and c-).  DARE-TIES keeps, instead, every nonzero rescaled delta s = d sigma
  // whose keep word passes (no magnitude trim; keep_signed).  A TIES delta d is kept positive when d >= thr and kept
  // negative when d <= -thr (thr > 0: |d| >= thr and the sign in one compare each); the keep
  // factors k+ and k- are 1 or 0, and P = fma(k+, d, P), N = fma(k-, d, N): a factor 1 adds d with
  // the one rounding of P + d, a factor 0 adds a zero, which leaves P and N unchanged (they start
  // at +0 and are never -0).  Two elements per packed instruction.
  float Pp[VPT][V], Nn[VPT][V], Cc[VPT][V];
  float (&acc)[VPT][V] = Pp;
  // a class whose largest chunk is one group keeps its state for one group only
  constexpr bool kWhole = GF >= KC;
  for (uint32_t c = 0;; ++c) {
    const uint32_t e = c % NS;
    if (!warp_wait(&S.full[e], (c / NS) & 1u, abort_flag, wl)) {
      atomicOr(p.err, kErrTimeout);
      S.abort = 1;
      break;
    }
    const auto& ce = S.ce[e];
    const uint32_t begin = ce.flags;
    if (begin & kEndGroup) break;
    uint32_t s = ce.s0;
    const uint32_t nexp = ce.nexp;
    // whether the thread's vectors lie inside the bulk-copied bytes
    const bool in_slot = (tid + (uint32_t)(VPT - 1) * kConsumers + 1u) * V <= ((ce.n * ES) & ~15u) / ES;
    if (begin & kNone) {  // uniform over the CTA
      // no expert selected: the output is M_0 plus the zero the operator adds (lambda * +0
      // for TIES, +0 for DARE)
      const uint32_t n = ce.n;
      const uint64_t off = ce.off;
      float xb[VPT][V];
#pragma unroll
      for (int u = 0; u < VPT; ++u)
        read_vec<BF16>(S.slot[s], p.base, off, (tid + (uint32_t)u * kConsumers) * V, n, ((n * ES) & ~15u) / ES, xb[u]);
      mbar_arrive(&S.empty[e]);
      const float z = kTiesLike<OPC> ? __fmul_rn(p.lambda, 0.0f) : 0.0f;
#pragma unroll
      for (int u = 0; u < VPT; ++u) {
        uint32_t w[4];
#pragma unroll
        for (int v = 0; v < V; v += 2) {
          float y0, y1;
          f2_add(xb[u][v], xb[u][v + 1], z, z, y0, y1);
          put_pair<BF16>(w, v, y0, y1);
        }
        const uint32_t k0 = (tid + (uint32_t)u * kConsumers) * V;
        if (k0 < n) store_words<BF16>(p.out, off + k0, n - k0, w);
      }
      continue;
    }
    if (kWhole || (begin & kFirst)) {
#pragma unroll
      for (int u = 0; u < VPT; ++u) {
        const uint32_t k0 = (tid + (uint32_t)u * kConsumers) * V, n = ce.n;
        read_vec<BF16>(S.slot[s], p.base, ce.off, k0, n, ((n * ES) & ~15u) / ES, x0[u]);
#pragma unroll
        for (int v = 0; v < V; ++v) {
          Pp[u][v] = 0.0f;
          if (OPC != OP_DARE) {
            Nn[u][v] = 0.0f;
            Cc[u][v] = 8388608.0f;  // 2^23
          }
        }
      }
      s = s + 1 == (uint32_t)NS ? 0u : s + 1;
    }
    DareVec dv[VPT];
    if constexpr (OPC != OP_TIES) {
#pragma unroll
      for (int u = 0; u < VPT; ++u) dv[u] = dare_vec(ce.off + (tid + (uint32_t)u * kConsumers) * V, p);
    }
#pragma unroll 1
    for (uint32_t j = 0; j < nexp; ++j) {
      const float thr = OPC == OP_TIES ? ce.thr[j] : 0.0f;
#pragma unroll
      for (int u = 0; u < VPT; ++u) {
        const uint32_t k0 = (tid + (uint32_t)u * kConsumers) * V;
        uint4 r;
        if (in_slot) {
          r = *reinterpret_cast<const uint4*>(S.slot[s] + k0 * ES);
        } else {  // the ragged tail of a tensor, from global memory
          const uint32_t n = ce.n;
          r = read_raw<BF16>(S.slot[s], p.experts.p[ce.ex[j]], ce.off - p.expert_origin, k0, n, ((n * ES) & ~15u) / ES);
        }
        uint32_t kw[V];
        float a = 0.0f;
        if constexpr (OPC != OP_TIES) {
          const uint4 pe = ce.pe[j];
          a = __uint_as_float(pe.w);
          dare_keep_words<BF16>(p, dv[u], pe, kw);
        }
        // one element pair at a time, so that only the raw vector stays live
        auto fold_pair = [&](int v, float d0, float d1) {
          if constexpr (OPC != OP_TIES) f2_mul(d0, d1, p.sigma, p.sigma, d0, d1);
          if constexpr (OPC == OP_DARE) {
            // a dropped entry is omitted from the sum, as an unselected one is
            if (kw[v] >= p.dare_T16) acc[u][v] = __fmaf_rn(a, d0, acc[u][v]);
            if (kw[v + 1] >= p.dare_T16) acc[u][v + 1] = __fmaf_rn(a, d1, acc[u][v + 1]);
            return;
          }
          if constexpr (OPC == OP_DTIES) {
            keep_signed(kw[v], p.dare_T16, d0, Pp[u][v], Nn[u][v], Cc[u][v]);
            keep_signed(kw[v + 1], p.dare_T16, d1, Pp[u][v + 1], Nn[u][v + 1], Cc[u][v + 1]);
            return;
          }
          float t0, t1;
          const float kp0 = d0 >= thr ? 1.0f : 0.0f, kp1 = d1 >= thr ? 1.0f : 0.0f;
          const float kn0 = d0 <= -thr ? 1.0f : 0.0f, kn1 = d1 <= -thr ? 1.0f : 0.0f;
          f2_fma(kp0, kp1, d0, d1, Pp[u][v], Pp[u][v + 1], Pp[u][v], Pp[u][v + 1]);
          f2_fma(kn0, kn1, d0, d1, Nn[u][v], Nn[u][v + 1], Nn[u][v], Nn[u][v + 1]);
          f2_fma(kn0, kn1, (float)(1u << CB), (float)(1u << CB), Cc[u][v], Cc[u][v + 1], t0, t1);
          f2_add(kp0, kp1, t0, t1, Cc[u][v], Cc[u][v + 1]);
        };
        delta_pairs<BF16>(r, x0[u], fold_pair);
      }
      s = s + 1 == (uint32_t)NS ? 0u : s + 1;
    }
    const uint32_t n = ce.n, flags = begin;
    const uint64_t off = ce.off;
    mbar_arrive(&S.empty[e]);  // every read of the group's slots and entry is done
    if (!kWhole && !(flags & kLast)) continue;
    // the chunk's output from f(u, v, y0, y1), elements v and v + 1 of vector u
    uint32_t w[VPT][4];
    auto fill_words = [&](auto f) {
#pragma unroll
      for (int u = 0; u < VPT; ++u)
#pragma unroll
        for (int v = 0; v < V; v += 2) {
          float y0, y1;
          f(u, v, y0, y1);
          put_pair<BF16>(w[u], v, y0, y1);
        }
    };
    auto store = [&]() {
#pragma unroll
      for (int u = 0; u < VPT; ++u) {
        const uint32_t k0 = (tid + (uint32_t)u * kConsumers) * V;
        if (k0 < n) store_words<BF16>(p.out, off + k0, n - k0, w[u]);
      }
    };
    if constexpr (OPC == OP_DARE) {
      fill_words([&](int u, int v, float& y0, float& y1) {
        f2_add(x0[u][v], x0[u][v + 1], acc[u][v], acc[u][v + 1], y0, y1);
      });
      store();
      continue;
    }
    // the elected side's sum and count: the sign of P + N taken exactly as P > -N or P < -N
    // (then that side holds at least one entry, so c >= 1); otherwise the numerator +0, whose
    // quotient is +0 whatever count (<= 32, a valid table entry) is paired with it
    auto num_c = [&](int u, int v, float& num, uint32_t& cv) {
      const bool pos = Pp[u][v] > -Nn[u][v], any = Pp[u][v] != -Nn[u][v];
      num = any ? (pos ? Pp[u][v] : Nn[u][v]) : 0.0f;
      const uint32_t cb = __float_as_uint(Cc[u][v]);
      static_assert(CB == 8u && kTcMaxK < 256u, "a byte holds a count");
      cv = __byte_perm(cb, 0u, pos ? 0x4440u : 0x4441u);  // byte 0 or 1
    };
    // q = RN(num * y), then Markstein's correction q + RN(num - q c) * y, and the output
    // fma(lambda, q, M_0), two elements per instruction.  Numerators 0 < |num| < 2^-100 need the
    // IEEE division: where one may occur (`checked`: DARE-TIES, whose rescaled deltas may be tiny,
    // and TIES chunks with a threshold below 2^-100) the warp looks for them, and then takes its
    // elements one by one.
    auto one = [&](int u, int v) {
      float a;
      uint32_t cv;
      num_c(u, v, a, cv);
      return __fmaf_rn(p.lambda, div_small(a, -S.nneg[cv], S.nrcp[cv]), x0[u][v]);
    };
    auto finalise = [&](auto checked) {
      // 2 |bits| - 2 wraps the zeros to the top: its minimum over the vector is below
      // 2 * bits(2^-100) - 2 exactly when some numerator has 0 < |num| < 2^-100
      static_assert(0x0D800000u * 2u - 2u == 0x1AFFFFFEu, "bits of 2^-100");
      uint32_t lowest = 0xFFFFFFFFu;
      auto look = [&](float a0, float a1) {
        lowest = min(lowest, min(__float_as_uint(a0) * 2u - 2u, __float_as_uint(a1) * 2u - 2u));
      };
      auto by_element = [&]() -> bool {
        if (!__any_sync(0xFFFFFFFFu, lowest < 0x1AFFFFFEu)) return false;
        fill_words([&](int u, int v, float& y0, float& y1) {
          y0 = one(u, v);
          y1 = one(u, v + 1);
        });
        return true;
      };
      auto fast = [&](int u, int v, float& y0, float& y1) {
        float a0, a1, q0, q1, r0, r1;
        uint32_t c0, c1;
        num_c(u, v, a0, c0);
        num_c(u, v + 1, a1, c1);
        if constexpr (decltype(checked)::value && kWhole) look(a0, a1);
        const float n0 = S.nneg[c0], n1 = S.nneg[c1], i0 = S.nrcp[c0], i1 = S.nrcp[c1];
        f2_mul(a0, a1, i0, i1, q0, q1);
        f2_fma(q0, q1, n0, n1, a0, a1, r0, r1);
        f2_fma(r0, r1, i0, i1, q0, q1, q0, q1);
        f2_fma(p.lambda, p.lambda, q0, q1, x0[u][v], x0[u][v + 1], y0, y1);
      };
      // a class that keeps its state over groups has no registers for the words beside it: it
      // looks first, at both sums (one of them is the numerator)
      if constexpr (decltype(checked)::value && !kWhole) {
#pragma unroll
        for (int u = 0; u < VPT; ++u)
#pragma unroll
          for (int v = 0; v < V; ++v) look(Pp[u][v], Nn[u][v]);
        if (by_element()) return;
      }
      fill_words(fast);
      if constexpr (decltype(checked)::value && kWhole) by_element();
    };
    if (OPC == OP_TIES && (flags & kFast)) finalise(std::false_type{});  // uniform over the CTA
    else finalise(std::true_type{});
    store();
  }
  merge_end<kConsumers + 32>(p, &S.last);
}

// Chunks taken per counter increment: at most G, fewer where the CTAs would get less than eight
// grabs each.  Eight at once left most CTAs of a small merge without work and the others with one
// grab more or less: 1.5M elements, blocks of 4096, 4 experts, AVG 16.8 -> 9.0 us, TIES 23.9 ->
// 11.9, DARE 21.8 -> 11.0; 20M in blocks of 16384, TIES 48.7 -> 36.4.  With two grabs per CTA the
// latter takes 48.1, with 16 40.9 us (each grab waits for its blocks' entries in the tables).
template <uint32_t G>
uint32_t grab_of(uint64_t n_chunks, uint64_t grid) {
  const uint64_t g = n_chunks / (grid * 8u);
  return (uint32_t)(g < 1 ? 1 : (g > G ? G : g));
}

template <bool BF16, int OPC, int KC>
cudaError_t launch_chunk(const MergeLaunch& p, cudaStream_t st) {
  using Geo = TcGeo<OPC, KC>;
  constexpr uint32_t chunk = Geo::kSlotBytes / (BF16 ? 2u : 4u);
  const uint32_t cpb = (p.block_elems + chunk - 1) / chunk;
  const uint64_t n_chunks = (p.b_end - p.b_begin) * cpb;
  if (n_chunks == 0) return cudaSuccess;
  if (n_chunks >= 0xFFFFFFFFull) return cudaErrorInvalidValue;
  int dev = 0, sms = 0;
  cudaError_t e;
  if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
  if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
  using Smem = TcSmem<Geo::kSlots, Geo::kSlotBytes, Geo::kGrab, KC, Geo::kGroup, OPC == OP_TIES>;
  // every CTA also holds 1 KB of the SM's 228 KB for the system
  static_assert(Geo::kCtasPerSm * (sizeof(Smem) + 1024) <= 228u * 1024u,
                "the CTAs per SM that the grid assumes fit one SM's shared memory");
  const size_t smem = sizeof(Smem);
  auto kern = merge_chunk_kernel<BF16, OPC, KC>;
  if ((e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)) != cudaSuccess)
    return e;
  uint64_t grid = (uint64_t)sms * Geo::kCtasPerSm;
  if (grid > n_chunks) grid = n_chunks;
  return launch_kernel(p.follows, kern, (unsigned)grid, Geo::kThreads, smem, st, p, cpb,
                       grab_of<Geo::kGrab>(n_chunks, grid), n_chunks, p.work);
}

template <bool BF16, int OPC>
cudaError_t launch_groups(const MergeLaunch& p, cudaStream_t st) {
  if (p.K <= 4) return launch_chunk<BF16, OPC, 4>(p, st);
  if (p.K <= 8) return launch_chunk<BF16, OPC, 8>(p, st);
  return launch_chunk<BF16, OPC, kMaxK>(p, st);
}

template <bool BF16, int OPC>
cudaError_t launch_op(const MergeLaunch& p, cudaStream_t st) {
  const uint32_t chunk = Geo::kSlotBytes / (BF16 ? 2u : 4u);
  const uint32_t cpb = (p.block_elems + chunk - 1) / chunk;
  const uint64_t n_chunks = (p.b_end - p.b_begin) * cpb;
  if (n_chunks == 0) return cudaSuccess;
  if (n_chunks >= 0xFFFFFFFFull) return cudaErrorInvalidValue;
  int dev = 0, sms = 0;
  cudaError_t e;
  if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
  if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
  const size_t smem = sizeof(Smem<Geo::kSlots, Geo::kSlotBytes, Geo::kGrab>);
  if ((e = cudaFuncSetAttribute(merge_tma_kernel<BF16, OPC>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)) !=
      cudaSuccess)
    return e;
  uint64_t grid = (uint64_t)sms * Geo::kCtasPerSm;
  if (grid > n_chunks) grid = n_chunks;
  return launch_kernel(p.follows, merge_tma_kernel<BF16, OPC>, (unsigned)grid, Geo::kThreads, smem, st, p, cpb,
                       grab_of<Geo::kGrab>(n_chunks, grid), n_chunks, p.work);
}

template <bool BF16>
cudaError_t launch_dtype(const MergeLaunch& p, cudaStream_t st) {
  switch (p.op_kind) {
    case MP_OP_AVG:
    case MP_OP_TA: return launch_op<BF16, OP_ADD>(p, st);
    case MP_OP_TIES: return launch_groups<BF16, OP_TIES>(p, st);
    case MP_OP_DARE: return launch_groups<BF16, OP_DARE>(p, st);
    case MP_OP_AVG_RENORM: return launch_op<BF16, OP_RENORM>(p, st);
    case MP_OP_DARE_TIES: return launch_groups<BF16, OP_DTIES>(p, st);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace

cudaError_t launch_merge(const MergeLaunch& p, cudaStream_t st) {
  return p.dtype == MP_BF16 ? launch_dtype<true>(p, st) : launch_dtype<false>(p, st);
}

}  // namespace mp
