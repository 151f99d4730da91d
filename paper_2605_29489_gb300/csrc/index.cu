// Catalog pass (Sec. 3 "Catalog"; the Analyze reads of Sec. 2): per-(expert, block)
// statistics of Delta = M_i - M_0 and, for TIES, the per-(expert, trim group) threshold.
//
// Mapping: an item is a block and up to 8 of its experts (4 for TIES).  Consumer thread l is
// lane l of the fixed summation order: it streams 16-byte vectors l, l+256, ... of the
// block (base once, each expert of the group), keeps a sequential fma chain of delta^2
// per expert, then the lanes are combined by a xor butterfly inside each warp and over
// the 8 warp sums.  That order is part of the definition of the norm (it decides the
// plan), so it must not change with tuning.
//
// TIES threshold (k-th largest 15-bit key bits(bf16(|delta|)) & 0x7FFF per trim group): a sample
// predicts a window of keys, the index pass counts those in shared memory and the threshold
// comes from the counts.  Where it lies outside the window a two-level radix select finds it:
// the upper 8 key bits' bins, the bin holding the k-th key, a second pass over only the blocks
// that can hold keys in that bin with bins of the lower 7 bits, the key.
#include <cuda_bf16.h>

#include <type_traits>

#include "mp_internal.cuh"
#include "tma.cuh"

namespace mp {
namespace {

constexpr uint32_t kNoBin = 0xFFFFFFFFu;

__device__ __forceinline__ uint4 load_vec_raw(const void* base_ptr, bool bf16, uint64_t elem0, uint32_t v,
                                              uint32_t len) {
  // vector v of a block starting at element elem0 with len elements; zero fill past len
  const uint32_t V = bf16 ? 8u : 4u;
  uint32_t k0 = v * V;
  if (k0 + V <= len) {
    const uint4* q = reinterpret_cast<const uint4*>(static_cast<const char*>(base_ptr) +
                                                    (elem0 + k0) * (bf16 ? 2u : 4u));
    return __ldcs(q);
  }
  uint32_t w[4] = {0u, 0u, 0u, 0u};
  if (k0 < len) {
    if (bf16) {
      const uint16_t* s = static_cast<const uint16_t*>(base_ptr) + elem0 + k0;
      for (uint32_t e = 0; e < V && k0 + e < len; ++e) w[e >> 1] |= (uint32_t)s[e] << (16u * (e & 1u));
    } else {
      const uint32_t* s = static_cast<const uint32_t*>(base_ptr) + elem0 + k0;
      for (uint32_t e = 0; e < V && k0 + e < len; ++e) w[e] = s[e];
    }
  }
  return make_uint4(w[0], w[1], w[2], w[3]);
}

template <bool BF16>
__device__ __forceinline__ void unpack(const uint4 r, float (&x)[BF16 ? 8 : 4]) {
  if constexpr (BF16) {
    // the lower element moved up by a multiply (FMA pipe), the upper one by a mask (ALU)
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

__device__ __forceinline__ uint32_t ties_key(float d) {
  return (uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(fabsf(d))) & 0x7FFFu;
}

// ---- the catalog pass: TMA producer / consumer pipeline ---------------------------------
//
// Work item = (block, group of up to KG experts); items are handed out through a global
// counter.  The producer thread streams every chunk of the item's block — the base chunk,
// then each expert's chunk — into a ring of shared-memory slots (cp.async.bulk, completion
// on the slot's "full" mbarrier).  Consumer thread l (0..255) is lane l of the fixed
// summation order: a chunk of VPT * 256 vectors starts at vector VPT * 256 * c, and thread
// l takes its vectors VPT * 256 * c + 256 u + l (u < VPT), i.e. exactly its own vectors l,
// l + 256, ... in increasing order.  At the end of the block the 256 lane sums are
// combined by the xor butterfly.
constexpr int kIxConsumers = 256;
constexpr int kIxThreads = kIxConsumers + 32;
static_assert(kIxConsumers == 256, "one consumer thread per coarse TIES bin at the end of a block");
constexpr uint32_t kIxEnd = 0xFFFFFFFFu;

// ring geometry.  The plain catalog is bound by HBM: three CTAs per SM with 72 KiB rings (two
// with 96 KiB held fewer warps: 1.52 -> 1.42 ms on Qwen2.5-0.5B with 8 experts, 0.80 -> 0.73 with
// 4, with the mixed-precision subtract on both sides of the second).  With 8 experts per item a
// chunk is nine fills, each of which a consumer waited for and released: 4 KiB slots published a
// chunk at a time took that to 1.30 ms (16 experts on 8 layers of Qwen2.5-1.5B: 3.59 -> 3.00 ms
// in all).  With up to 4 experts 8 KiB slots stay, released fill by fill:
// a chunk published at once leaves too little of the ring for the next (0.77 ms with 4 KiB slots,
// 0.85 with 8 KiB ones).  The TIES catalog also bins every delta, which makes it bound by
// instruction latency: four CTAs per SM (more warps to hide it; the state fits 56 registers) with
// twelve 4 KiB slots (one vector per consumer thread and fill), and at most 4 experts per item.
template <bool TIES, int KG = 1, bool UNITS = false>
struct IxGeo {
  static_assert(!TIES || KG <= 4, "the TIES catalog takes at most 4 experts per item");
  static constexpr int kCtasPerSm = TIES ? 4 : 3;
  static constexpr uint32_t kSlotBytes = TIES || KG > 4 ? 4096u : 8192u;
  static constexpr int kSlots = TIES ? (UNITS ? 11 : 12) : (KG > 4 ? 18 : 9);  // UNITS: kBinUnits' larger histograms
  // whole chunks: the base fill and the item's expert fills of one chunk sit in consecutive
  // ring slots under one "full" and one "empty" mbarrier
  static constexpr bool kWhole = TIES || KG > 4;
};

struct IxMeta {
  uint64_t off;    // element offset of the chunk
  uint32_t item;   // work item, or kIxEnd
  uint32_t n;      // elements in the chunk
  uint32_t last;   // 1 on the block's last chunk
  uint32_t s0;     // whole-chunk publication: ring slot of the base fill (experts follow)
  // whole-chunk publication, window bins: the windows of the item's experts (win_words)
  uint32_t wneg[4], wtop[4];
};

// How the TIES catalog bins the keys of the deltas:
//  * kBinCoarse: 256 bins of the upper 8 key bits (the two-level select: a second pass then
//    counts the lower 7 bits inside the chosen bin);
//  * kBinWindow: the W keys [L, L + W) of a window predicted from a sample, one bin each, and
//    one bin below and one above it, so that the threshold is found without a second pass
//    whenever it lies inside the window;
//  * kBinUnits (TIES after masking): both at once, and kept for each (expert, block), because a
//    plan's threshold is that of the blocks it selects: the keys of a window one bin each, the
//    others by their upper 8 bits.
enum { kBinNone = 0, kBinCoarse = 1, kBinWindow = 2, kBinUnits = 3 };
constexpr uint32_t kWinKeys = 384;           // most keys of a window (three binades)
constexpr uint32_t kWinBins = kWinKeys + 2;  // + below + above

// The window of one (expert, trim group), as ties_window_select leaves it: L | W << 16.
// Groups of kWinNarrowBlocks blocks or more get a window of kWinNarrow keys (80 keys, a factor of
// 1.45 or more, either side of the predicted bin of 32), smaller ones, whose sample is small, three
// whole binades.  The increments are what bounds the pass: with three binades for every group
// they took 5.5 wavefronts each and the LSU data pipe was 88 % busy (every block active); in a
// narrow window most lanes share the bins below and above it (1.5 wavefronts).  A pair that misses
// its window costs a pass over its group's blocks.  TIES index in ms by the keys of a narrow window
// (four Llama layers with 4 experts, three seeds / two layers, every block active / Qwen2.5-0.5B with 8
// experts, two seeds / with 16 / Qwen2.5-1.5B, 8 layers, with 16 / Llama-3-8B with 4):
//    96: 1.61 1.56 1.42 / 0.91 / 1.59 1.83 / 3.30 / 3.98 / 12.95   (misses)
//   128: 1.42 1.56 1.42 / 0.91 / 1.59 1.78 / 3.25 / 3.97 / 12.44   (a miss)
//   160: 1.43 1.44 1.44 / 0.93 / 1.62 1.81 / 3.30 / 3.91 / 12.58
//   192: 1.43 1.43 1.43 / 0.93 / 1.61 1.80 / 3.27 / 3.86 / 12.47
//   256: 1.45 1.45 1.45 / 1.01 / 1.66 1.84 / 3.35 / 3.89 / 12.73
//   384: 1.59 1.59 1.59 / 1.14 / 1.78 1.95 / 3.61 / 3.91 / 13.94
constexpr uint32_t kWinNarrow = 192, kWinNarrowBlocks = 16;
static_assert(kWinNarrow >= 1 && kWinNarrow <= kWinKeys, "the counts of a window fit its bins, and key - L + 1 16 bits");

// the window in 16-bit lanes: 1 - L (added to the keys) and W + 1 (the clamp, the bin above)
__device__ __forceinline__ void win_words(uint32_t win, uint32_t& neg, uint32_t& top) {
  neg = ((1u - (win & 0xFFFFu)) & 0xFFFFu) * 0x00010001u;
  top = ((win >> 16) + 1u) * 0x00010001u;
}

// The bins of kBinUnits: key k adds to bin clamp(k - L, 0, W) + (k >> 7), which is one bin per key
// inside [L, L + W) (W = 384, L a multiple of 128) and one per binade outside, in the order of the
// keys.  Bin 0 of what is stored is the count of nonzero deltas: the zeros of a trim group are
// what its other bins leave, also for the elements that a plan omits.  Three instructions more per
// pair of keys than the window alone; without it the catalog read the experts twice (coarse, then
// fine bins) and each plan's threshold read the selected ones a third time: two Llama layers with
// 4 experts, catalog 1.71 -> 0.81 ms, merge with its thresholds 1.54 -> 0.59 ms (floors 0.65, 0.52).
constexpr uint32_t kUnitBins = kUnitHistBins;
static_assert(kUnitBins == 256 + kWinKeys, "bins of kBinUnits");

template <int BM>
constexpr uint32_t key_bins() {
  return BM == kBinNone ? 1u : (BM == kBinWindow ? kWinBins : (BM == kBinUnits ? kUnitBins : 256u));
}

template <int KG, int NS, uint32_t SB, uint32_t NB>
struct __align__(128) IxSmem {
  uint32_t hist[KG][NB];  // first: its byte addresses stay below 2^16 (ties_win2 packs two)
  alignas(128) uint8_t slot[NS][SB];
  IxMeta meta[NS];
  uint64_t full[NS];
  uint64_t empty[NS];
  uint32_t nf[NS];  // whole-chunk publication: fills held by the chunk of each entry
  float red_ss[KG][8];
  float red_mx[KG][8];
  uint32_t red_nz[KG][8];
  uint64_t cbar;  // consumer-only barrier (one arrival per consumer warp)
  int abort, last;
};

// raw 16-byte vector at element k0 of a fill: from the slot when inside the bulk-copied
// bytes, else (the ragged tail of a tensor) from global memory, zero past the chunk
template <bool BF16>
__device__ __forceinline__ uint4 ix_read_raw(const uint8_t* slot, const void* gsrc, uint64_t off, uint32_t k0,
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

__device__ __forceinline__ bool same_vec(const uint4 a, const uint4 b) {
  return a.x == b.x && a.y == b.y && a.z == b.z && a.w == b.w;
}

// TIES coarse bins of two deltas: bin = upper 8 bits of the 15-bit key bits(bf16(|d|)),
// i.e. bits 7..14 of the round-to-nearest-even bf16 of d (the sign bit 15 is masked off);
// both are converted by one packed cvt.  A nonzero delta adds 1 to its bin of the
// shared histogram at hist (byte address in the shared window); a zero delta adds
// nothing, so the histogram's total is the block's nonzero count.  Predicated, so that no
// branch is taken per element.
__device__ __forceinline__ void ties_bin2(float d0, float d1, uint32_t hist) {
  asm volatile(
      "{\n"
      " .reg .pred p0, p1;\n"
      " .reg .b32 w, a0, a1;\n"
      " cvt.rn.bf16x2.f32 w, %2, %1;\n"
      " setp.ne.f32 p0, %1, 0f00000000;\n"
      " setp.ne.f32 p1, %2, 0f00000000;\n"
      " shr.b32 a0, w, 5;\n"
      " and.b32 a0, a0, 1020;\n"
      " add.u32 a0, a0, %0;\n"
      " shr.b32 a1, w, 21;\n"
      " and.b32 a1, a1, 1020;\n"
      " add.u32 a1, a1, %0;\n"
      " @p0 red.shared.add.u32 [a0], 1;\n"
      " @p1 red.shared.add.u32 [a1], 1;\n"
      "}\n" ::"r"(hist),
      "f"(d0), "f"(d1)
      : "memory");
}

// (d0, d1) = (a0 - b0, a1 - b1), each rounded to nearest: one packed subtract
__device__ __forceinline__ void f2_sub(float a0, float a1, float b0, float b1, float& d0, float& d1) {
  asm("{\n .reg .b64 ra, rb, rd;\n mov.b64 ra, {%2, %3};\n mov.b64 rb, {%4, %5};\n sub.rn.f32x2 rd, ra, rb;\n"
      " mov.b64 {%0, %1}, rd;\n}"
      : "=f"(d0), "=f"(d1)
      : "f"(a0), "f"(a1), "f"(b0), "f"(b1));
}

// the deltas of a raw vector against the base elements x0, each one IEEE fp32 subtraction; bf16
// elements are converted by the mixed-precision subtract itself (8 instructions per vector where
// unpacking and a packed subtract take 12: 1.519 -> 1.442 ms on Qwen2.5-0.5B with 8 experts)
template <bool BF16>
__device__ __forceinline__ void deltas(const uint4 r, const float* x0, float* d) {
  if constexpr (BF16) {
    const uint32_t w[4] = {r.x, r.y, r.z, r.w};
#pragma unroll
    for (int k = 0; k < 4; ++k)
      asm("{\n .reg .b16 l, h;\n mov.b32 {l, h}, %2;\n sub.rn.f32.bf16 %0, l, %3;\n sub.rn.f32.bf16 %1, h, %4;\n}"
          : "=f"(d[2 * k]), "=f"(d[2 * k + 1])
          : "r"(w[k]), "f"(x0[2 * k]), "f"(x0[2 * k + 1]));
  } else {
    f2_sub(__uint_as_float(r.x), __uint_as_float(r.y), x0[0], x0[1], d[0], d[1]);
    f2_sub(__uint_as_float(r.z), __uint_as_float(r.w), x0[2], x0[3], d[2], d[3]);
  }
}

// TIES window bins of two deltas: key k adds 1 to bin clamp(k - L + 1, 0, W + 1) of the shared
// histogram at h, also to bin 0 (below the window), which nothing reads: lanes that increment
// one address share a wavefront, and a predicate on the increment cost more than it saved (it
// becomes a branch: 537 instead of 425 million warp instructions on a Llama layer).  Both keys
// at once in 16-bit lanes:
// one add and one clamp at zero and W + 1 (L is at most 32768 - W, so k - L + 1 lies in
// [W - 32767, 32768], from -32607 up in a narrow window; it wraps only for the NaN key 0x7FFF at
// L = 0, whose bin the clamp still keeps in range and whose NaN the statistics report), and one
// multiply-add for both byte addresses (h2 = h in both lanes, which the caller keeps below
// 2^16 - 4 * 385).  An exact zero has key 0: below the window, or, with L = 0, in key 0's bin, where it
// can only decide a threshold of key 0, the one that an uncounted zero gives too.  Returns the two
// keys.
__device__ __forceinline__ uint32_t ties_win2(float d0, float d1, uint32_t neg, uint32_t top, uint32_t h2) {
  const __nv_bfloat162 hb = __floats2bfloat162_rn(d0, d1);
  const uint32_t w = *reinterpret_cast<const uint32_t*>(&hb) & 0x7FFF7FFFu;
  uint32_t kk;
  asm("{\n .reg .b32 t;\n add.s16x2 t, %1, %2;\n min.s16x2.relu %0, t, %3;\n}" : "=r"(kk) : "r"(w), "r"(neg), "r"(top));
  const uint32_t a2 = kk * 4u + h2;  // lanes: h + 4 b0 and h + 4 b1 (no carry between them)
  asm volatile(
      "{\n"
      " .reg .b32 a0, a1;\n"
      " and.b32 a0, %0, 65535;\n"
      " shr.u32 a1, %0, 16;\n"
      " red.shared.add.u32 [a0], 1;\n"
      " red.shared.add.u32 [a1], 1;\n"
      "}\n" ::"r"(a2)
      : "memory");
  return w;
}

// kBinUnits bins of two deltas, both keys in 16-bit lanes as in ties_win2; neg = -L in both lanes
__device__ __forceinline__ uint32_t ties_units2(float d0, float d1, uint32_t neg, uint32_t h2) {
  const __nv_bfloat162 hb = __floats2bfloat162_rn(d0, d1);
  const uint32_t w = *reinterpret_cast<const uint32_t*>(&hb) & 0x7FFF7FFFu;
  uint32_t t;
  asm("{\n .reg .b32 t;\n add.s16x2 t, %1, %2;\n min.s16x2.relu %0, t, %3;\n}"
      : "=r"(t)
      : "r"(w), "r"(neg), "r"(kWinKeys * 0x00010001u));
  const uint32_t a2 = t * 4u + (((w >> 5) & 0x03FC03FCu) + h2);
  asm volatile(
      "{\n"
      " .reg .b32 a0, a1;\n"
      " and.b32 a0, %0, 65535;\n"
      " shr.u32 a1, %0, 16;\n"
      " red.shared.add.u32 [a0], 1;\n"
      " red.shared.add.u32 [a1], 1;\n"
      "}\n" ::"r"(a2)
      : "memory");
  return w;
}

// number of nonzero keys among the four key words of a vector, in two 16-bit lanes
__device__ __forceinline__ uint32_t nz_halves(uint32_t w0, uint32_t w1, uint32_t w2, uint32_t w3) {
  uint32_t m0, m1, m2, m3;
  asm("min.u16x2 %0, %1, %2;" : "=r"(m0) : "r"(w0), "r"(0x00010001u));
  asm("min.u16x2 %0, %1, %2;" : "=r"(m1) : "r"(w1), "r"(0x00010001u));
  asm("min.u16x2 %0, %1, %2;" : "=r"(m2) : "r"(w2), "r"(0x00010001u));
  asm("min.u16x2 %0, %1, %2;" : "=r"(m3) : "r"(w3), "r"(0x00010001u));
  return m0 + m1 + m2 + m3;
}

// TIES fine bins of two deltas: a nonzero delta whose coarse bin (key bits 7..14) is es
// adds 1 to fine bin (key & 127) of the shared histogram at hist; predicated, no branch
__device__ __forceinline__ void ties_fine2(float d0, float d1, uint32_t es, uint32_t hist) {
  asm volatile(
      "{\n"
      " .reg .pred p0, p1;\n"
      " .reg .b32 w, k0, k1, e0, e1, a0, a1;\n"
      " cvt.rn.bf16x2.f32 w, %2, %1;\n"
      " and.b32 k0, w, 32767;\n"
      " shr.b32 k1, w, 16;\n"
      " and.b32 k1, k1, 32767;\n"
      " shr.b32 e0, k0, 7;\n"
      " shr.b32 e1, k1, 7;\n"
      " setp.ne.f32 p0, %1, 0f00000000;\n"
      " setp.ne.f32 p1, %2, 0f00000000;\n"
      " setp.eq.and.u32 p0, e0, %3, p0;\n"
      " setp.eq.and.u32 p1, e1, %3, p1;\n"
      " and.b32 a0, k0, 127;\n"
      " and.b32 a1, k1, 127;\n"
      " shl.b32 a0, a0, 2;\n"
      " shl.b32 a1, a1, 2;\n"
      " add.u32 a0, a0, %0;\n"
      " add.u32 a1, a1, %0;\n"
      " @p0 red.shared.add.u32 [a0], 1;\n"
      " @p1 red.shared.add.u32 [a1], 1;\n"
      "}\n" ::"r"(hist),
      "f"(d0), "f"(d1), "r"(es)
      : "memory");
}

// Checked build: a work item (block b, experts i0 .. i0 + kc - 1) must lie in the launch's
// block range before the block table is read for it, and the whole block, read from the
// base and those experts, must pass chunk_in_bounds (with its TIES trim group below
// n_groups) before anything is copied or loaded; a failure is recorded in the call's error
// word and the item is skipped.  Constant true in the default build.
template <bool TIES>
__device__ __forceinline__ bool checked_item(const IndexLaunch& p, uint64_t b, uint32_t i0, uint32_t kc,
                                             uint32_t es) {
  if constexpr (!kChecked) return true;
  if (b >= p.b_begin && b < p.b_end && b < p.n_blocks && i0 < p.K && (!TIES || p.blk_group[b] < p.n_groups) &&
      chunk_in_bounds(b, p.b_begin, p.b_end, p.blk_off[b], p.blk_len[b], p.blk_off[b], p.blk_len[b],
                      expert_run(i0, kc), p.K, es, p.expert_origin, p.ext))
    return true;
  atomicOr(p.err, kErrBounds);
  return false;
}

// The k-th largest of the keys counted in h[0 .. 32 N) (SKIP0: h[0] apart), by one warp: lane l
// sums the N bins that rank l-th from the top, a warp scan finds the lane where the running count
// reaches k, and that lane walks its own bins.  True (on every lane) when h holds at least k keys;
// then bin is the bin of the k-th largest and before the number of keys above it; false: before
// is the number of keys.  One thread walking the bins waits for a load per bin: 256 to 384 of
// them took 30-46 us whatever the number of pairs, this takes two.
template <int N, bool SKIP0 = false>
__device__ __forceinline__ bool warp_kth(const unsigned long long* h, unsigned long long k, uint32_t& bin,
                                         unsigned long long& before) {
  const uint32_t lane = threadIdx.x & 31u;
  const uint32_t top = 32u * N - 1u - lane * N;  // this lane's highest bin
  unsigned long long c[N], sum = 0;
#pragma unroll
  for (int j = 0; j < N; ++j) {
    c[j] = SKIP0 && top == (uint32_t)j ? 0ull : h[top - j];
    sum += c[j];
  }
  unsigned long long cum = sum;
#pragma unroll
  for (int s = 1; s < 32; s <<= 1) {
    const unsigned long long o = __shfl_up_sync(0xFFFFFFFFu, cum, s);
    if (lane >= (uint32_t)s) cum += o;
  }
  const uint32_t hit = __ballot_sync(0xFFFFFFFFu, cum >= k);
  if (hit == 0u) {
    before = __shfl_sync(0xFFFFFFFFu, cum, 31);
    return false;
  }
  const int src = __ffs(hit) - 1;
  unsigned long long run = cum - sum;
  uint32_t e = top;
  bool done = false;
#pragma unroll
  for (int j = 0; j < N; ++j) {
    if (!done && run + c[j] >= k) {
      e = top - j;
      done = true;
    }
    if (!done) run += c[j];
  }
  bin = __shfl_sync(0xFFFFFFFFu, e, src);
  before = __shfl_sync(0xFFFFFFFFu, run, src);
  return true;
}

// coarse select of pair x = (expert, trim group), by one warp: bin e* of the upper 8 key bits
// holding the k-th largest key, and the rank of that key inside the bin
__device__ __forceinline__ void coarse_select_pair(const IndexLaunch& p, uint64_t x) {
  if (p.gmiss && p.gmiss[x] == 0u) return;  // its window already gave the threshold
  const unsigned long long k = p.kth[x % p.n_groups];
  uint32_t e = kNoBin;
  unsigned long long before = 0, r = 0;
  if (k != 0) {
    // bin 0 is what the others leave: after masking the omitted elements, zeros, are not counted
    if (!warp_kth<8, true>(p.coarse + x * 256u, k, e, before)) e = 0u;
    r = k - before;
  }
  if ((threadIdx.x & 31u) == 0) {
    p.estar[x] = e;
    p.rank[x] = r;
  }
}

// fine select of pair x, by one warp: the threshold from the fine bins of its coarse bin
__device__ __forceinline__ void fine_select_pair(const IndexLaunch& p, uint64_t x) {
  if (p.gmiss && p.gmiss[x] == 0u) return;  // its window already gave the threshold
  const uint32_t es = p.estar[x];
  uint32_t tau = kTauNone, m;
  unsigned long long before;
  if (es != kNoBin) {
    // only bin 0 can fall short: its uncounted members are exact zeros, key 0
    tau = es << 7;
    if (warp_kth<4>(p.fine + x * 128u, p.rank[x], m, before)) tau |= m;
  }
  if ((threadIdx.x & 31u) == 0) p.tau[x] = tau;
}

// true on every thread of the launch's last CTA to get here (barrier id 1, THREADS threads,
// which may come from different places); what the others wrote before is then visible
template <int THREADS>
__device__ __forceinline__ bool last_cta(unsigned long long* done, volatile int* s_last) {
  __syncwarp();
  asm volatile("bar.sync 1, %0;" ::"n"(THREADS) : "memory");
  if (threadIdx.x == 0) {
    __threadfence();
    *s_last = atomicAdd(done, 1ull) == (unsigned long long)(gridDim.x - 1) ? 1 : 0;
  }
  asm volatile("bar.sync 1, %0;" ::"n"(THREADS) : "memory");
  if (!*s_last) return false;
  __threadfence();
  return true;
}

// f(x) for every marked pair x, by one warp each of the WARPS of a CTA.  The marks are read 32 to a
// warp: a warp that read one pair's after the other's took 84 us for 2,948 pairs.
template <int WARPS, typename F>
__device__ __forceinline__ void for_marked_pairs(const IndexLaunch& p, F f) {
  const uint64_t n = (uint64_t)p.K * p.n_groups;
  const uint32_t lane = threadIdx.x & 31u;
  for (uint64_t x0 = (threadIdx.x >> 5) * 32u; x0 < n; x0 += WARPS * 32u) {
    uint32_t m = __ballot_sync(0xFFFFFFFFu, x0 + lane < n && p.gmiss[x0 + lane] != 0u);
    for (; m; m &= m - 1u) f(x0 + (uint32_t)(__ffs(m) - 1));
  }
}

// The selects of the fallback ride in its passes, whose last CTA makes those of the marked pairs, up to
// so many (expert, group) pairs; above they are launches of their own, with a warp for each pair.  A
// launch that finds no pair marked costs 1 us; one CTA that selects them all costs more the more there
// are, as with density 1 on deltas without zeros, where every pair misses its window.  Index of fp32
// families in blocks of 4096, us, in the pass / own launches: 256 pairs, none marked 53 / 55, all 132 /
// 86; 512 63 / 65, 185 / 104; 1,024 69 / 71, 279 / 110; 2,948 123 / 126, 818 / 234; 9,600 337 / 342,
// 2551 / 686.
constexpr uint64_t kPassSelectPairs = 512;
inline uint32_t selects_in_pass(uint64_t pairs) { return pairs <= kPassSelectPairs ? 1u : 0u; }

// the end of a fallback coarse pass: with few pairs its last CTA makes the coarse select of the marked
// ones, which saves a launch that as a rule would return at once
__device__ __forceinline__ void coarse_pass_end(const IndexLaunch& p, volatile int* s_last) {
  if (!p.select_in_pass || !last_cta<kIxThreads>(p.work + 2, s_last)) return;
  for_marked_pairs<kIxThreads / 32>(p, [&](uint64_t x) { coarse_select_pair(p, x); });
}

template <bool BF16, int KG, int BM>
__global__ void __launch_bounds__(kIxThreads, IxGeo<BM != kBinNone, KG, BM == kBinUnits>::kCtasPerSm)
    index_tma_kernel(const IndexLaunch p, uint32_t G, uint64_t n_items, unsigned long long* work) {
  kernel_begin();
  constexpr bool TIES = BM != kBinNone;
  constexpr uint32_t NB = key_bins<BM>();  // key bins per expert
  using Geo = IxGeo<TIES, KG, BM == kBinUnits>;
  // Whole chunks (IxGeo): one "full" mbarrier counts all the bytes of a chunk's fills and one
  // "empty" mbarrier its releases, so that a consumer waits and releases once per chunk instead
  // of once per fill.
  constexpr bool CW = Geo::kWhole;
  // window bins: the nonzero deltas are counted apart (the bins leave out those below the
  // window); for bf16 from the keys (nz_halves), where key 0 holds exactly the zero deltas (the
  // difference of two distinct bf16 values is at least the smallest bf16 subnormal, whose key
  // is 1)
  constexpr bool KNZ = BM == kBinWindow || BM == kBinUnits;
  constexpr int kIxSlots = Geo::kSlots;
  static_assert(!CW || kIxSlots >= 2 * (KG + 1), "two whole chunks fit the ring");
  constexpr uint32_t kIxSlotBytes = Geo::kSlotBytes;
  constexpr uint32_t ES = BF16 ? 2u : 4u;
  constexpr uint32_t CH = kIxSlotBytes / ES;
  constexpr int V = BF16 ? 8 : 4;
  constexpr int VPT = (int)(CH / (kIxConsumers * V));
  static_assert(VPT >= 1 && CH == (uint32_t)(VPT * kIxConsumers * V), "chunk geometry");
  extern __shared__ __align__(128) uint8_t smem_raw[];
  using Sm = IxSmem<KG, kIxSlots, kIxSlotBytes, NB>;
  Sm& S = *reinterpret_cast<Sm*>(smem_raw);
  const uint32_t tid = threadIdx.x, warp = tid >> 5, lane = tid & 31u;
  // the fallback pass of the windowed catalog runs only when some threshold left its window
  if (BM == kBinCoarse && p.miss && *p.miss == 0u) return;
  if constexpr (KNZ) {  // the packed bin addresses need the histograms below 2^16 - 4 NB
    if (su32(&S.hist[KG - 1][NB - 1]) >= 65536u - 4u * NB) {
      if (threadIdx.x == 0) atomicOr(p.err, kErrInternal);
      return;
    }
  }
  volatile int* abort_flag = &S.abort;
  const uint32_t wl = wait_limit_of(p.wait_limit);

  if (tid == 0) {
    for (int s = 0; s < kIxSlots; ++s) {
      mbar_init(&S.full[s], 1);
      mbar_init(&S.empty[s], kIxConsumers);  // every consumer thread arrives
    }
    mbar_init(&S.cbar, kIxConsumers / 32);
    S.abort = 0;
    mbar_fence_init();
  }
  for (uint32_t x = tid; x < (uint32_t)KG * NB; x += blockDim.x) (&S.hist[0][0])[x] = 0u;
  __syncthreads();

  if (warp == kIxConsumers / 32) {
    // ---------------- producer ----------------
    if (lane == 0) {
      uint32_t fill = 0;
      bool ok = true;
      // whole-chunk publication: chunks published (seq), the oldest one not yet seen released
      // (head) and the ring slots held by chunks head .. seq - 1 (used)
      uint32_t seq = 0, head = 0, used = 0;
      auto reserve = [&](uint32_t nfill) -> bool {
        while (seq - head >= (uint32_t)kIxSlots || used + nfill > (uint32_t)kIxSlots) {
          const uint32_t he = head % kIxSlots;
          if (!mbar_wait(&S.empty[he], (head / kIxSlots) & 1u, abort_flag, wl)) return false;
          used -= S.nf[he];
          ++head;
        }
        return true;
      };
      // publishes one chunk: the base fill and kc expert fills in consecutive slots
      uint32_t item_neg[4] = {0, 0, 0, 0}, item_top[4] = {0, 0, 0, 0};  // the current item's windows
      auto publish = [&](uint32_t item, uint64_t off, uint32_t n, uint32_t last, uint32_t i0,
                         uint32_t kc) -> bool {
        const uint32_t nfill = item == kIxEnd ? 0u : 1u + kc;
        if (!reserve(nfill)) return false;
        if (fill >= (uint32_t)kIxSlots) fence_proxy_async_smem();  // slots the consumers have read are refilled
        const uint32_t e = seq % kIxSlots;
        const uint32_t bytes = (n * ES) & ~15u;
        S.meta[e].off = off;
        S.meta[e].item = item;
        S.meta[e].n = n;
        S.meta[e].last = last;
        S.meta[e].s0 = fill % kIxSlots;
        if constexpr (KNZ) {
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            S.meta[e].wneg[k] = item_neg[k];
            S.meta[e].wtop[k] = item_top[k];
          }
        }
        S.nf[e] = nfill;
        const bool arm = !(seq == 0 && p.stall);  // test hook: the first chunk is never armed
        if (arm) mbar_arrive_expect_tx(&S.full[e], nfill * bytes);
        if (nfill) {
          if (bytes && arm)
            tma_load_1d(S.slot[fill % kIxSlots], static_cast<const char*>(p.base) + off * ES, bytes, &S.full[e]);
          ++fill;
          for (uint32_t k = 0; k < kc; ++k) {
            if (bytes && arm)
              tma_load_1d(S.slot[fill % kIxSlots],
                          static_cast<const char*>(p.experts.p[i0 + k]) + (off - p.expert_origin) * ES, bytes,
                          &S.full[e]);
            ++fill;
          }
        }
        used += nfill;
        ++seq;
        return true;
      };
      auto produce = [&](uint32_t item, uint64_t off, uint32_t n, uint32_t last, const char* src_row,
                         uint32_t bytes) -> bool {
        const uint32_t s = fill % kIxSlots, r = fill / kIxSlots;
        if (fill == 0 && p.stall) {  // test hook: slot 0 is never armed, so its wait runs out
          ++fill;
          return true;
        }
        if (r > 0 && !mbar_wait(&S.empty[s], (r - 1) & 1u, abort_flag, wl)) return false;
        if (r > 0) fence_proxy_async_smem();
        S.meta[s].off = off;
        S.meta[s].item = item;
        S.meta[s].n = n;
        S.meta[s].last = last;
        mbar_arrive_expect_tx(&S.full[s], bytes);
        if (bytes) tma_load_1d(S.slot[s], src_row, bytes, &S.full[s]);
        ++fill;
        return true;
      };
      while (ok) {
        const unsigned long long it = atomicAdd(work, 1ull);
        if (it >= n_items) break;
        const uint64_t b = p.b_begin + it / G;
        const uint32_t i0 = (uint32_t)(it % G) * KG;
        const uint32_t kc = min((uint32_t)KG, p.K - i0);
        if (!checked_item<TIES>(p, b, i0, kc, ES)) continue;
        if (BM == kBinCoarse && p.gmiss) {  // windowed fallback: the marked pairs' groups only
          const uint32_t grp = p.blk_group[b];
          bool any = false;
          for (uint32_t k = 0; k < kc; ++k) any = any || p.gmiss[(uint64_t)(i0 + k) * p.n_groups + grp] != 0u;
          if (!any) continue;
        }
        const uint32_t len = p.blk_len[b];
        const uint64_t off0 = p.blk_off[b];
        const uint32_t nch = (len + CH - 1) / CH;
        if constexpr (CW && KNZ) {
          const uint32_t grp = p.blk_group[b];
#pragma unroll
          for (int k = 0; k < 4; ++k)
            if ((uint32_t)k < kc) {
              win_words(p.win[(uint64_t)(i0 + k) * p.n_groups + grp], item_neg[k], item_top[k]);
              if constexpr (BM == kBinUnits) item_neg[k] -= 0x00010001u;  // -L: no bin apart below the window
            }
        }
        for (uint32_t c = 0; c < nch && ok; ++c) {
          const uint32_t n = min(CH, len - c * CH);
          const uint64_t off = off0 + (uint64_t)c * CH;
          const uint32_t bytes = (n * ES) & ~15u;
          const uint32_t last = c + 1 == nch ? 1u : 0u;
          if constexpr (CW) {
            ok = publish((uint32_t)it, off, n, last, i0, kc);
          } else {
            ok = produce((uint32_t)it, off, n, last, static_cast<const char*>(p.base) + off * ES, bytes);
            for (uint32_t k = 0; k < kc && ok; ++k)
              ok = produce((uint32_t)it, off, n, last,
                           static_cast<const char*>(p.experts.p[i0 + k]) + (off - p.expert_origin) * ES, bytes);
          }
        }
      }
      if (ok) ok = CW ? publish(kIxEnd, 0, 0, 0, 0, 0) : produce(kIxEnd, 0, 0, 0, nullptr, 0);
      if (!ok) {
        atomicOr(p.err, kErrTimeout);
        S.abort = 1;
      }
      // drain: the last use of every slot (entry, when publishing whole chunks) must have
      // landed before the CTA may exit
      const uint32_t nuse = CW ? seq : fill;
      for (uint32_t s = 0; s < (uint32_t)kIxSlots && s < nuse; ++s) {
        const uint32_t lastf = nuse - 1 - ((nuse - 1 + kIxSlots - s) % kIxSlots);
        if (lastf == 0 && p.stall) continue;  // never armed: nothing in flight
        mbar_wait_drain(&S.full[s], (lastf / kIxSlots) & 1u);
      }
    }
    if constexpr (BM == kBinCoarse) {
      __syncwarp();
      coarse_pass_end(p, &S.last);
    }
    return;
  }

  // ---------------- consumers (lane l of the summation order) ----------------
  float ss[KG], mx[KG];
  uint32_t nz[KG];
#pragma unroll
  for (int k = 0; k < KG; ++k) {
    ss[k] = 0.0f;
    mx[k] = 0.0f;
    nz[k] = 0u;
  }
  uint32_t fill = 0, cphase = 0;
  bool alive = true;
  auto wait_full = [&](uint32_t f) -> bool {
    if (!warp_wait(&S.full[f % kIxSlots], (f / kIxSlots) & 1u, abort_flag, wl)) {
      atomicOr(p.err, kErrTimeout);
      S.abort = 1;
      return false;
    }
    return true;
  };
  auto release = [&](uint32_t f) {
    mbar_arrive(&S.empty[f % kIxSlots]);  // every consumer thread: its own reads of the slot are done
  };
  while (alive) {
    if (!wait_full(fill)) break;
    const IxMeta mt = S.meta[fill % kIxSlots];
    if (mt.item == kIxEnd) break;
    const uint64_t b = p.b_begin + mt.item / G;
    const uint32_t i0 = (mt.item % G) * KG;
    const uint32_t kc = min((uint32_t)KG, p.K - i0);
    const uint32_t n = mt.n, n_tma = ((n * ES) & ~15u) / ES;
    const uint64_t off = mt.off;
    float xb[VPT][V];
    uint4 rb[VPT];     // the base vectors as read, for the equality test
    bool bfin = true;  // every base element finite (Inf - Inf and NaN - NaN are not zero)
    const uint32_t s0 = mt.s0;  // whole-chunk publication: the base fill's slot
    {
      const uint8_t* slot = S.slot[CW ? s0 : fill % kIxSlots];
#pragma unroll
      for (int u = 0; u < VPT; ++u) {
        rb[u] = ix_read_raw<BF16>(slot, p.base, off, (tid + (uint32_t)u * kIxConsumers) * V, n, n_tma);
        unpack<BF16>(rb[u], xb[u]);
#pragma unroll
        for (int e = 0; e < V; ++e) bfin = bfin && fabsf(xb[u][e]) < __int_as_float(0x7F800000);
      }
      if constexpr (!CW) {
        release(fill);
        ++fill;
      }
    }
#pragma unroll
    for (int k = 0; k < KG; ++k) {
      if ((uint32_t)k >= kc) break;
      if constexpr (!CW) {
        if (!wait_full(fill)) {
          alive = false;
          break;
        }
      }
      const uint8_t* slot = S.slot[CW ? (s0 + 1u + (uint32_t)k) % kIxSlots : fill % kIxSlots];
      uint4 re[VPT];
      // the equality test pays off only for TIES, whose per-element binning it skips; for
      // the other operators the comparison and vote cost more than the arithmetic they save
      bool same = TIES && bfin;
#pragma unroll
      for (int u = 0; u < VPT; ++u) {
        re[u] = ix_read_raw<BF16>(slot, p.experts.p[i0 + k], off - p.expert_origin,
                                  (tid + (uint32_t)u * kIxConsumers) * V, n, n_tma);
        same = same && same_vec(re[u], rb[u]);
      }
      // a finite vector equal bit for bit to the base gives deltas of exactly +0, which
      // change neither the sum of squares (>= +0), the max (>= +0), the count nor the bins:
      // a warp whose vectors all match skips them (warp-uniform, so the summation order is
      // untouched)
      if (!__all_sync(0xFFFFFFFFu, same)) {
        // kBinWindow, kBinUnits: this expert's window in the block's trim group
        uint32_t wneg = 0, wtop = 0;
        if constexpr (KNZ) {
          wneg = mt.wneg[k < 4 ? k : 0];
          wtop = mt.wtop[k < 4 ? k : 0];
        }
#pragma unroll
        for (int u = 0; u < VPT; ++u) {
          float d[V];
          deltas<BF16>(re[u], xb[u], d);
          // the sum of squares is one fma chain in element order (the canonical order);
          // max |d| and the counts are exact in any order, so they take a tree
#pragma unroll
          for (int e = 0; e < V; ++e) ss[k] = __fmaf_rn(d[e], d[e], ss[k]);
          float m[V / 2];
#pragma unroll
          for (int e = 0; e < V / 2; ++e) m[e] = fmaxf(fabsf(d[2 * e]), fabsf(d[2 * e + 1]));
#pragma unroll
          for (int w = V / 4; w >= 1; w >>= 1)
#pragma unroll
            for (int e = 0; e < w; ++e) m[e] = fmaxf(m[e], m[e + w]);
          mx[k] = fmaxf(mx[k], m[0]);
          if constexpr (KNZ) {
            const uint32_t h2 = su32(&S.hist[k][0]) * 0x00010001u;
            uint32_t wk[V / 2];
#pragma unroll
            for (int e = 0; e < V; e += 2)
              wk[e / 2] = BM == kBinUnits ? ties_units2(d[e], d[e + 1], wneg, h2)
                                          : ties_win2(d[e], d[e + 1], wneg, wtop, h2);
            if constexpr (BF16) nz[k] += nz_halves(wk[0], wk[1], wk[2], wk[3]);
          }
#pragma unroll
          for (int e = 0; e < V; e += 2) {
            if constexpr (BM == kBinCoarse) {
              ties_bin2(d[e], d[e + 1], su32(&S.hist[k][0]));
            } else if constexpr (BM == kBinNone || !BF16) {
              nz[k] += d[e] != 0.0f ? 1u : 0u;
              nz[k] += d[e + 1] != 0.0f ? 1u : 0u;
            }
          }
        }
      }
      if constexpr (!CW) {
        release(fill);
        ++fill;
      }
    }
    if constexpr (CW) {  // every read of the chunk's slots and entry is done
      release(fill);
      ++fill;
    }
    if (!alive || !mt.last) continue;

    // end of the block: the canonical combine, then the statistics (and TIES bins)
#pragma unroll
    for (int k = 0; k < KG; ++k) {
      if constexpr (KNZ && BF16) nz[k] = (nz[k] & 0xFFFFu) + (nz[k] >> 16);  // the two 16-bit lanes
#pragma unroll
      for (int s = 16; s >= 1; s >>= 1) {
        ss[k] = __fadd_rn(ss[k], __shfl_xor_sync(0xFFFFFFFFu, ss[k], s));
        mx[k] = fmaxf(mx[k], __shfl_xor_sync(0xFFFFFFFFu, mx[k], s));
        nz[k] += __shfl_xor_sync(0xFFFFFFFFu, nz[k], s);
      }
      if (lane == 0) {
        S.red_ss[k][warp] = ss[k];
        S.red_mx[k][warp] = mx[k];
        S.red_nz[k][warp] = nz[k];
      }
      ss[k] = 0.0f;
      mx[k] = 0.0f;
      nz[k] = 0u;
    }
    if (!consumer_barrier(&S.cbar, cphase, abort_flag, wl)) {
      atomicOr(p.err, kErrTimeout);
      S.abort = 1;
      break;
    }
    if (warp == 0) {
      uint32_t bad = 0u;
#pragma unroll
      for (int k = 0; k < KG; ++k) {
        float a = lane < 8 ? S.red_ss[k][lane] : 0.0f;
        float m = lane < 8 ? S.red_mx[k][lane] : 0.0f;
        uint32_t c = lane < 8 ? S.red_nz[k][lane] : 0u;
#pragma unroll
        for (int s = 4; s >= 1; s >>= 1) {
          a = __fadd_rn(a, __shfl_xor_sync(0xFFFFFFFFu, a, s));
          m = fmaxf(m, __shfl_xor_sync(0xFFFFFFFFu, m, s));
          c += __shfl_xor_sync(0xFFFFFFFFu, c, s);
        }
        if (lane == 0 && (uint32_t)k < kc) {
          const uint64_t u = (uint64_t)(i0 + k) * p.n_blocks + b;
          p.norm[u] = __fsqrt_rn(a);
          p.maxabs[u] = m;
          if constexpr (!TIES || KNZ) p.nnz[u] = c;
          // a NaN delta makes the sum of squares NaN; an infinite one makes max |delta| infinite
          if (isnan(a) || isinf(m)) bad = 1u;
        }
      }
      if (lane == 0 && bad) atomicOr(p.err, kErrNonfinite);
    }
    if constexpr (TIES) {
      // coarse bins: every nonzero delta added 1 to exactly one bin, the histogram's total is nnz
      if (!consumer_barrier(&S.cbar, cphase, abort_flag, wl)) {
        atomicOr(p.err, kErrTimeout);
        S.abort = 1;
        break;
      }
      // thread t holds bin t (and bins t + 256 and t + 512 where there are as many)
      uint32_t hc[KG], hd[KG], he[KG];
#pragma unroll
      for (int k = 0; k < KG; ++k) {
        hc[k] = S.hist[k][tid];
        S.hist[k][tid] = 0u;
        hd[k] = he[k] = 0u;
        if (KNZ && tid + 256u < NB) {
          hd[k] = S.hist[k][tid + 256u];
          S.hist[k][tid + 256u] = 0u;
        }
        if (KNZ && NB > 512u && tid + 512u < NB) {
          he[k] = S.hist[k][tid + 512u];
          S.hist[k][tid + 512u] = 0u;
        }
        if constexpr (!KNZ) {
          uint32_t w = hc[k] + hd[k];
#pragma unroll
          for (int s = 16; s >= 1; s >>= 1) w += __shfl_xor_sync(0xFFFFFFFFu, w, s);
          if (lane == 0) S.red_nz[k][warp] = w;
        }
      }
      if constexpr (!KNZ) {
        if (!consumer_barrier(&S.cbar, cphase, abort_flag, wl)) {
          atomicOr(p.err, kErrTimeout);
          S.abort = 1;
          break;
        }
      }
      const uint32_t grp = p.blk_group[b];
      const uint32_t len = p.blk_len[b];
#pragma unroll
      for (int k = 0; k < KG; ++k) {
        if ((uint32_t)k >= kc) break;
        uint32_t nzk = 0;
        if constexpr (!KNZ) {
#pragma unroll
          for (int w = 0; w < kIxConsumers / 32; ++w) nzk += S.red_nz[k][w];
          if (tid == 0) p.nnz[(uint64_t)(i0 + k) * p.n_blocks + b] = nzk;
        }
        const uint64_t x = (uint64_t)(i0 + k) * p.n_groups + grp;
        if constexpr (BM == kBinCoarse) {
          unsigned long long c = hc[k];
          if (tid == 0) c += len - nzk;  // zero deltas have key 0
          if (p.unit_hist) p.unit_hist[(((uint64_t)(i0 + k) * p.n_blocks + b) << 8) + tid] = (uint32_t)c;
          if (c) atomicAdd(&p.coarse[x * 256u + tid], c);
        } else if constexpr (BM == kBinUnits) {
          if (tid == 0) {
            hc[k] = 0u;
#pragma unroll
            for (int w = 0; w < kIxConsumers / 32; ++w) hc[k] += S.red_nz[k][w];
          }
          uint32_t* uh = p.unit_hist + ((uint64_t)(i0 + k) * p.n_blocks + b) * kUnitBins;
          unsigned long long* us = p.usum + x * kUnitBins;
          auto flush = [&](uint32_t j, uint32_t n) {
            uh[j] = n;
            if (n) atomicAdd(&us[j], (unsigned long long)n);
          };
          flush(tid, hc[k]);
          flush(tid + 256u, hd[k]);
          if (NB > 512u && tid + 512u < NB) flush(tid + 512u, he[k]);
        } else {
          // bins 1..W are the window's keys, bin W + 1 is above it (bin 0, below it, is dropped)
          const uint32_t W = p.win[x] >> 16;
          auto flush = [&](uint32_t j, uint32_t n) {
            if (n) atomicAdd(j <= W ? &p.wfine[x * kWinKeys + j - 1u] : &p.wabove[x], (unsigned long long)n);
          };
          if (tid > 0) flush(tid, hc[k]);
          flush(tid + 256u, hd[k]);
        }
      }
    }
    if (!consumer_barrier(&S.cbar, cphase, abort_flag, wl)) {
      atomicOr(p.err, kErrTimeout);
      S.abort = 1;
      break;
    }
  }
  if constexpr (BM == kBinCoarse) coarse_pass_end(p, &S.last);
}

// the pair (expert, trim group) of this warp in the select kernels, one warp each
constexpr int kSelThreads = 128;
__device__ __forceinline__ uint64_t select_pair() {
  return (uint64_t)blockIdx.x * (kSelThreads / 32) + (threadIdx.x >> 5);
}
inline unsigned select_grid(uint64_t pairs) { return (unsigned)((pairs + kSelThreads / 32 - 1) / (kSelThreads / 32)); }

__global__ void __launch_bounds__(kSelThreads) ties_coarse_select(const IndexLaunch p) {
  kernel_begin();
  if (p.miss && *p.miss == 0u) return;  // windowed thresholds: no pair needs it
  const uint64_t x = select_pair();
  if (x < (uint64_t)p.K * p.n_groups) coarse_select_pair(p, x);
}

template <bool BF16, int KG>
__global__ void __launch_bounds__(256) ties_fine_kernel(const IndexLaunch p) {
  kernel_begin();
  constexpr int V = BF16 ? 8 : 4;
  __shared__ uint32_t s_fine[KG][128];
  __shared__ int s_last;
  if (p.miss && *p.miss == 0u) return;  // windowed thresholds: no pair needs this pass
  const uint32_t G = (p.K + KG - 1) / KG;
  const uint64_t n_items = p.n_blocks * G;
  const uint32_t tid = threadIdx.x;
  // items (block, group of KG experts) in a grid-stride loop: a grid of resident CTAs
  for (uint64_t it = blockIdx.x; it < n_items; it += gridDim.x) {
    const uint64_t b = it / G;
    const uint32_t i0 = (uint32_t)(it % G) * KG;
    const uint32_t kc = min((uint32_t)KG, p.K - i0);
    if (!checked_item<true>(p, b, i0, kc, BF16 ? 2u : 4u)) continue;  // uniform over the CTA
    const uint32_t grp = p.blk_group[b];

    uint32_t estar[KG];
    uint32_t want = 0u;  // bit k: expert i0+k may hold keys in its bin e*
#pragma unroll
    for (int k = 0; k < KG; ++k) {
      estar[k] = kNoBin;
      if ((uint32_t)k < kc) {
        uint32_t i = i0 + k;
        uint32_t es = p.estar[(uint64_t)i * p.n_groups + grp];
        uint64_t u = (uint64_t)i * p.n_blocks + b;
        const bool read = (!p.mask || ((p.mask[b] >> i) & 1u)) &&  // TIES_MASKED: selected blocks only
                          (!p.gmiss || p.gmiss[(uint64_t)i * p.n_groups + grp] != 0u);  // windowed: missed pairs only
        if (read && es != kNoBin && p.nnz[u] != 0u && (ties_key(p.maxabs[u]) >> 7) >= es) {
          estar[k] = es;
          want |= 1u << k;
        }
      }
    }
    if (want == 0u) continue;  // uniform over the CTA
    if (p.thr_reads && threadIdx.x == 0)
      atomicAdd(p.thr_reads, (unsigned long long)__popc(want) * p.blk_len[b] * (BF16 ? 2u : 4u));
    for (uint32_t x = tid; x < (uint32_t)KG * 128u; x += 256u) (&s_fine[0][0])[x] = 0u;
    __syncthreads();

    const uint64_t off = p.blk_off[b];
    const uint32_t len = p.blk_len[b];
    const uint32_t nvec = (len + V - 1) / V;
    for (uint32_t v = tid; v < nvec; v += kLanes) {
      float xb[V];
      unpack<BF16>(load_vec_raw(p.base, BF16, off, v, len), xb);
#pragma unroll
      for (int k = 0; k < KG; ++k) {
        if (!((want >> k) & 1u)) continue;
        float xe[V];
        unpack<BF16>(load_vec_raw(p.experts.p[i0 + k], BF16, off, v, len), xe);
#pragma unroll
        for (int e = 0; e < V; e += 2)
          ties_fine2(__fsub_rn(xe[e], xb[e]), __fsub_rn(xe[e + 1], xb[e + 1]), estar[k], su32(&s_fine[k][0]));
      }
    }
    __syncthreads();
    for (uint32_t x = tid; x < (uint32_t)KG * 128u; x += 256u) {
      uint32_t k = x >> 7, m = x & 127u;
      if (!((want >> k) & 1u)) continue;
      uint32_t c = s_fine[k][m];
      if (c) atomicAdd(&p.fine[((uint64_t)(i0 + k) * p.n_groups + grp) * 128u + m], (unsigned long long)c);
    }
    __syncthreads();  // the next item clears s_fine
  }
  // the windowed catalog's fallback, with few pairs: the last CTA makes the fine select of the marked ones
  if (!p.select_in_pass || !last_cta<256>(p.work + 3, &s_last)) return;
  for_marked_pairs<8>(p, [&](uint64_t x) { fine_select_pair(p, x); });
}

__global__ void __launch_bounds__(kSelThreads) ties_fine_select(const IndexLaunch p) {
  kernel_begin();
  if (p.miss && *p.miss == 0u) return;
  const uint64_t x = select_pair();
  if (x < (uint64_t)p.K * p.n_groups) fine_select_pair(p, x);
}

// ---- TIES thresholds with a predicted window ----------------------------------------------
//
// The threshold of a trim group is the k-th largest key of its deltas.  A sample predicts
// the bin e of 32 keys that holds it: from every block of the group, vectors at jittered, evenly
// spaced positions (sample_vectors) — every block contributes because the scale of the deltas
// changes from block to block; e is the bin of the k_s-th largest sampled key,
// k_s = max(1, floor(rho * sampled elements)).  The catalog pass then counts the keys of a window
// around it at full resolution (ties_window_select), plus the keys above it, and
// ties_window_finish takes the threshold from those counts.  A pair whose
// threshold lies outside its window is marked, and the two-level select (coarse pass over
// the marked pairs' groups, coarse select, fine pass, fine select) runs for the marked
// pairs only; it does nothing when none is marked.  The prediction affects only which of
// the two exact paths gives a threshold, never its value.

// Vectors sampled from a block of nvec vectors in a group of n_b blocks whose whole blocks have
// nvec0: 8 of each whole block in groups of 256 blocks or more, 32 in groups of 64 or more, up to
// 128 (every one of a small tensor) in smaller groups, so that every group that gets a narrow
// window has 2,000 vectors or more (with 500, one pair in some hundred missed it); a partial
// block in proportion, so that it weighs in the sample what it weighs in the group.  Reading
// every vector of each block up to 4096 elements, and 32 of larger ones, cost 241 us on 371 blocks
// of 4096 elements with 3 experts.
constexpr uint32_t kSampleWide = 8, kSampleWideBlocks = 256;
__device__ __forceinline__ uint32_t sample_vectors(uint32_t n_b, uint32_t nvec, uint32_t nvec0) {
  const uint32_t want = n_b >= kSampleWideBlocks ? kSampleWide : (n_b >= 64u ? 32u : 128u);
  const uint32_t share = (uint32_t)(((uint64_t)want * nvec + nvec0 / 2u) / nvec0);
  return min(max(share, 1u), nvec);
}

// The sample counts 1024 bins of 32 keys.  The deltas of bf16 checkpoints are multiples of the
// elements' last place, so their keys sit on a few values of each binade and a whole binade's
// count does not say where in it the threshold lies (a narrow window placed by interpolation
// missed it, and with the second pass the index of four Llama layers took 2.45 instead of 1.82 ms).
constexpr uint32_t kSampleBins = 1024;

template <bool BF16, int KG>
__global__ void __launch_bounds__(256, 4) ties_sample_kernel(const IndexLaunch p) {
  kernel_begin();
  constexpr uint32_t V = BF16 ? 8u : 4u;
  __shared__ uint32_t hist[KG][kSampleBins];
  __shared__ unsigned long long s_n;  // sampled elements
  const uint2 span = p.samp_span[blockIdx.x];  // {group, first block}: up to p.samp_blocks blocks
  const uint32_t g = span.x, i0 = blockIdx.y * KG;
  const uint32_t kc = min((uint32_t)KG, p.K - i0);
  if (kChecked && (g >= p.n_groups || i0 >= p.K)) {  // uniform over the CTA
    if (threadIdx.x == 0) atomicOr(p.err, kErrBounds);
    return;
  }
  const uint32_t tid = threadIdx.x, warp = tid >> 5, lane = tid & 31u;
  for (uint32_t x = tid; x < (uint32_t)KG * kSampleBins; x += blockDim.x) (&hist[0][0])[x] = 0u;
  if (tid == 0) s_n = 0;
  __syncthreads();
  const uint64_t gb0 = p.n_groups == 1 ? 0 : p.grp_blk0[g], gb1 = p.n_groups == 1 ? p.n_blocks : p.grp_blk0[g + 1];
  const uint64_t b1 = min((uint64_t)span.y + p.samp_blocks, gb1);
  const uint32_t n_b = (uint32_t)min(gb1 - gb0, (uint64_t)0xFFFFFFFFu);
  const uint32_t nvec0 = ((p.n_groups == 1 ? p.max_blk_len : p.blk_len[gb0]) + V - 1) / V;  // of a whole block
  // a warp takes one block with 32 lanes, or (8 vectors each) four blocks with 8 lanes each
  const bool wide = n_b >= kSampleWideBlocks;
  const uint32_t per_warp = wide ? 32u / kSampleWide : 1u, step = wide ? kSampleWide : 32u;
  const uint32_t sub = wide ? lane / kSampleWide : 0u, l = wide ? lane % kSampleWide : lane;
  unsigned long long my_n = 0;
  for (uint64_t b = span.y + warp * per_warp + sub; b < b1; b += 8u * per_warp) {
    if (!checked_item<false>(p, b, i0, kc, BF16 ? 2u : 4u)) continue;
    const uint32_t len = p.blk_len[b];
    const uint64_t off = p.blk_off[b];
    const uint32_t nvec = (len + V - 1) / V;
    const uint32_t n_v = sample_vectors(n_b, nvec, nvec0), per = nvec / n_v;
    for (uint32_t v0 = l; v0 < n_v; v0 += step) {
      uint32_t v = v0;
      if (n_v < nvec) {  // a position in stretch v0 from a hash of (block, stretch)
        uint32_t h = (uint32_t)b * 0x9E3779B1u ^ (v0 + 1u) * 0x85EBCA77u;
        h ^= h >> 15;
        h *= 0x2C1B3C6Du;
        h ^= h >> 12;
        v = v0 * per + h % per;
      }
      my_n += min(V, len - v * V);
      // every checkpoint's vector in flight at once: one memory round trip per position
      const uint4 rb = load_vec_raw(p.base, BF16, off, v, len);
      uint4 re[KG];
#pragma unroll
      for (int k = 0; k < KG; ++k)
        if ((uint32_t)k < kc) re[k] = load_vec_raw(p.experts.p[i0 + k], BF16, off, v, len);
      float xb[V];
      unpack<BF16>(rb, xb);
#pragma unroll
      for (int k = 0; k < KG; ++k) {
        if ((uint32_t)k >= kc) break;
        float xe[V];
        unpack<BF16>(re[k], xe);
#pragma unroll
        for (uint32_t e = 0; e < V; ++e) {
          const float d = __fsub_rn(xe[e], xb[e]);
          if (d != 0.0f) atomicAdd(&hist[k][ties_key(d) >> 5], 1u);
        }
      }
    }
  }
#pragma unroll
  for (int s = 16; s >= 1; s >>= 1) my_n += __shfl_xor_sync(0xFFFFFFFFu, my_n, s);
  if (lane == 0) atomicAdd(&s_n, my_n);
  __syncthreads();
  for (uint32_t x = tid; x < kc * kSampleBins; x += blockDim.x) {
    const uint32_t k = x / kSampleBins, e = x % kSampleBins;
    if (hist[k][e]) atomicAdd(&p.shist[((uint64_t)(i0 + k) * p.n_groups + g) * kSampleBins + e], hist[k][e]);
  }
  if (tid == 0 && blockIdx.y == 0) atomicAdd(&p.scnt[g], s_n);
}

// the window of each (expert, group) from its sample, by one warp: around the bin e of the k_s-th
// largest sampled key, or the three binades around that bin's binade
__global__ void __launch_bounds__(kSelThreads) ties_window_select(const IndexLaunch p) {
  kernel_begin();
  const uint64_t x = select_pair();
  if (x >= (uint64_t)p.K * p.n_groups) return;
  const uint32_t lane = threadIdx.x & 31u, g = (uint32_t)(x % p.n_groups);
  const uint64_t n_b = p.n_groups == 1 ? p.n_blocks : p.grp_blk0[g + 1] - p.grp_blk0[g];
  unsigned long long ks = (unsigned long long)floor((double)p.density * (double)p.scnt[g]);
  if (ks == 0) ks = 1;
  // lane l sums the 32 bins that rank l-th from the top; the first lane whose running count
  // reaches k_s holds e, and its bins go one to a lane for the same again
  static_assert(kSampleBins == 32 * 32, "one run of 32 bins per lane");
  const uint32_t* h = p.shist + x * kSampleBins;
  auto suffix = [&](unsigned long long v) {
#pragma unroll
    for (int s = 1; s < 32; s <<= 1) {
      const unsigned long long o = __shfl_up_sync(0xFFFFFFFFu, v, s);
      if (lane >= (uint32_t)s) v += o;
    }
    return v;
  };
  unsigned long long sum = 0;
  const uint4* h4 = reinterpret_cast<const uint4*>(h + (31u - lane) * 32u);
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    const uint4 c = h4[j];
    sum += (unsigned long long)c.x + c.y + c.z + c.w;
  }
  unsigned long long cum = suffix(sum);
  uint32_t hit = __ballot_sync(0xFFFFFFFFu, cum >= ks), e = 0;
  const bool found = hit != 0u;  // or: fewer nonzero samples than k_s
  if (found) {
    const uint32_t run = 31u - (uint32_t)(__ffs(hit) - 1);
    const unsigned long long before = __shfl_sync(0xFFFFFFFFu, cum - sum, 31 - (int)run);
    cum = before + suffix(h[run * 32u + 31u - lane]);
    hit = __ballot_sync(0xFFFFFFFFu, cum >= ks);
    e = run * 32u + 31u - (uint32_t)(__ffs(hit) - 1);
  }
  if (lane != 0) return;
  uint32_t L = e >= 4u ? min(e / 4u - 1u, 253u) << 7 : 0u, W = kWinKeys;
  if (p.usum) {
    // kBinUnits: the threshold of a plan is that of all blocks or lower, so most of the window
    // lies below the predicted bin: it ends 80 to 207 keys above its middle
    const uint32_t top = (e * 32u + 16u + 80u + 127u) & ~127u;
    L = min(top > kWinKeys ? top - kWinKeys : 0u, 32768u - kWinKeys);
  } else if (found && n_b >= kWinNarrowBlocks) {
    L = (uint32_t)min(max((int32_t)(e * 32u + 16u) - (int32_t)kWinNarrow / 2, 0), 32768 - (int32_t)kWinNarrow);
    W = kWinNarrow;
  }
  p.win[x] = L | W << 16;
}

// the threshold of each (expert, group) from its window counts, or a mark for the
// two-level select when it lies outside the window
__global__ void __launch_bounds__(kSelThreads) ties_window_finish(const IndexLaunch p) {
  kernel_begin();
  const uint64_t x = select_pair();
  if (x >= (uint64_t)p.K * p.n_groups) return;
  const unsigned long long k = p.kth[x % p.n_groups];
  const unsigned long long above = p.wabove[x];
  const uint32_t L = p.win[x] & 0xFFFFu;
  uint32_t tau = kTauNone, j;
  unsigned long long before;
  bool miss = false;
  if (k != 0) {
    miss = above >= k;
    if (!miss) {
      if (warp_kth<(int)kWinKeys / 32>(p.wfine + x * kWinKeys, k - above, j, before)) tau = L + j;
      else if (L == 0) tau = 0;  // every uncounted delta is an exact zero, key 0
      else miss = true;
    }
  }
  if ((threadIdx.x & 31u) != 0) return;
  if (miss) {
    p.gmiss[x] = 1u;
    atomicOr(p.miss, 1u);
  } else {
    p.tau[x] = tau;
  }
}

// TIES after masking: the threshold of each (expert, group) from the sums of its units' bins (all
// units for the catalog, the selected ones for a plan), by one warp, or a mark with the coarse bin
// and rank for the fine pass when it lies outside the window
__global__ void __launch_bounds__(kSelThreads) ties_units_finish(const IndexLaunch p) {
  kernel_begin();
  const uint64_t x = select_pair();
  if (x >= (uint64_t)p.K * p.n_groups) return;
  const unsigned long long k = p.kth[x % p.n_groups];
  const unsigned long long* h = p.usum + x * kUnitBins;
  const uint32_t L = p.win[x] & 0xFFFFu;
  uint32_t tau = kTauNone, j = 0;
  unsigned long long before = 0;
  bool miss = false;
  if (k > h[0]) {
    tau = 0;  // more than there are nonzero deltas
  } else if (k != 0) {
    if (!warp_kth<(int)kUnitBins / 32, true>(h, k, j, before)) {
      // in bin 0, which is key 0 (L = 0) or the keys below 128
      tau = j = 0;
      miss = L != 0;
    } else if (j < L >> 7) {
      miss = true;  // below the window: bin j is coarse bin j
    } else if (j > (L >> 7) + kWinKeys + 1u) {
      miss = true;
      j -= kWinKeys;
    } else {  // key t + L at bin t + (L + t) / 128
      const uint32_t v = j - (L >> 7);
      tau = L + 128u * (v / 129u) + v % 129u;
    }
  }
  if ((threadIdx.x & 31u) != 0) return;
  if (miss) {
    p.estar[x] = j;
    p.rank[x] = k - before;
    p.gmiss[x] = 1u;
    atomicOr(p.miss, 1u);
  } else {
    p.tau[x] = tau;
  }
}

// The sums of a plan's selected units (NB = kUnitBins: for ties_units_finish, 256: the coarse bins).
// One CTA per (expert, window of kUnitWin blocks); a thread owns four bins and adds them for each
// group the window touches, several units' bins in flight.  (One thread per bin that walked 256
// blocks one after the other, each behind its mask word, took 43 us on 1,104 blocks with 7 experts.)
constexpr uint32_t kUnitWin = 32;

template <uint32_t NB>
__global__ void __launch_bounds__(NB / 4) ties_units_sum(const IndexLaunch p, uint32_t n_win) {
  kernel_begin();
  __shared__ uint32_t s_b[kUnitWin], s_g[kUnitWin], s_n;
  const uint32_t i = blockIdx.x / n_win, tid = threadIdx.x;
  const uint64_t b0 = (uint64_t)(blockIdx.x % n_win) * kUnitWin;
  if (tid < 32u) {  // the selected blocks of the window
    const uint64_t b = b0 + tid;
    const bool sel = b < p.n_blocks && ((p.mask[b] >> i) & 1u);
    const uint32_t v = __ballot_sync(0xFFFFFFFFu, sel), at = __popc(v & ((1u << tid) - 1u));
    if (sel) {
      s_b[at] = tid;
      s_g[at] = p.blk_group[b];
    }
    if (tid == 0) s_n = __popc(v);
  }
  __syncthreads();
  const uint32_t n = s_n;
  const uint4* uh = reinterpret_cast<const uint4*>(p.unit_hist + ((uint64_t)i * p.n_blocks + b0) * NB) + tid;
  for (uint32_t a = 0; a < n;) {
    const uint32_t g = s_g[a];
    unsigned long long c[4] = {0, 0, 0, 0};
#pragma unroll 4
    for (; a < n && s_g[a] == g; ++a) {
      const uint4 q = uh[(size_t)s_b[a] * (NB / 4)];
      c[0] += q.x;
      c[1] += q.y;
      c[2] += q.z;
      c[3] += q.w;
    }
    unsigned long long* us = (NB == kUnitBins ? p.usum : p.coarse) + ((uint64_t)i * p.n_groups + g) * NB + tid * 4u;
#pragma unroll
    for (int e = 0; e < 4; ++e)
      if (c[e]) atomicAdd(us + e, c[e]);
  }
}

// the TIES threshold from the coarse bins of the whole family: select the bin, count
// the lower key bits inside it (a second pass over the blocks that can reach it; experts
// addressed with origin 0), select the threshold
template <bool BF16, int KG>
cudaError_t ties_finish_t(const IndexLaunch& p, bool follows, cudaStream_t st) {
  const uint32_t G = (p.K + KG - 1) / KG;
  const uint64_t nsel = (uint64_t)p.K * p.n_groups;
  const unsigned sgrid = select_grid(nsel);
  int dev = 0, sms = 0;
  cudaError_t e;
  if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
  if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
  int per_sm = 0;  // resident CTAs of 256 threads; items by grid stride
  if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, ties_fine_kernel<BF16, KG>, 256, 0)) != cudaSuccess)
    return e;
  uint64_t fgrid = (uint64_t)sms * (per_sm > 0 ? per_sm : 1);
  if (fgrid > p.n_blocks * G) fgrid = p.n_blocks * G;
  if (fgrid == 0) fgrid = 1;
  if (!p.select_in_pass && !p.usum) {  // after masking the units' bins have given the coarse bin
    if ((e = launch_kernel(follows, ties_coarse_select, sgrid, kSelThreads, 0, st, p)) != cudaSuccess) return e;
    follows = true;
  }
  if ((e = launch_kernel(follows, ties_fine_kernel<BF16, KG>, (unsigned)fgrid, 256, 0, st, p)) != cudaSuccess) return e;
  if (!p.select_in_pass) e = launch_kernel(true, ties_fine_select, sgrid, kSelThreads, 0, st, p);
  return e;
}

// one persistent launch of the catalog kernel with binning mode BM
template <bool BF16, int KG, int BM>
cudaError_t launch_pass(const IndexLaunch& p, bool follows, uint32_t G, uint64_t n_items, int sms,
                        unsigned long long* work, cudaStream_t st) {
  constexpr bool ties = BM != kBinNone;
  constexpr uint32_t NB = key_bins<BM>();
  using Geo = IxGeo<ties, KG, BM == kBinUnits>;
  const size_t smem = sizeof(IxSmem<KG, Geo::kSlots, Geo::kSlotBytes, NB>);
  static_assert(Geo::kCtasPerSm * (sizeof(IxSmem<KG, Geo::kSlots, Geo::kSlotBytes, NB>) + 1024) <= 228u * 1024u,
                "the CTAs per SM that the grid assumes fit one SM's shared memory");
  uint64_t grid = (uint64_t)sms * Geo::kCtasPerSm;
  if (grid > n_items) grid = n_items;
  cudaError_t e;
  auto k = index_tma_kernel<BF16, KG, BM>;
  if ((e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)) != cudaSuccess) return e;
  return launch_kernel(follows, k, (unsigned)grid, kIxThreads, smem, st, p, G, n_items, work);
}

template <bool BF16, int KG>
cudaError_t launch_plain_t(const IndexLaunch& p, cudaStream_t st) {
  const uint32_t G = (p.K + KG - 1) / KG;
  const uint64_t n_items = (p.b_end - p.b_begin) * G;
  if (n_items == 0) return cudaSuccess;
  if (n_items > 0x7FFFFFFFull) return cudaErrorInvalidValue;
  int dev = 0, sms = 0;
  cudaError_t e;
  if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
  if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
  return launch_pass<BF16, KG, kBinNone>(p, p.follows, G, n_items, sms, p.work, st);
}

template <bool BF16, int KG>
cudaError_t window_begin_t(const IndexLaunch& p, cudaStream_t st) {
  const uint32_t G = (p.K + KG - 1) / KG;
  const uint64_t nsel = (uint64_t)p.K * p.n_groups;
  if (p.n_samp_spans == 0 || nsel == 0) return cudaSuccess;
  const cudaError_t e = launch_kernel(p.follows, ties_sample_kernel<BF16, KG>, dim3(p.n_samp_spans, G), 256, 0, st, p);
  if (e != cudaSuccess) return e;
  return launch_kernel(true, ties_window_select, select_grid(nsel), kSelThreads, 0, st, p);
}

template <bool BF16, int KG>
cudaError_t launch_ties_t(const IndexLaunch& p, cudaStream_t st) {
  const uint32_t G = (p.K + KG - 1) / KG;
  const uint64_t n_items = (p.b_end - p.b_begin) * G;
  if (n_items == 0) return cudaSuccess;
  if (n_items > 0x7FFFFFFFull) return cudaErrorInvalidValue;
  int dev = 0, sms = 0;
  cudaError_t e;
  if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
  if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
  if (!p.win) {  // the two-level select for every pair
    if ((e = launch_pass<BF16, KG, kBinCoarse>(p, p.follows, G, n_items, sms, p.work, st)) != cudaSuccess) return e;
    if (p.defer_ties_select) return cudaSuccess;
    return ties_finish_t<BF16, KG>(p, true, st);
  }
  // predicted windows: sample, windowed catalog pass, thresholds from the windows, then the
  // two-level select for the pairs whose threshold left its window (a no-op when none did)
  const unsigned sgrid = select_grid((uint64_t)p.K * p.n_groups);
  if ((e = window_begin_t<BF16, KG>(p, st)) != cudaSuccess) return e;
  IndexLaunch q = p;
  q.select_in_pass = selects_in_pass((uint64_t)p.K * p.n_groups);
  if (p.usum) {  // TIES after masking: one pass gives the units' bins and the coarse bins too
    if ((e = launch_pass<BF16, KG, kBinUnits>(p, true, G, n_items, sms, p.work, st)) != cudaSuccess) return e;
    if ((e = launch_kernel(true, ties_units_finish, sgrid, kSelThreads, 0, st, p)) != cudaSuccess) return e;
    return ties_finish_t<BF16, KG>(q, true, st);
  }
  if ((e = launch_pass<BF16, KG, kBinWindow>(p, true, G, n_items, sms, p.work, st)) != cudaSuccess) return e;
  if ((e = launch_kernel(true, ties_window_finish, sgrid, kSelThreads, 0, st, p)) != cudaSuccess) return e;
  if ((e = launch_pass<BF16, KG, kBinCoarse>(q, true, G, n_items, sms, p.work + 1, st)) != cudaSuccess) return e;
  return ties_finish_t<BF16, KG>(q, true, st);
}

template <bool BF16, int KG>
cudaError_t pass_t(const IndexLaunch& p, bool window, cudaStream_t st) {
  const uint32_t G = (p.K + KG - 1) / KG;
  const uint64_t n_items = (p.b_end - p.b_begin) * G;
  if (n_items == 0) return cudaSuccess;
  if (n_items > 0x7FFFFFFFull) return cudaErrorInvalidValue;
  int dev = 0, sms = 0;
  cudaError_t e;
  if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
  if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
  return window ? launch_pass<BF16, KG, kBinWindow>(p, false, G, n_items, sms, p.work, st)
                : launch_pass<BF16, KG, kBinCoarse>(p, false, G, n_items, sms, p.work, st);
}

// f(KG) with the experts per item of the TIES kernels as a constant.  More than 4 experts take
// several items of 4, which read the base again (from L2: neighbouring items run together):
// with 8 per item the histograms leave three CTAs per SM and a chunk's nine fills are waited for
// one by one, 2.45 instead of 1.95 ms on Qwen2.5-0.5B with 8 experts, 4.45 instead of 3.63 with 16.
template <int KG>
using Kg = std::integral_constant<int, KG>;
template <typename F>
cudaError_t by_ties_items(uint32_t K, F f) {
  if (K <= 1) return f(Kg<1>());
  if (K <= 2) return f(Kg<2>());
  return f(Kg<4>());
}

template <bool BF16>
cudaError_t launch_dtype(const IndexLaunch& p, cudaStream_t st) {
  if (p.kth) return by_ties_items(p.K, [&](auto kg) { return launch_ties_t<BF16, decltype(kg)::value>(p, st); });
  if (p.K <= 1) return launch_plain_t<BF16, 1>(p, st);
  if (p.K <= 2) return launch_plain_t<BF16, 2>(p, st);
  if (p.K <= 4) return launch_plain_t<BF16, 4>(p, st);
  return launch_plain_t<BF16, 8>(p, st);
}

}  // namespace

cudaError_t launch_index(const IndexLaunch& p, cudaStream_t st) {
  return p.dtype == MP_BF16 ? launch_dtype<true>(p, st) : launch_dtype<false>(p, st);
}

cudaError_t launch_ties_window_begin(const IndexLaunch& p, cudaStream_t st) {
  if (!p.win || !p.coarse) return cudaErrorInvalidValue;
  return by_ties_items(p.K, [&](auto kg) {
    constexpr int KG = decltype(kg)::value;
    return p.dtype == MP_BF16 ? window_begin_t<true, KG>(p, st) : window_begin_t<false, KG>(p, st);
  });
}

cudaError_t launch_index_pass(const IndexLaunch& p, bool window, cudaStream_t st) {
  if (!p.win || !p.coarse) return cudaErrorInvalidValue;
  return by_ties_items(p.K, [&](auto kg) {
    constexpr int KG = decltype(kg)::value;
    return p.dtype == MP_BF16 ? pass_t<true, KG>(p, window, st) : pass_t<false, KG>(p, window, st);
  });
}

cudaError_t launch_ties_window_end(const IndexLaunch& p, cudaStream_t st) {
  if (!p.win || !p.coarse) return cudaErrorInvalidValue;
  const uint64_t nsel = (uint64_t)p.K * p.n_groups;
  if (nsel == 0) return cudaSuccess;
  return launch_kernel(false, ties_window_finish, select_grid(nsel), kSelThreads, 0, st, p);
}

cudaError_t launch_ties_masked(const IndexLaunch& p, cudaStream_t st) {
  if (!p.unit_hist || !p.mask || p.n_blocks == 0) return cudaErrorInvalidValue;
  const uint32_t n_win = (uint32_t)((p.n_blocks + kUnitWin - 1) / kUnitWin);
  IndexLaunch q = p;
  cudaError_t e;
  if (p.usum) {
    e = launch_kernel(p.follows, ties_units_sum<kUnitBins>, p.K * n_win, kUnitBins / 4, 0, st, p, n_win);
    if (e != cudaSuccess) return e;
    e = launch_kernel(true, ties_units_finish, select_grid((uint64_t)p.K * p.n_groups), kSelThreads, 0, st, p);
    q.select_in_pass = selects_in_pass((uint64_t)p.K * p.n_groups);
  } else {
    e = launch_kernel(p.follows, ties_units_sum<256>, p.K * n_win, 64, 0, st, p, n_win);
  }
  if (e != cudaSuccess) return e;
  q.follows = true;
  return launch_ties_finish(q, st);
}

cudaError_t launch_ties_finish(const IndexLaunch& p, cudaStream_t st) {
  return by_ties_items(p.K, [&](auto kg) {
    constexpr int KG = decltype(kg)::value;
    return p.dtype == MP_BF16 ? ties_finish_t<true, KG>(p, p.follows, st) : ties_finish_t<false, KG>(p, p.follows, st);
  });
}

}  // namespace mp
