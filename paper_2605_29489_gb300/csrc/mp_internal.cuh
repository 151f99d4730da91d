// Internal declarations of the merge library: handle layouts, kernel parameter blocks
// and the launch functions each translation unit provides to api.cu.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <atomic>
#include <memory>
#include <mutex>
#include <string>
#include <utility>
#include <vector>

#include "checked.cuh"
#include "mergepipe.h"

namespace mp {

constexpr uint32_t kMagicIndex = 0x58495043u;  // handle tags
constexpr uint32_t kMagicPlan = 0x4C505043u;
constexpr uint32_t kMagicManifest = 0x464D5043u;

constexpr uint32_t kTauNone = 0x8000u;  // TIES threshold meaning "keep nothing"
constexpr int kLanes = 256;             // lanes of the canonical norm order (one CTA)
constexpr int kMaxK = 32;
constexpr int kCounterSlots = 64;  // realized-byte counters are spread over slots
constexpr int kBackTail = 4;       // words after the summary: the error word (16 bytes), the threshold reads (16)

// device error word bits
// (kErrBounds: a range failed a check of the checked build and was skipped)
enum : uint32_t { kErrNonfinite = 1u, kErrTimeout = 2u, kErrInternal = 4u, kErrMissing = 8u, kErrBounds = 16u };
// nnz of a catalog entry without block statistics (no block holds 2^32 - 1 elements)
constexpr uint32_t kNnzMissing = 0xFFFFFFFFu;

struct ExpertPtrs {
  const void* p[kMaxK];
};

// geometry shared by every handle built from one family
struct Geometry {
  mp_dtype dtype = MP_BF16;
  uint32_t elem_size = 2;
  uint32_t K = 0;
  uint32_t block_elems = 0;
  uint32_t n_tensors = 0;
  uint64_t n_blocks = 0;
  uint64_t n_params = 0;      // sum of numel
  uint64_t span_elems = 0;    // max(offset + numel)
  uint32_t max_blk_len = 0;
  std::vector<uint64_t> t_off, t_numel, t_first_block;
  bool same_as(const Geometry& o) const {
    return dtype == o.dtype && K == o.K && block_elems == o.block_elems && t_off == o.t_off &&
           t_numel == o.t_numel;
  }
};

struct Alloc {
  void* ptr = nullptr;
  size_t bytes = 0;
  cudaStream_t stream = nullptr;
};

// a timing-less event, shared between the handle whose work it ends and the handles which that
// work uses; destroyed with the last of them
class Event {
 public:
  // again: the event may be recorded more than once (what has been waited for is not remembered then)
  cudaError_t make(bool again = false);
  cudaError_t sync() const;  // waits on the host; no runtime call once that has succeeded
  bool over() const { return p->over.load(std::memory_order_acquire); }
  cudaEvent_t get() const { return p ? p->e : nullptr; }
  explicit operator bool() const { return (bool)p; }
  bool operator==(const Event& o) const { return p == o.p; }

 private:
  struct Box {
    cudaEvent_t e = nullptr;
    bool again = false;
    std::atomic<bool> over{false};
    ~Box();
  };
  std::shared_ptr<Box> p;
};

// The ends of the calls that use a handle's device memory (the plans, merges, hashes and validations
// enqueued on it), which mp_free waits for before the memory goes back to the pool.  Calls under
// stream capture are not among them: their events cannot be waited for from the host, and a
// graph's replays need its handles anyway.
class Users {
 public:
  void add(const Event& e);
  void wait();

 private:
  static constexpr size_t kUsersAsk = 16;
  std::mutex mu;
  std::vector<Event> ev;
  size_t ask = kUsersAsk;  // from so many remembered calls on, the runtime is asked which of them are done
};

}  // namespace mp

struct mp_index_s {
  uint32_t magic;
  uint64_t id;
  int device;
  mp::Geometry g;
  int op_kind;
  float density;
  uint32_t trim_scope;
  uint32_t n_groups;
  mp::Alloc mem;
  uint64_t* d_blk_off;     // [n_blocks] element offset of each block
  uint32_t* d_blk_len;     // [n_blocks] elements of each block
  uint32_t* d_blk_group;   // [n_blocks] TIES trim group of each block
  uint32_t* d_blk_tensor;  // [n_blocks] tensor of each block
  uint32_t* d_t_blk0;      // [n_tensors + 1] first block of each tensor, then n_blocks
  bool has_missing;        // some entry has nnz == kNnzMissing (imported catalogs only)
  // TIES_MASKED only: the units' key histograms, [K][n_blocks][256] (coarse bins) or, with a
  // window, [K][n_blocks][kUnitHistBins]; the windows; k of each trim group
  uint32_t* d_unit_hist;
  uint32_t* d_win;                  // null: coarse bins only
  const unsigned long long* d_kth;  // [n_groups]
  // the traversal order of the first operator planned on this index, kept for later plans
  // with the same operator (written once, then only read; guarded by order_mu on the host)
  mp::Alloc order_mem;
  uint32_t* d_order_cache;           // [K * n_blocks]
  unsigned long long* d_order_q;     // candidates
  std::vector<uint8_t> order_key;    // the operator's digest header without the budget
  bool order_captured;               // the cached order was written under stream capture
  cudaEvent_t order_ready;
  std::mutex* order_mu;
  mp::Alloc hash_mem;      // the catalog's block hashes, once computed or imported
  unsigned long long* d_base_hash;    // [n_blocks]
  unsigned long long* d_expert_hash;  // [K][n_blocks]
  float* d_norm;           // [K][n_blocks]
  float* d_maxabs;         // [K][n_blocks]
  uint32_t* d_nnz;         // [K][n_blocks]
  uint32_t* d_tau;         // [K][n_groups] (TIES only)
  uint32_t* d_err;         // error word
  mp::Event done;
  mutable mp::Users users;
  bool captured;           // built under stream capture: waits go through the device
  std::vector<std::pair<void*, size_t>> pinned;  // pinned staging of the uploads (released by mp_free)
  std::vector<uint64_t> h_blk_off;  // host copy of the block table (segments of a host pool)
  std::vector<uint32_t> h_blk_len;
};

struct mp_plan_s {
  uint32_t magic;
  uint64_t id;
  uint64_t index_id;
  int device;
  mp::Geometry g;
  int op_kind;
  float alpha[mp::kMaxK];
  float lambda, density;
  uint32_t trim_scope;
  double drop_p;
  uint64_t seed;
  uint64_t budget;
  uint32_t n_groups;
  mp::Alloc mem;
  uint32_t* d_mask;        // [n_blocks] access mask
  uint32_t* d_order;       // [K*n_blocks] traversal order (first n_cand valid)
  uint64_t* d_summary;     // [8] chat, n_sel, n_cand, set_hash, digest, touched, err, pad
  uint64_t* h_summary;     // pinned host copy of d_summary
  mp::Event done;
  mutable mp::Users users;
  bool captured;           // built under stream capture: waits go through the device
};

struct mp_manifest_s {
  uint32_t magic;
  uint64_t plan_id;
  int device;
  uint32_t K;
  mp::Alloc mem;
  unsigned long long* d_realized;  // [kCounterSlots][K]
  uint32_t* d_err;
  unsigned long long* h_realized;  // pinned host copy (slots summed on host)
  uint32_t* h_err;
  uint64_t planned, touched, digest;
  uint64_t lineage[mp::kMaxK + 1];  // caller ids of M_0..M_K (zeros when none were given)
  mp::Event done;
  bool captured;                    // built under stream capture: waits go through the device
  // hash validation (mp_manifest_validate): checked / mismatched / first bad item, and
  // the output's block hashes
  mp::Alloc valid_mem;
  unsigned long long* d_vresult;   // [3]
  unsigned long long* d_out_hash;  // [n_blocks]
  uint64_t n_blocks;
  mp::Event valid_done;
  bool valid_captured;             // the validation was enqueued under stream capture
};

namespace mp {

// ---- launch accounting (api.cu) ------------------------------------------------------------
void count_launches(uint64_t n);

// Launches kernel k.  follows: the operation ahead of it on the stream is a kernel that this call
// has just launched, so that it may take up its SMs while that one ends (k starts with
// kernel_begin).  That saves about 2 us of the 2.3 us between two such kernels, which counts where a
// call is a chain of kernels of a few us each: 371 ragged blocks with 3 experts, TIES, seven such
// launches, the three calls 122 -> 107 us; 20M elements in blocks of 4096 with 4 experts, TIES
// 290 -> 277, after masking 294 -> 277, AVG/TA 209 -> 203 us.
template <typename... P, typename... A>
inline cudaError_t launch_kernel(bool follows, void (*k)(P...), dim3 grid, unsigned threads, size_t smem,
                                 cudaStream_t st, const A&... a) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = follows ? 1 : 0;
  count_launches(1);
  return cudaLaunchKernelEx(&cfg, k, P(a)...);
}

// ---- error reporting (api.cu) -----------------------------------------------------------
void set_error(const std::string& msg);
// records a string literal as the last error without allocating
void set_static_error(const char* msg);
// test hook: this launch of the planner is to find no room for its cluster
bool cluster_refused();
mp_status cuda_fail(cudaError_t e, const char* what);

// CUDA graphs: a call made while its stream is being captured records its work (and its
// handle's completion event) into the graph.  Such an event cannot be waited for from the
// host, so the waits of a handle built under capture go through the whole device, which
// covers every replay of the graph enqueued so far.
bool capturing(cudaStream_t st);
cudaError_t wait_handle(cudaEvent_t done, bool captured);
cudaError_t stream_wait(cudaStream_t cs, cudaEvent_t ev, bool ev_captured, bool now_captured);

// device-time ranges of the calls (trace.cu): trace_begin records the start of a range on
// st and returns its ticket, or -1 while no trace is recording (or it is full); trace_end
// records the end on the stream that ran the range's work
int trace_begin(uint32_t kind, uint32_t segment, uint32_t stream_kind, cudaStream_t st);
void trace_end(int ticket, cudaStream_t st);
struct TraceScope {
  int ticket;
  cudaStream_t st;
  TraceScope(uint32_t kind, cudaStream_t s) : ticket(trace_begin(kind, 0, 0, s)), st(s) {}
  ~TraceScope() { trace_end(ticket, st); }
};
// host-side NVTX range of an entry point, for the lifetime of the object
struct NvtxScope {
  explicit NvtxScope(const char* name);
  ~NvtxScope();
};

// ---- index (index.cu) -------------------------------------------------------------------
constexpr uint32_t kUnitHistBins = 640;  // bins of a unit's histogram with a window: 384 keys and 256 binades

// Such histograms for blocks of this many elements or more on average: 2.5 KiB per unit instead of
// 1 KiB, in exchange for a second and a third pass over the experts.  Catalog / merge of two Llama
// layers with 4 experts 1.71 / 1.54 -> 0.81 / 0.59 ms; 20M elements with 4 experts in blocks of 4096
// 168 / 220 -> 136 / 73 us; with 16 experts in blocks of 2,504 644 / 377 -> 638 / 182 us.  With 16
// experts in blocks of 1000 (where writing the histograms moves more than the experts hold) the
// merge took 437 instead of 701 us but the catalog 1436 instead of 1224.
constexpr uint64_t kUnitHistElems = 2048;

// And only where the 1.5 KiB per unit that they take more are little against the memory which the
// device has left for the caller's next allocations, an output for instance: at blocks of 2,048 bf16
// elements the larger histograms come to 0.6 of the experts.  Up to kUnitHistSmall bytes nothing is asked.
constexpr uint64_t kUnitHistSmall = 64ull << 20;
constexpr uint64_t kUnitHistShare = 32;  // of the free memory, the part that they may take more

struct IndexLaunch {
  mp_dtype dtype;
  uint32_t K;
  uint64_t n_blocks;
  uint32_t n_groups;
  const void* base;
  ExpertPtrs experts;
  const uint64_t* blk_off;
  const uint32_t* blk_len;
  const uint32_t* blk_group;
  float* norm;
  float* maxabs;
  uint32_t* nnz;
  uint32_t* err;
  // TIES (null when not TIES)
  unsigned long long* coarse;  // [K][n_groups][256]
  unsigned long long* fine;    // [K][n_groups][128]
  const unsigned long long* kth;  // [n_groups] k = floor(density * numel_g)
  uint32_t* estar;             // [K][n_groups] coarse bin of tau (or 0xFFFFFFFF)
  unsigned long long* rank;    // [K][n_groups] rank of tau inside that bin
  uint32_t* tau;               // [K][n_groups]
  // TIES after masking: the catalog keeps each unit's coarse key histogram (256 bins, zero
  // deltas in bin 0); the fine pass then reads only the blocks the plan selected and counts
  // the expert bytes it reads
  uint32_t* unit_hist;         // [K][n_blocks][256], with usum [K][n_blocks][kUnitHistBins], or null
  // with a window for each (expert, group) (device-resident experts, large blocks): the sums
  // of the units' histograms over all blocks (catalog) or the plan's, or null
  unsigned long long* usum;    // [K][n_groups][kUnitHistBins]
  // TIES with a predicted window (also after masking, with usum; null
  // otherwise): a sample of each trim group predicts the coarse bin of its threshold, the
  // catalog pass counts the keys of a window around it at full resolution, and the
  // two-level select runs only for the (expert, group) pairs whose threshold left the window
  float density;                  // rho
  const uint32_t* grp_blk0;       // [n_groups + 1] first block of each trim group, then n_blocks
  const uint2* samp_span;         // [n_samp_spans] {group, first block} of each sampling CTA
  uint32_t n_samp_spans;
  uint32_t samp_blocks;           // blocks per span at most
  uint32_t max_blk_len;           // elements of the longest block
  uint32_t* shist;                // [K][n_groups][1024] bins of 32 keys of the sampled deltas
  unsigned long long* scnt;       // [n_groups] sampled elements
  uint32_t* win;                  // [K][n_groups] the window: first key L | keys W << 16
  unsigned long long* wfine;      // [K][n_groups][384] counts of the keys L .. L + W - 1
  unsigned long long* wabove;     // [K][n_groups] keys above the window
  uint32_t* gmiss;                // [K][n_groups] 1: the pair needs the two-level select
  uint32_t* miss;                 // [1] nonzero when some pair does
  const uint32_t* mask;        // the access mask for the fine pass, or null (every block)
  unsigned long long* thr_reads;  // expert bytes read by the fine pass, or null
  // item counters of the dynamic scheduler, zeroed with the handle: work[0] of the catalog
  // pass, work[1] of the fallback pass; work[2] and work[3] count the CTAs of the fallback pass
  // and of the fine pass that are done (the last one selects, when select_in_pass is set: few pairs)
  unsigned long long* work;
  uint32_t select_in_pass;
  // the launch covers blocks [b_begin, b_end); expert pointers address element
  // expert_origin of the flat layout (0 for resident experts, a segment start when they
  // point into a staging buffer)
  uint64_t b_begin, b_end, expert_origin;
  Extents ext;            // buffer extents, for the checks of the checked build
  bool follows;           // the first launch directly follows another kernel of the call (launch_kernel)
  int defer_ties_select;  // 1: leave the TIES selection to launch_ties_finish
  uint32_t wait_limit;    // try_wait rounds of the pipeline waits (0: the default)
  uint32_t stall;         // test hook: every CTA's first ring fill is never armed
};
cudaError_t launch_index(const IndexLaunch& p, cudaStream_t st);
cudaError_t launch_ties_finish(const IndexLaunch& p, cudaStream_t st);
// the windowed TIES catalog in stages, for a host-resident pool walked in segments: the
// sample and window select over the whole family (experts read in place over the host
// mapping); one pass over blocks [b_begin, b_end) of staged experts with window bins, or with
// coarse bins for the pairs the window finish marked (a launch that returns at once when
// none is); the window finish
cudaError_t launch_ties_window_begin(const IndexLaunch& p, cudaStream_t st);
cudaError_t launch_index_pass(const IndexLaunch& p, bool window, cudaStream_t st);
cudaError_t launch_ties_window_end(const IndexLaunch& p, cudaStream_t st);
// the TIES_MASKED threshold of a plan.  With windows (p.usum): the sums of the selected blocks'
// histograms, which give it unless it leaves its window.  Without: coarse bins summed from the
// per-unit histograms of the selected blocks (zero entries for the others), then the select, fine
// pass and select of launch_ties_finish restricted to the selected blocks (p.mask)
cudaError_t launch_ties_masked(const IndexLaunch& p, cudaStream_t st);

// ---- plan (plan.cu) ---------------------------------------------------------------------
struct PlanLaunch {
  uint32_t K;
  uint64_t n_blocks;
  uint32_t n_groups;
  uint32_t elem_size;
  int op_kind;
  uint32_t score_mode;  // 0: |coef_i| * norm; 1: that per byte of the block
  float coef[kMaxK];   // |alpha_i| or |lambda|
  const uint32_t* blk_len;
  const uint32_t* blk_group;
  const float* norm;
  const float* maxabs;
  const uint32_t* nnz;
  const uint32_t* tau;
  const uint32_t* index_err;
  // tensor-level fallback: with fallback = 1, an (expert, tensor) pair holding an entry
  // with nnz == kNnzMissing is planned as one unit (blk_tensor, t_blk0 as in mp_index_s);
  // with fallback = 0 such an entry is reported (kErrMissing) and never read
  uint32_t fallback;
  uint32_t n_tensors;
  const uint32_t* blk_tensor;
  const uint32_t* t_blk0;
  // the candidates' traversal order does not depend on the budget: a plan may take it
  // from an earlier plan of the same index and operator (cache_*_in), or leave it for
  // later ones (cache_*_out); all null for a plan on its own
  const uint32_t* cache_order_in;
  const unsigned long long* cache_q_in;
  uint32_t* cache_order_out;
  unsigned long long* cache_q_out;
  uint64_t budget;
  uint32_t* mask;
  uint32_t* order;
  uint64_t* summary;
  // pinned host copy of the summary, or null: written at the end of the kernel, but the error word also
  // by a CTA that gives up a barrier
  uint64_t* host_summary;
  uint32_t wait_limit;     // polls of the grid barrier (0: the default)
  uint32_t stall;          // test hook: one CTA of a cooperative launch never comes to a barrier
  uint64_t digest_state;   // FNV-1a state after the digest header (plan_digest_state)
};
// FNV-1a 64 over the digest header (op, theta, B): the part of the digest known to the host
uint64_t plan_digest_state(const uint8_t* header, size_t n);
// scratch bytes the planner needs for n_units units and n_pairs (expert, tensor) pairs
// (n_pairs = 0 without the tensor-level fallback)
size_t plan_scratch_bytes(uint64_t n_units, uint64_t n_pairs);
cudaError_t launch_plan(const PlanLaunch& p, void* scratch, cudaStream_t st);

// ---- merge (merge.cu) -------------------------------------------------------------------
struct MergeLaunch {
  mp_dtype dtype;
  int op_kind;
  uint32_t K;
  uint64_t n_blocks;
  uint32_t block_elems;
  uint32_t n_groups;
  const void* base;
  ExpertPtrs experts;
  void* out;
  const uint64_t* blk_off;
  const uint32_t* blk_len;
  const uint32_t* blk_group;
  const uint32_t* mask;
  const uint32_t* tau;  // TIES
  const uint32_t* nnz;  // renormalised AVG: catalog nonzero counts [K][n_blocks]
  float alpha[kMaxK];
  float lambda;
  float sigma;          // DARE rescale
  uint32_t dare_T;      // DARE keep threshold on 16-bit words
  uint32_t dare_T16;    // min(dare_T, 65535) << 16: the same test on a word in the upper half
                        // (p = 1 has sigma = 0, so a word kept by the clamp adds exactly +-0)
  uint32_t dare_rk[10][2];  // DARE: Philox round keys of the seed (precomputed on the host)
  uint64_t seed;
  unsigned long long* realized;  // [kCounterSlots][K]
  unsigned long long* work;      // chunk counter of the dynamic scheduler (zeroed with the manifest)
  uint32_t* err;
  // the manifest's way back, by the last CTA of the launch that has it set: the realized
  // counters and kBackTail words after the summary's place, with the plan's summary between
  // them, into the host's pinned copy; done counts the CTAs (zeroed with the manifest)
  unsigned long long* back_host;  // or null
  const uint64_t* back_summary;
  unsigned long long* done;
  uint64_t b_begin, b_end, expert_origin;  // as in IndexLaunch
  Extents ext;                             // as in IndexLaunch
  uint32_t touched_only;  // 1: blocks with an empty mask are neither read nor written
  uint32_t wait_limit;    // try_wait rounds of the pipeline waits (0: the default)
  bool follows;           // the launch directly follows another kernel of the call (launch_kernel)
  uint32_t stall;         // test hook: every CTA's first ring fill is never armed
};
cudaError_t launch_merge(const MergeLaunch& p, cudaStream_t st);

// ---- host-pool gather (gather.cu) ---------------------------------------------------------
// copies the planned (block, expert) pairs of blocks [b_begin, b_end) from the experts'
// pinned host memory into staging buffers laid out like the flat checkpoint from element
// `origin` on
struct GatherLaunch {
  uint32_t K;
  uint32_t elem_size;
  uint64_t b_begin, b_end, origin;
  const uint64_t* blk_off;
  const uint32_t* blk_len;
  const uint32_t* mask;   // the access mask of the plan; NULL copies every expert block
  ExpertPtrs src;         // device views of the host experts
  ExpertPtrs dst;         // staging buffers
  unsigned long long* gathered;  // bytes copied, accumulated (may be NULL)
  const uint32_t* gate;          // when set, the launch copies nothing unless *gate != 0
  Extents ext;                   // span: the host experts; x_span: the staging from origin
  uint32_t* err;                 // the call's error word (checked build)
};
cudaError_t launch_gather(const GatherLaunch& g, cudaStream_t st);
// fills by kernel on st (no copy engine)
cudaError_t launch_fill(void* dst, uint32_t byte_value, size_t bytes, cudaStream_t st);
// what a handle's memory starts from, in one launch: copies from pinned host memory (src) and
// zeroed ranges (src null); every address is 16-byte aligned
struct InitSeg {
  void* dst;
  const void* src;
  size_t bytes;
};
struct InitList {
  static constexpr uint32_t kMax = 8;
  InitSeg seg[kMax];
  uint32_t n = 0;
  void add(void* dst, const void* src, size_t bytes) {
    if (bytes) seg[n++] = InitSeg{dst, src, bytes};
  }
};
cudaError_t launch_init(const InitList& l, cudaStream_t st);

// ---- block content hashes (hash.cu) --------------------------------------------------------
// catalog mode (validate = 0): hash every block of the base and of each expert into
// base_hash / expert_hash.  Validation: hash the base, the expert blocks selected by mask
// and every block of out; compare the first two with the catalog (result[0] += blocks
// checked, result[1] += mismatches, result[2] = min mismatching item), write out_hash.
struct HashLaunch {
  uint32_t K;
  uint32_t elem_size;
  uint64_t n_blocks;
  const uint64_t* blk_off;
  const uint32_t* blk_len;
  const void* base;
  ExpertPtrs experts;
  const void* out;
  const uint32_t* mask;
  uint32_t validate;
  unsigned long long* base_hash;    // [n_blocks]
  unsigned long long* expert_hash;  // [K][n_blocks]
  unsigned long long* out_hash;     // [n_blocks]
  unsigned long long* result;       // [3]
  Extents ext;                      // every buffer spans the family (x_span = span)
  uint32_t* err;                    // the call's error word (checked build)
};
cudaError_t launch_hash(const HashLaunch& p, cudaStream_t st);

}  // namespace mp
