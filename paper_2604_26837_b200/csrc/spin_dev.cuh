// Device-side data layout shared by the kernels and the host runtime.
//
// A "set" is one (request, layer, kv head).  Everything a set owns in HBM is reached from
// its SetState and its five directories (two-level indexing, Section 5.4): a directory entry
// names a fixed-size second-level segment in a shared pool; segments are mapped on demand by
// the host runtime's bitmap allocators, so metadata grows with the mapped pages.
#pragma once
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

namespace spin {

constexpr int kHeadDim = 128;
constexpr int kPageTokens = 16;
constexpr int kRowBytes = kHeadDim * 2;                     // one K or V row, bf16
constexpr int kHalfPageBytes = kPageTokens * kRowBytes;     // K half or V half: 4 KiB
constexpr int kPageBytes = 2 * kHalfPageBytes;              // K rows then V rows: 8 KiB
constexpr int kMaxBatch = 256;                              // requests per decode step
constexpr int kMaxBuckets = 64;

enum : int { kKindPage = 0, kKindToken = 1, kKindCluster = 2, kKindPageMean = 3 };
// sticky device error bits (same values as SPIN_DEV_ERR_* of the public header)
enum : int { kOnceSummaries = 1, kOncePages = 2 };
constexpr unsigned kErrBounds = 1u, kErrPageList = 2u, kErrTimeout = 4u, kErrState = 8u;
constexpr int kChunkPages = 8;                              // a set of n pages has room for ceil(n / 8) attention partials
constexpr int kAttnCtaSmem = 8 * kPageTokens * (2 * kRowBytes + 16);   // staged pages of an attention CTA

// Per-set scalars (device resident, updated only by kernels).
struct SetState {
  int32_t n_tokens;       // tokens appended
  int32_t n_partitions;   // indexed partitions = rows of the Meta-partition table
  int32_t n_host_pages;   // entries of the set's CPU page table
  int32_t tail_first;     // CPU-page-table index of the first tail page
  int32_t tail_pages;     // tail pages (0/1 for the page-sized kinds)
  int32_t tail_len;       // tokens in the newest tail page
  int32_t step;           // decode steps done
  int32_t slots;          // S: GPU page table entries
};

// Meta-partition table entry (GPU): token count + residency (Section 5.2).
struct MetaEntry { int32_t tokens; int32_t resident; };
// GPU page table entry: page-centric (slot -> owner) with the recency timestamp.
struct GptEntry { int32_t partition; int32_t phys; int32_t page_idx; int32_t ts; };

struct Counters {
  unsigned long long set_steps, selected_partitions, selected_pages, tail_pages, hit_pages,
      miss_pages, evicted_pages, bypass_pages, candidates_scored;
  unsigned int error_bits;
  unsigned int first_site;   // where the first device-side error was raised (file id * 100000 + line)
  unsigned int dbg[4];       // payload of the first state mismatch: set, device value, host value, epoch
};

struct FetchItem { int32_t host_page; int32_t gpu_page; };

// Everything a kernel needs to find its data; passed by value (fits the 4 KiB param space
// together with a Batch).
struct DevCtx {
  // geometry
  int32_t num_layers, Hq, Hkv, G, kind, topk, n_buckets, trace;
  int32_t seg_shift;            // log2(entries per metadata segment)
  int32_t sum_shift;            // log2(entries per summary segment)
  int32_t sum_entry_bytes;      // 512 (min+max) or 256 (key / centroid)
  int32_t dir_part, dir_slot, dir_page, dir_sum;   // directory lengths per set
  int32_t max_sel, max_parts, max_pages, tail_cap; // scratch strides per batch set
  int32_t max_cand;             // score stride per batch set
  float sm_scale;
  // pools
  int32_t n_gpu_pages, n_host_pages;   // pool sizes, for range checks
  uint8_t *gpu_pages;           // HBM KV pages (cache slots + tails)
  uint8_t *host_pages;          // pinned host KV pages (device-visible address)
  uint8_t *summaries;           // summary segments (64 KiB each)
  MetaEntry *meta_pool;         // GPU
  GptEntry *gpt_pool;           // GPU
  int32_t *off_pool;            // pinned host: Partition Offset table segments
  int32_t *cpt_pool;            // pinned host: CPU page table segments
  int32_t *off_mirror;          // HBM copies of the two host tables (same segment layout), or null:
  int32_t *cpt_mirror;          //   what the decode kernels read, kept up to date by the append kernels
  // per set
  SetState *state;
  int32_t *dir_meta, *dir_gpt, *dir_off, *dir_cpt, *dir_sumseg;
  int32_t *tail_phys;           // [set][tail_cap] GPU pages of the tail
  int32_t *evict_trace;         // [set][max_slots][2] (trace only)
  int32_t max_slots;
  // per-step scratch, indexed by batch set b = i_req * Hkv + head
  float *scores;                // [b][max_cand]
  float *score_xfer;            // [b][max_cand] hand-over buffer of the streaming scoring kernel: all words hold the
                                //   "not written" pattern between steps; the set's selection takes a score out
                                //   (into `scores`) and puts the pattern back
  int32_t *sel_ids;             // [b][max_sel]   chosen candidates, ascending
  int32_t *n_sel;               // [b]
  int32_t *parts;               // [b][max_parts] partitions for the cache manager
  uint32_t *part_mask;          // [b][max_parts] token masks (token kind)
  int32_t *part_state;          // [b][max_parts] 0 hit / 1 admitted / 2 bypassed
  int32_t *n_parts;             // [b]
  int32_t *page_src;            // [b][max_pages+tail_cap] >=0 GPU page, <0 ~host page
  uint32_t *page_mask;          // [b][...]
  int32_t *page_fill;           // [b][...] host page to copy into page_src first, or -1
  int4 *page_desc;              // [b][...] attention's work list, misses first: {page_src, page_fill, mask, list index}
  int32_t *page_slot;           // [b][...] set-local slot / -1 bypass / -2 tail
  int32_t *page_part;           // [b][...] owning partition (-1 tail)
  int32_t *page_pidx;           // [b][...]
  int32_t *n_pages;             // [b]
  FetchItem *fetch_queue;       // misses of the whole batch
  int32_t *fetch_count;
  int32_t fetch_cap;
  float *att_part;              // split-K partials: outputs [b][max_chunks][G][kHeadDim]
  float2 *att_ml;               // ... and their (max, sum) [b][max_chunks][G]
  int32_t *att_count;           // [b] CTAs of the set that have finished (zero before attention)
  unsigned long long *att_words;   // the same for the allocation-free call (null in a context), with
  uint32_t att_call;            //   the call's number in the upper half of each word
  int32_t *link;                // turns on the host link: [0] taken, [64] done (words of their own lines)
  int32_t *sel_count;           // [b] scoring CTAs of the set that have finished (zero between steps)
  int32_t *score_queue;         // next work item of the resident scoring grid (zero between steps)
  int32_t *score_done;          // CTAs of that grid that have left (zero between steps)
  int32_t *scored;              // [b] epoch of the last step whose scores are complete (stand-alone top-k waits on it)
  int32_t *ready;               // [b] how far the set's step is: 2 x epoch once its page list is complete (slots of missed pages
                                //   may be open), 1 more once the missed pages have their slots (page_src)
  int32_t *tail_ready;          // [b] epoch of the last step whose appended rows are in the tail page
  unsigned long long *ready1;   // [b] first flag: epoch of the last step whose missed pages are listed (upper half), with the
                                //   length of the page list and its early descriptors (see first_flag)
  int32_t max_chunks;
  int32_t fetch_mode;           // 0: misses are fetched by the attention kernel; 1: by k_fetch
  int32_t evict_exact;          // 1: exact-demand eviction variant (see spin_config)
  int32_t resident_scoring;     // 0 automatic, 1 always, -1 never (see spin_config)
  Counters *counters;
};

struct Batch {
  int32_t n_req;
  int32_t layer;
  int32_t req[kMaxBatch];
  // local tail of each request after this step's append, as the host has counted it: lets
  // the cache manager lay out the page list without waiting for the append kernel
  int16_t tail_pages[kMaxBatch];
  int16_t tail_len[kMaxBatch];
  // what the host knows of every request's sets without asking the device (all kv heads of a
  // request and layer agree): GPU slots, decode steps done, indexed partitions
  int32_t slots[kMaxBatch];
  int32_t step[kMaxBatch];
  int32_t n_partitions[kMaxBatch];
  int32_t n_tokens[kMaxBatch];   // tokens before this step's append
  int32_t epoch;            // number of this decode call: value of the ready flags it sets
  int32_t append_in_grid;   // the scoring kernel's tail CTAs append this step's tokens
  int32_t attn_set_major;   // attention CTAs ordered set by set (sets become ready one after the
                            // other over a long scoring phase) instead of row 0 of every set first
  int32_t attn_rows, attn_share;   // attention: CTAs of a set as a rule; pages per CTA beyond which a list gets more (see attn_rows_of)
  int32_t read_once;        // what leaves L2 first, kOnceSummaries | kOncePages (see step_reads_once, lists_read_once)
  int32_t attn_cluster, attn_least;   // CTAs of a set are a cluster (their number, else 0); pages that a CTA has at least
};

__host__ __device__ inline int set_index(const DevCtx &c, int req, int layer, int head) {
  return (req * c.num_layers + layer) * c.Hkv + head;
}

#ifdef __CUDACC__
// Records the error bits and, for the first error only, where it was raised (source file id *
// 100000 + line), so that a sticky bit can be traced to its check.
__device__ __forceinline__ void dev_error_site(const DevCtx &c, unsigned bits, unsigned site) {
  if (!c.counters) return;                       // a caller without a context has no status words
  atomicOr(&c.counters->error_bits, bits);
  atomicCAS(&c.counters->first_site, 0u, site);
}
#ifndef SPIN_FILE_ID
#define SPIN_FILE_ID 0
#endif
#define dev_error(c, bits) dev_error_site((c), (bits), (unsigned)(SPIN_FILE_ID * 100000 + __LINE__))
// Two-level lookups.  A negative directory entry means "not mapped": the caller gets nullptr
// and records a bounds error instead of touching memory.
__device__ __forceinline__ MetaEntry *meta_at(const DevCtx &c, int set, int p) {
  int seg = c.dir_meta[(size_t)set * c.dir_part + (p >> c.seg_shift)];
  return seg < 0 ? nullptr : c.meta_pool + ((size_t)seg << c.seg_shift) + (p & ((1 << c.seg_shift) - 1));
}
__device__ __forceinline__ GptEntry *gpt_at(const DevCtx &c, int set, int s) {
  int seg = c.dir_gpt[(size_t)set * c.dir_slot + (s >> c.seg_shift)];
  return seg < 0 ? nullptr : c.gpt_pool + ((size_t)seg << c.seg_shift) + (s & ((1 << c.seg_shift) - 1));
}
__device__ __forceinline__ int32_t *off_at(const DevCtx &c, int set, int p) {
  int seg = c.dir_off[(size_t)set * c.dir_part + (p >> c.seg_shift)];
  return seg < 0 ? nullptr : c.off_pool + ((size_t)seg << c.seg_shift) + (p & ((1 << c.seg_shift) - 1));
}
__device__ __forceinline__ int32_t *cpt_at(const DevCtx &c, int set, int i) {
  int seg = c.dir_cpt[(size_t)set * c.dir_page + (i >> c.seg_shift)];
  return seg < 0 ? nullptr : c.cpt_pool + ((size_t)seg << c.seg_shift) + (i & ((1 << c.seg_shift) - 1));
}
// Lookups for the decode path: the HBM mirror when there is one, else the pinned host table.
__device__ __forceinline__ const int32_t *off_lookup(const DevCtx &c, int set, int p) {
  int seg = c.dir_off[(size_t)set * c.dir_part + (p >> c.seg_shift)];
  if (seg < 0) return nullptr;
  return (c.off_mirror ? c.off_mirror : c.off_pool) + ((size_t)seg << c.seg_shift) + (p & ((1 << c.seg_shift) - 1));
}
__device__ __forceinline__ const int32_t *cpt_lookup(const DevCtx &c, int set, int i) {
  int seg = c.dir_cpt[(size_t)set * c.dir_page + (i >> c.seg_shift)];
  if (seg < 0) return nullptr;
  return (c.cpt_mirror ? c.cpt_mirror : c.cpt_pool) + ((size_t)seg << c.seg_shift) + (i & ((1 << c.seg_shift) - 1));
}
// Append-side helpers: record an entry of a host table in its HBM mirror.
__device__ __forceinline__ void off_mirror_set(const DevCtx &c, int set, int p, int32_t v) {
  if (!c.off_mirror) return;
  int seg = c.dir_off[(size_t)set * c.dir_part + (p >> c.seg_shift)];
  if (seg >= 0) c.off_mirror[((size_t)seg << c.seg_shift) + (p & ((1 << c.seg_shift) - 1))] = v;
}
__device__ __forceinline__ void cpt_mirror_set(const DevCtx &c, int set, int i, int32_t v) {
  if (!c.cpt_mirror) return;
  int seg = c.dir_cpt[(size_t)set * c.dir_page + (i >> c.seg_shift)];
  if (seg >= 0) c.cpt_mirror[((size_t)seg << c.seg_shift) + (i & ((1 << c.seg_shift) - 1))] = v;
}
// Entry e of both host tables of a set -> their HBM copies.
__device__ __forceinline__ void mirror_tables(const DevCtx &c, int set, int e, int n_part, int n_pages) {
  if (!c.off_mirror) return;
  if (e < n_part) { const int32_t *o = off_at(c, set, e); if (o) off_mirror_set(c, set, e, *o); }
  if (e < n_pages) { const int32_t *p = cpt_at(c, set, e); if (p) cpt_mirror_set(c, set, e, *p); }
}
__device__ __forceinline__ uint8_t *summary_at(const DevCtx &c, int set, int e) {
  int seg = c.dir_sumseg[(size_t)set * c.dir_sum + (e >> c.sum_shift)];
  return seg < 0 ? nullptr
                 : c.summaries + (((size_t)seg << c.sum_shift) + (e & ((1 << c.sum_shift) - 1))) *
                                     (size_t)c.sum_entry_bytes;
}
// Programmatic dependent launch: the kernels of a decode step are launched back to back with
// the "programmatic stream serialization" attribute, so a kernel's CTAs may become resident
// while the previous kernel drains.  pdl_launch_next() lets the next kernel start launching;
// pdl_wait_prev() blocks until the previous kernel has completed and its writes are visible.
// Every kernel launched this way calls pdl_wait_prev() before it reads or writes anything
// another kernel touches.
__device__ __forceinline__ void pdl_launch_next() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait_prev() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// The L2 policy of what a call streams through.  Where there is much of it, it is first to leave L2 again, so that what every
// step comes back for stays: the kernels' code (a set's continuation runs through 30 KB of it once per launch), page
// tables, directories.
__device__ __forceinline__ uint64_t stream_policy(bool read_once) {
  uint64_t first, normal;
  asm("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(first));
  asm("createpolicy.fractional.L2::evict_normal.b64 %0, 1.0;" : "=l"(normal));
  return read_once ? first : normal;
}
// A decode step: its pages, where they and the summaries are more than a quarter of L2; its summaries too where L2 (126 MB) does
// not hold both, and in token granularity, where there are few pages.  Steps on three contexts in turn and on the same one
// again, us, with no policy, for the pages, for both:
//   64 sets of 512 candidates, 65 pages (50 MB)      37.6 35.8 36.9   33.9 34.4 36.2
//   128 sets of 250, 33 pages (50 MB)                36.1 34.0 35.1   33.2 33.7 35.1
//   128 sets of up to 375 mean keys, 65 pages (76)   50.3 44.9 45.8   45.5 45.4 46.3
//   4 sets of 65536 tokens (67 MB of summaries)     133.6 133.4 130.6  128.0 128.8 130.0
//   64 sets of 2048, 129 pages (134 MB)              96.7 94.7 95.9   95.2 91.1 93.7, on another GPU in turn - 99.6 98.8
// For the pages and for both: 48 sets of 512 to 8192 candidates, 257 pages (177 MB) 1143 and 1136, 64 sets of 8192 (403 MB) 1275
// and 1271.  8 sets of 2048 (17 MB): 35.8 with none, 36.3 with both.
inline int step_reads_once(int kind, double summaries, double pages) {
  const double all = summaries + pages;
  return all <= 32e6 ? 0 : kOncePages | (kind == kKindToken || all > 110e6 ? kOnceSummaries : 0);
}
// Plain lists: where they do not stay.  Lists that do are found in L2 by the next call on them, which the policy spoils: the same lists
// again, us, without and with it, 444 of 10 pages (36 MB) 7.1 and 8.2, 1024 of 8 (67 MB) 15.2 and 19.4, 256 of 40 (84 MB)
// 17.1 and 18.6, 222 of 48 (87 MB) 15.3 and 14.6, 148 of 80 (97 MB) 18.4 and 16.9; three such sets of lists in turn 9.3 and 9.0, 20.3
// and 19.4, 18.6 and 18.6.
inline int lists_read_once(double pages) { return pages > 85e6 ? kOncePages : 0; }

// Per-set flags that let the attention kernel start on a set as soon as that set's page list
// is complete, while the scoring kernel is still working on other sets.  The producer is
// always resident before a consumer can exist (the consumer kernel is launched with
// programmatic stream serialization after every producer CTA has started), so a consumer only
// ever waits for work that is already running.  The wait is bounded all the same: it gives up
// after ~0.1 s, reports SPIN_DEV_ERR_TIMEOUT and the CTA returns without touching the set.
__device__ __forceinline__ void flag_publish(int32_t *flag, int32_t value) {
  // a release store: everything this thread has written or observed (through the CTA barrier
  // before the call: the other threads' writes too) is visible to whoever acquires the flag
  asm volatile("st.release.gpu.global.s32 [%0], %1;" ::"l"(flag), "r"(value) : "memory");
}
// The first flag of a set carries what its consumers need first: the pages in its list (20 bits; a
// list has at most 50 K selected and 32 K tail pages) and how many of them lead it as early
// descriptors (12 bits; a count beyond that is only a smaller head start).
__device__ __forceinline__ unsigned long long first_flag(int epoch, int n_pages, int n_early) {
  return (unsigned long long)(uint32_t)epoch << 32 | (uint32_t)n_pages << 12 | (uint32_t)min(n_early, 4095);
}
__device__ __forceinline__ void first_flag_publish(unsigned long long *flag, unsigned long long value) {
  asm volatile("st.release.gpu.global.u64 [%0], %1;" ::"l"(flag), "l"(value) : "memory");
}
constexpr int kFlagWaitPolls = 1 << 19;          // ~0.1 s of polls at the capped back-off
__device__ __forceinline__ bool flag_wait(const DevCtx &c, const int32_t *flag, int32_t value,
                                          int max_polls = kFlagWaitPolls) {
  // polls back off from 32 ns to 256 ns: hundreds of waiting CTAs should not keep the L2
  // lines of the flags busy, and a raised flag should still be seen within a fraction of a
  // microsecond
  unsigned pause = 32;
  for (int spin = 0; spin < max_polls; ++spin) {
    int32_t v;
    asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(flag) : "memory");
    if (v == value) return true;
    __nanosleep(pause);
    if (pause < 256) pause <<= 1;
  }
  dev_error(c, kErrTimeout);
  return false;
}

// The same for a set's first flag; its lower half in *word.
__device__ __forceinline__ bool first_flag_wait(const DevCtx &c, const unsigned long long *flag, int32_t epoch, uint32_t *word) {
  unsigned pause = 32;
  for (int spin = 0; spin < kFlagWaitPolls; ++spin) {
    unsigned long long v;
    asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(flag) : "memory");
    *word = (uint32_t)v;
    if ((int32_t)(v >> 32) == epoch) return true;
    __nanosleep(pause);
    if (pause < 256) pause <<= 1;
  }
  dev_error(c, kErrTimeout);
  return false;
}

// A set's `ready` word: the list is complete; its missed pages have their slots too.
__device__ __forceinline__ int32_t list_ready(int32_t epoch) { return (int32_t)(2u * (uint32_t)epoch); }
__device__ __forceinline__ int32_t slots_ready(int32_t epoch) { return (int32_t)(2u * (uint32_t)epoch + 1u); }
// A complete list and the tail page, polled together.
__device__ __forceinline__ bool list_wait(const DevCtx &c, const int32_t *ready, const int32_t *tail_ready, int32_t epoch) {
  unsigned pause = 32;
  for (int spin = 0; spin < kFlagWaitPolls; ++spin) {
    int32_t v0, v1;
    asm volatile("ld.acquire.gpu.global.s32 %0, [%2];\nld.acquire.gpu.global.s32 %1, [%3];" : "=&r"(v0), "=r"(v1) : "l"(ready), "l"(tail_ready) : "memory");
    if ((v0 & ~1) == list_ready(epoch) && v1 == epoch) return true;
    __nanosleep(pause);
    if (pause < 256) pause <<= 1;
  }
  dev_error(c, kErrTimeout);
  return false;
}

// Scores handed from the streaming scoring kernel to a set's selection without a fence: a score
// is one naturally aligned 4-byte store, so the word itself says whether it has arrived.  The
// buffer holds kScoreUnset (a NaN pattern no finite computation produces) in every word between
// steps; the reader polls a word until it differs (bounded), copies it and restores the pattern.
constexpr uint32_t kScoreUnset = 0xffffffffu;
__device__ __forceinline__ float take_score(const DevCtx &c, float *xfer) {
  uint32_t v = kScoreUnset;
  for (int spin = 0; spin < (1 << 20); ++spin) {
    asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(xfer) : "memory");
    if (v != kScoreUnset) break;
    __nanosleep(64);
  }
  if (v == kScoreUnset) { dev_error(c, kErrTimeout); v = 0u; }
  *reinterpret_cast<uint32_t *>(xfer) = kScoreUnset;
  return __uint_as_float(v);
}

__device__ __forceinline__ const uint8_t *page_ptr(const DevCtx &c, int src) {
  return src >= 0 ? c.gpu_pages + (size_t)src * kPageBytes : c.host_pages + (size_t)(~src) * kPageBytes;
}
#endif

// Function attributes (opt-in shared memory), occupancy and SM counts are properties of a device:
// what a launcher remembers about them is kept per device ordinal (the current device, which a
// launcher's caller has made the stream's device).
constexpr int kMaxDevices = 64;
inline int current_device_slot() {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0) dev = 0;
  return dev % kMaxDevices;
}

// Optional per-kernel timing: an event after every launch; durations are read afterwards.
enum : int { kProfAppend = 0, kProfScore, kProfTopk, kProfCache, kProfFetch, kProfAttnSplit,
             kProfAttnMerge, kProfKernels };
struct Prof {
  bool on = false;
  static constexpr size_t kMaxMarks = 1 << 15;
  cudaEvent_t *ev = nullptr;       // kMaxMarks events, created on first use
  int *id = nullptr;               // kernel that ended at mark i (-1 = start of a sequence)
  size_t used = 0;
  void mark(cudaStream_t st, int kernel);
};
inline void prof_mark(Prof *p, cudaStream_t st, int kernel) { if (p && p->on) p->mark(st, kernel); }

// Launch with programmatic stream serialization (and optionally a cluster size).
template <typename... KArgs, typename... Args>
inline cudaError_t launch_pdl(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st,
                              dim3 cluster, Args &&...args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  int na = 0;
  attr[na].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[na].val.programmaticStreamSerializationAllowed = 1;
  ++na;
  if (cluster.x * cluster.y > 1) {
    attr[na].id = cudaLaunchAttributeClusterDimension;
    attr[na].val.clusterDim.x = cluster.x;
    attr[na].val.clusterDim.y = cluster.y;
    attr[na].val.clusterDim.z = 1;
    ++na;
  }
  cfg.attrs = attr;
  cfg.numAttrs = na;
  return cudaLaunchKernelEx(&cfg, kernel, KArgs(args)...);
}

// ---- kernel launchers (each returns the number of kernels it launched) -----------------
struct AppendEdgeArgs {     // one (request) per entry; all its kv heads are processed
  int32_t n_req, layer;
  int32_t req[kMaxBatch];
  int32_t n_tokens[kMaxBatch];   // tokens of the request before this append, as the host has counted them
};
// A directory entry to be written: its index from dir_meta (the five directories follow one another in the
// context's pool) and its value.  The index is 64 bits wide: 256 requests of 80 layers and 8 heads with a million
// tokens each and 16-entry segments have 3.4e9 words of directories.
struct DirUpdate { int64_t at; int32_t value; };
inline DirUpdate dir_update(const int32_t *dirs, const int32_t *entry, int32_t value) { return DirUpdate{(int64_t)(entry - dirs), value}; }
int launch_dir_update(const DevCtx &c, const DirUpdate *u, int n, cudaStream_t st);
int launch_append_bulk(const DevCtx &c, int req, int layer, const __nv_bfloat16 *k,
                       const __nv_bfloat16 *v, int first_page, int n_pages, int first_token_of_call,
                       cudaStream_t st, Prof *prof, uint8_t *stage = nullptr, const int32_t *stage_hp = nullptr);
int launch_append_edge(const DevCtx &c, const AppendEdgeArgs &a, const __nv_bfloat16 *k,
                       const __nv_bfloat16 *v, int n_new, cudaStream_t st, Prof *prof,
                       void *dq = nullptr, const void *sq = nullptr, size_t q_bytes = 0);
int launch_cluster_count(const int32_t *tp, size_t first, size_t rows, int H, int C, int c0, int nc, int32_t *count, unsigned long long *bad,
                         cudaStream_t st);
int launch_cluster_place(const DevCtx &c, int req, int layer, const int32_t *tp, int64_t n, int C, bool first_chunk, bool last_chunk, int32_t *place,
                         cudaStream_t st);
int launch_cluster_tables(const DevCtx &c, int req, int layer, int C, int c0, int nc, int n_pages, int n_tokens, const int32_t *count, int slots,
                          cudaStream_t st);
int launch_cluster_scatter(const DevCtx &c, int req, int layer, const __nv_bfloat16 *k, const __nv_bfloat16 *v,
                           const int32_t *place, int64_t n_tokens, cudaStream_t st);
int launch_cluster_scatter_staged(const DevCtx &c, const __nv_bfloat16 *k, const __nv_bfloat16 *v, const int32_t *place,
                                  int n_tokens, int p0, int m, uint8_t *stage, cudaStream_t st);
int launch_stage_in(void *dq, const void *sq, size_t q_bytes, cudaStream_t st);
int launch_copy_centroids(const DevCtx &c, int req, int layer, const __nv_bfloat16 *cen,
                          int n_clusters, cudaStream_t st);
int launch_select(const DevCtx &c, Batch &b, const __nv_bfloat16 *q, const __nv_bfloat16 *k_new,
                  const __nv_bfloat16 *v_new, int max_cand, cudaStream_t st, Prof *prof);
int launch_cache(const DevCtx &c, const Batch &b, cudaStream_t st, Prof *prof);
int launch_fetch(const DevCtx &c, cudaStream_t st, int sm_count, Prof *prof);
int launch_shrink(const DevCtx &c, int req, int old_S, int new_S, cudaStream_t st);
int launch_wait_probe(const DevCtx &c, int max_polls, cudaStream_t st);
int launch_floor(const DevCtx &c, int token, cudaStream_t st);
int launch_link_probe(const DevCtx &c, int n_pages, cudaStream_t st, int sm_count);
int launch_assign(const DevCtx &c, int req, int layer, int n_clusters, int n_tokens, int32_t *assign, cudaStream_t st);
int launch_move_rows(const DevCtx &c, int req, int layer, const int64_t *dest, int n_tokens, cudaStream_t st);
int launch_reindex_apply(const DevCtx &c, int req, int layer, int n_clusters, int n_folded_pages, int tail_first,
                         int tail_pages, int tail_len, int n_host_pages, const int32_t *assign, cudaStream_t st);
size_t cache_smem_bytes(const DevCtx &c);
int launch_attention(const DevCtx &c, const Batch &b, const __nv_bfloat16 *q,
                     __nv_bfloat16 *out, int max_pages_hint, long long est_pages, cudaStream_t st, Prof *prof);   // est_pages: of all sets' lists together, about

}  // namespace spin
