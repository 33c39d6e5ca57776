// Attention over the selected pages plus the local tail (Section 4.1 "Attention"), fused with
// the page fetch of Retrieve step 4 (Section 5.2): paged GQA decode attention, split over
// CTAs and merged by log-sum-exp.
//
// k_attn: a set's page list is dealt out to the warps of its CTAs (4 warps each), page by page in
// turn, so every warp has its share of the missed pages (which lead the list) and of the hits.  Sets
// have equal shares of the GPU as a rule, lists far above the average more (see attn_rows_of).
// A warp keeps two pages in flight in shared memory and one accumulator over all its pages; the
// CTA has one partial.  A page (8 KiB: 16 K rows, then 16 V rows) is brought in by one
// instruction, a 512-byte bulk copy (TMA) per lane of half the warp, each pair of rows to its own
// place at a stride of 528 bytes; a tile takes the even tokens as its rows 0..7 and the odd ones as
// rows 8..15, so ldmatrix reads 8 rows without a bank conflict.  (256 sets of 56 pages, 8 heads:
// 24.0 us; with a copy per row, twice as many for the SM's one copy unit, 32; per four rows, at a
// two-way conflict, 26.5; per page, at an eight-way conflict, 59.  Rounding against each page's maximum,
// see attend_page, has made the first 24.8 since.)  The page comes from an HBM
// slot for a hit and straight from pinned host memory for a miss, so the missed pages of the step
// are on the host link while the hits are being attended from HBM.  A missed page that was
// admitted to the cache goes from shared memory to its HBM slot by bulk copies too (that is the
// fetch); a bypassed page is only attended.  K Q^T and V^T P^T run on mma.sync m16n8k16 bf16 tiles
// with fp32 accumulators (the page's 16 tokens resp. 16 channels as M, the query heads as N = 8): at
// ~4 flop/byte the kernel is HBM/PCIe bound and tensor tiles are used to take instruction issue
// off the critical path, which is also why the 64..128-row tcgen05 tiles (>90% padding at GQA 4)
// are not.  A set's CTAs merge their partials through distributed shared memory where they are a cluster (up
// to eight of them); else the last one to finish merges them from HBM.
#define SPIN_FILE_ID 4
#include <atomic>
#include <cstdio>
#include <mutex>

#include "../../include/spin.h"
#include "attention_plan.cuh"
#include "spin_dev.cuh"

namespace spin {

#ifdef SPIN_TIMING
__device__ unsigned long long g_dbg_ta[256][16];
__device__ __forceinline__ void dbg_ta(int b, int slot) { if (threadIdx.x == 0) { unsigned long long t; asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t)); g_dbg_ta[b & 255][slot] = t; } }
#else
__device__ __forceinline__ void dbg_ta(int, int) {}
#endif

namespace {

constexpr int kAttnThreads = kAttnWarps * 32;
constexpr int kPairs = kPageTokens, kPairBytes = 2 * kRowBytes;   // pairs of rows of a page: 8 of K, 8 of V
constexpr int kPairStride = kPairBytes + 16;               // 8 pairs' 16-byte pieces fall into 8 bank groups
constexpr int kStageBytes = kPairs * kPairStride;
constexpr int kAttnSmem = kAttnWarps * kWarpStages * kStageBytes;
static_assert(kAttnSmem == kAttnCtaSmem, "what the scoring launcher leaves room for");
constexpr int kCombStride = kHeadDim + 4;                  // floats of a head's row in the warps' exchange area

__device__ __forceinline__ uint32_t smem_u32(const void *p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ void ldmatrix_x4(uint32_t addr, uint32_t &r0, uint32_t &r1, uint32_t &r2, uint32_t &r3) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];\n"
               : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3) : "r"(addr) : "memory");
}
__device__ __forceinline__ void ldmatrix_x4_trans(uint32_t addr, uint32_t &r0, uint32_t &r1, uint32_t &r2, uint32_t &r3) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];\n"
               : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3) : "r"(addr) : "memory");
}
__device__ __forceinline__ void mma_bf16(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3,
                                         uint32_t b0, uint32_t b1) {
  asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};\n"
               : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
               : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
__device__ __forceinline__ uint32_t movmatrix_trans(uint32_t x) {
  uint32_t y;
  asm volatile("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;\n" : "=r"(y) : "r"(x));
  return y;
}
__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
  __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<uint32_t *>(&v);
}

// One warp requests one page: lane i copies pair i of its rows; the stage's mbarrier counts the bytes.  kOnce: the page is to
// leave L2 first (policy).  The copy without a policy is an instruction of its own, since a normal policy costs plain lists 1 %
// (104 shapes, geometric mean).
template <bool kOnce>
__device__ __forceinline__ void request_page(uint32_t sdst, uint32_t bar, const uint8_t *src, int lane, uint64_t policy) {
  if (lane == 0) asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(bar), "r"(kPageBytes) : "memory");
  __syncwarp();
  if (kOnce && lane < kPairs)
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1], %2, [%3], %4;\n"
                 ::"r"(sdst + lane * kPairStride), "l"(src + lane * kPairBytes), "r"(kPairBytes), "r"(bar), "l"(policy) : "memory");
  if (!kOnce && lane < kPairs)
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n"
                 ::"r"(sdst + lane * kPairStride), "l"(src + lane * kPairBytes), "r"(kPairBytes), "r"(bar) : "memory");
}
// Pages that other SMs have written with ordinary stores and announced by a flag may now be read by
// bulk copies.
__device__ __forceinline__ void pages_visible() { asm volatile("fence.proxy.async.global;\n" ::: "memory"); }
__device__ __forceinline__ bool page_test(uint32_t bar, uint32_t parity) {
  uint32_t done;
  asm volatile("{\n.reg .pred p;\nmbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}\n"
               : "=r"(done) : "r"(bar), "r"(parity) : "memory");
  return __all_sync(0xffffffffu, done);
}
// Bounded wait for a stage: false (reported by the caller) if its copies have not landed after seconds.
// A warp that gives a page up waits once more, with the second limit, before its stages are used for
// anything else (see the end of the page loop).
#ifndef SPIN_LANDED_POLLS
#define SPIN_LANDED_POLLS (1 << 22)
#endif
constexpr int kLandedPolls = SPIN_LANDED_POLLS, kDrainPolls = 1 << 22;
__device__ __forceinline__ bool page_landed(uint32_t bar, uint32_t parity, int polls = kLandedPolls) {
  uint32_t done = 0;
#pragma unroll 1
  for (int spin = 0; spin < polls && !done; ++spin)
    asm volatile("{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}\n"
                 : "=r"(done) : "r"(bar), "r"(parity) : "memory");
  return __all_sync(0xffffffffu, done);
}

// A warp's running state.  The tiles are transposed (tokens resp. channels as M = 16, the query
// heads as N = 8): a head is a column, so no row of a tile is padding at 8 heads, and a page costs
// 16 mma instead of the 32 (and the accumulators half the registers) of heads padded to M = 16.
struct WarpAcc {
  float m[2], l[2];           // heads (lane % 4) * 2 + {0, 1}: running max (base-2 logits), this lane's share of the sum
  float o[8][4];              // 16-channel tiles: channels lane / 4 (+ 8), heads as above: [0], [1] resp. [2], [3]
};

// Attend one staged page: S^T = K Q^T (16 tokens x 8 heads), online softmax, O^T = corr O^T + beta V^T P^T.
__device__ __forceinline__ void attend_page(uint32_t spage, const uint32_t (&qb)[8][2], uint32_t mask,
                                            float scale2, WarpAcc &acc, int lane) {
  const int mat = lane >> 3, r8 = lane & 7;
  const uint32_t krow = spage + (uint32_t)(r8 * kPairStride + (mat & 1) * kRowBytes + (mat >> 1) * 16);
  const uint32_t vrow = spage + (uint32_t)((kPairs / 2 + r8) * kPairStride + (mat >> 1) * kRowBytes + (mat & 1) * 16);
  float s[4] = {0.f, 0.f, 0.f, 0.f}, s_odd[4] = {0.f, 0.f, 0.f, 0.f};      // two chains: half the serial mma latency
#pragma unroll
  for (int ks = 0; ks < 8; ks += 2) {
    uint32_t a0, a1, a2, a3, b0, b1, b2, b3;
    ldmatrix_x4(krow + ks * 32, a0, a1, a2, a3);
    ldmatrix_x4(krow + ks * 32 + 32, b0, b1, b2, b3);
    mma_bf16(s, a0, a1, a2, a3, qb[ks][0], qb[ks][1]);
    mma_bf16(s_odd, b0, b1, b2, b3, qb[ks + 1][0], qb[ks + 1][1]);
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) s[i] += s_odd[i];
  // this lane's tokens: 2 * (lane / 4) (tile row lane / 4: s[0], s[1]) and the next (row + 8: s[2], s[3])
  const uint32_t pair = mask >> (2 * (lane >> 2));
  const bool t0 = pair & 1u, t1 = pair & 2u;
  // A page's probabilities are taken against the page's own maximum, and its outputs then scaled into
  // the accumulator in 32 bits: the heaviest token of every page enters the bf16 tiles as exactly 1,
  // so what bf16 costs does not grow with the length of a warp's list.  (Against fp64, 256 sets of 56
  // pages, 8 heads, relative 2-norm: 2.12e-3 with a running maximum over the list, 1.95e-3 with this, at 24.8 us
  // instead of 24.0.)
  float corr[2], beta[2];
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    s[h] = t0 ? s[h] * scale2 : -INFINITY;
    s[2 + h] = t1 ? s[2 + h] * scale2 : -INFINITY;
    float mx = fmaxf(s[h], s[2 + h]);
    mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 4));
    mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 8));
    mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 16));
    const float mn = fmaxf(acc.m[h], mx);
    const float base = mn == -INFINITY ? 0.f : mn;         // all masked so far: every p is 0
    const float own = mx == -INFINITY ? 0.f : mx;
    corr[h] = exp2f(acc.m[h] - base);                      // acc.m = -inf -> 0
    beta[h] = exp2f(mx - base);                            // the page all masked -> 0
    s[h] = exp2f(s[h] - own);
    s[2 + h] = exp2f(s[2 + h] - own);
    acc.l[h] = acc.l[h] * corr[h] + (s[h] + s[2 + h]) * beta[h];
    acc.m[h] = mn;
  }
  // P (token rows, head columns) transposed into the B operand
  const uint32_t b0 = movmatrix_trans(pack_bf16(s[0], s[1])), b1 = movmatrix_trans(pack_bf16(s[2], s[3]));
#pragma unroll
  for (int nt = 0; nt < 8; ++nt) {
    uint32_t a0, a1, a2, a3;
    ldmatrix_x4_trans(vrow + nt * 32, a0, a1, a2, a3);
    float d[4] = {0.f, 0.f, 0.f, 0.f};
    mma_bf16(d, a0, a1, a2, a3, b0, b1);
    acc.o[nt][0] = fmaf(d[0], beta[0], acc.o[nt][0] * corr[0]); acc.o[nt][1] = fmaf(d[1], beta[1], acc.o[nt][1] * corr[1]);
    acc.o[nt][2] = fmaf(d[2], beta[0], acc.o[nt][2] * corr[0]); acc.o[nt][3] = fmaf(d[3], beta[1], acc.o[nt][3] * corr[1]);
  }
}

// Retrieve step 4 for one admitted miss: the staged page goes to its HBM slot, lane i moving pair i.
__device__ __forceinline__ void store_page(uint32_t spage, uint8_t *dst, int lane) {
  if (lane < kPairs)
    asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;\ncp.async.bulk.commit_group;\n"
                 ::"l"(dst + lane * kPairBytes), "r"(spage + lane * kPairStride), "r"(kPairBytes) : "memory");
}
// The lane's copies out of shared memory have read their source.
__device__ __forceinline__ void stores_read() { asm volatile("cp.async.bulk.wait_group.read 0;\n" ::: "memory"); }

// Turns on the host link.  The link needs a few hundred KB of reads in flight; whatever is asked of
// it beyond that waits inside the GPU's memory system, in front of everything else the same SMs
// want from HBM: page lists, flags, hits.  So a page takes a turn before it is requested, and at
// most kLinkWindow turns are open at a time; a page that has landed closes its own.  Both counters
// only ever grow (modulo 2^32).  The lowest open turn never waits for a higher one.
// Measured on the Llama-shaped step (64 sets, 396 missed pages): last set's list of missed pages
// 75-86 us into the step without a limit, 35 us with one; step 112 us without, 106 / 102 / 103 / 107 us
// with a window of 32 / 64 / 96 / 160 pages.
constexpr int kLinkWindow = 64, kLinkDone = 64, kLinkPolls = 1 << 20;
__device__ __forceinline__ int link_turn(const DevCtx &c, int lane) { return lane == 0 ? atomicAdd(c.link, 1) : 0; }   // lane 0's
__device__ __forceinline__ void link_close(const DevCtx &c, int lane) { if (lane == 0) atomicAdd(c.link + kLinkDone, 1); }
__device__ __forceinline__ int link_closed(const DevCtx &c) {
  int done;
  asm volatile("ld.relaxed.gpu.global.s32 %0, [%1];\n" : "=r"(done) : "l"(c.link + kLinkDone) : "memory");
  return done;
}
__device__ __forceinline__ bool link_open(int turn, int closed) {   // turn: lane 0's
  return __shfl_sync(0xffffffffu, (int)((unsigned)turn - (unsigned)closed), 0) < kLinkWindow;
}

// What a lane knows of one page of its warp.
struct PageRef {
  int src, fill, open_idx;    // HBM page (< 0: ~host page); host page to bring in (-1 none); list index of an open slot (-1 none)
  uint32_t mask;
};

// A descriptor that points outside the pools is dropped (and reported), never followed.
__device__ __forceinline__ PageRef in_range(const DevCtx &c, const PageRef &r) {
  const bool ok = (r.src >= 0 ? r.src < c.n_gpu_pages : ~r.src < c.n_host_pages) && r.fill < c.n_host_pages;
  if (ok) return r;
  dev_error(c, kErrBounds);
  return PageRef{0, -1, -1, 0u};
}
__device__ __forceinline__ PageRef page_ref(const DevCtx &c, const Batch &bt, int b, int i_req, int head, size_t pl, int pos) {
  PageRef r{0, -1, -1, 0u};
  if (c.page_desc) {                        // work-ordered descriptors written by the cache manager
    const int4 dsc = __ldcg(c.page_desc + pl + pos);
    r.src = dsc.x; r.fill = dsc.y; r.mask = (uint32_t)dsc.z;
    const bool open = dsc.x == -3;          // early descriptor: page_src[dsc.w] names the slot later
    if (open) { r.open_idx = dsc.w; r.src = 0; }
    if (r.fill == -2) {
      // Retrieve step 3 for a missed page: Partition Offset -> CPU page table, both in pinned
      // host memory (two dependent reads over the host link)
      const int set = set_index(c, bt.req[i_req], bt.layer, head);
      const int32_t *off = off_lookup(c, set, c.page_part[pl + dsc.w]);
      const int32_t *hp = off ? cpt_lookup(c, set, *off + c.page_pidx[pl + dsc.w]) : nullptr;
      const int host_page = hp ? *hp : -1;
      if (host_page < 0) { r.src = -1; r.fill = c.n_host_pages; }         // fails the range check below
      else if (open || r.src >= 0) r.fill = host_page;                    // fetched (admitted, or not yet known)
      else { r.src = ~host_page; r.fill = -1; }                           // bypassed: attend from host
    }
    if (open && r.fill < 0) { r.src = -1; r.fill = c.n_host_pages; }      // an early descriptor always names a host page
  } else {                                  // plain lists, attended in the order given
    r.src = c.page_src[pl + pos];
    r.mask = c.page_mask[pl + pos];
  }
  return in_range(c, r);
}

// Four outputs over their softmax denominator, as bf16; zero where nothing was attended.
__device__ __forceinline__ uint2 normalised(float4 o, float l) {
  if (!(l > 0.f)) return make_uint2(0u, 0u);
  return make_uint2(pack_bf16(o.x / l, o.y / l), pack_bf16(o.z / l, o.w / l));
}

// Four outputs to the caller's buffer, which need not be aligned to more than an element.
__device__ __forceinline__ void store_out(__nv_bfloat16 *dst, uint2 v) {
  if ((reinterpret_cast<uintptr_t>(dst) & 7) == 0) {
    *reinterpret_cast<uint2 *>(dst) = v;
  } else {
    uint16_t *d = reinterpret_cast<uint16_t *>(dst);
    d[0] = (uint16_t)v.x; d[1] = (uint16_t)(v.x >> 16); d[2] = (uint16_t)v.y; d[3] = (uint16_t)(v.y >> 16);
  }
}

// Counts the calling CTA in as one of the set's n_rows; true for the last one.  One thread calls it,
// between two CTA barriers: its release orders the CTA's partials before the count, its acquire the
// count before the CTA's reads of the other rows' partials.  The counters of a decode step are
// cleared by the set's cache manager.  Those of the allocation-free call are 64-bit words that start
// a call at zero because the last row of the call before left them so; the call's number in the
// upper half makes a word right again that an abandoned call has left behind.
__device__ __forceinline__ bool last_row(const DevCtx &c, int b, int n_rows) {
  if (c.att_words) {
    unsigned long long *w = c.att_words + b, old;
    const unsigned long long base = (unsigned long long)c.att_call << 32;
    atomicMax(w, base);
    asm volatile("atom.acq_rel.gpu.global.add.u64 %0, [%1], 1;\n" : "=l"(old) : "l"(w) : "memory");
    const bool last = old - base == (unsigned long long)(n_rows - 1);
    if (last) *w = 0ull;
    return last;
  }
  int old;
  asm volatile("atom.acq_rel.gpu.global.add.s32 %0, [%1], 1;\n" : "=r"(old) : "l"(c.att_count + b) : "memory");
  return old == n_rows - 1;
}

// Merge of a set's partials (one per CTA row; n_rows of them) by the last CTA to finish.  A warp
// owns a head (two of them for G = 8; for G < 4 the warps share a head's rows and meet in shared
// memory at the end), a lane four channels of it: 16-byte loads, kB of them in flight per lane,
// the first batch already while the rows' maxima are being reduced.  Rows are added in a fixed
// order, so the result does not depend on which CTA came last.
// Measured: 64 rows of 4 heads 10 us -> 4.5 us, 3 rows of 4 heads 3.7 -> 1 us.
template <int G>
__device__ __forceinline__ void merge_rows(const DevCtx &c, int b, int n_rows, __nv_bfloat16 *__restrict__ out_rows, float *s_comb) {
  constexpr int kWph = G >= kAttnWarps ? 1 : kAttnWarps / G;               // warps per head
  constexpr int kB = 16;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, sub = warp % kWph;
  const int nk = n_rows > sub ? (n_rows - sub + kWph - 1) / kWph : 0;      // this warp's rows: sub, sub + kWph, ...
#pragma unroll 1
  for (int g = warp / kWph; g < G; g += kAttnWarps) {
    const float2 *ml = c.att_ml + ((size_t)b * c.max_chunks + sub) * G + g;
    const float4 *po = reinterpret_cast<const float4 *>(c.att_part) + (((size_t)b * c.max_chunks + sub) * G + g) * (kHeadDim / 4) + lane;
    constexpr size_t kMlStep = (size_t)kWph * G, kPoStep = (size_t)kWph * G * (kHeadDim / 4);
    float4 v[kB];
    if (nk > 0) {
#pragma unroll
      for (int i = 0; i < kB; ++i) v[i] = __ldcg(po + (size_t)min(i, nk - 1) * kPoStep);
    }
    float2 first = make_float2(-INFINITY, 0.f);                            // rows 0..31 of the warp stay in registers
    if (lane < nk) first = __ldcg(ml + (size_t)lane * kMlStep);
    float mx = first.x;
#pragma unroll 1
    for (int k = lane + 32; k < nk; k += 32) mx = fmaxf(mx, __ldcg(ml + (size_t)k * kMlStep).x);
#pragma unroll
    for (int o = 16; o; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
    float den = 0.f, w = 0.f;
#pragma unroll 1
    for (int k0 = 0; k0 < nk; k0 += kB) {
      if ((k0 & 31) == 0) {                                                // weights of the next 32 rows, one per lane
        if (k0 > 0) first = k0 + lane < nk ? __ldcg(ml + (size_t)(k0 + lane) * kMlStep) : make_float2(-INFINITY, 0.f);
        w = first.x == -INFINITY ? 0.f : exp2f(first.x - mx);
        den += first.y * w;
      }
      if (k0 > 0) {
#pragma unroll
        for (int i = 0; i < kB; ++i) v[i] = __ldcg(po + (size_t)min(k0 + i, nk - 1) * kPoStep);
      }
#pragma unroll
      for (int i = 0; i < kB; ++i) {
        const float wi = __shfl_sync(0xffffffffu, w, (k0 & 31) + i);       // zero beyond the last row
        acc.x = fmaf(v[i].x, wi, acc.x); acc.y = fmaf(v[i].y, wi, acc.y);
        acc.z = fmaf(v[i].z, wi, acc.z); acc.w = fmaf(v[i].w, wi, acc.w);
      }
    }
#pragma unroll
    for (int o = 16; o; o >>= 1) den += __shfl_xor_sync(0xffffffffu, den, o);
    if (kWph > 1) {
      // s_comb: [warps][128 outputs, max, sum]
      float *mine = s_comb + warp * kCombStride;
      reinterpret_cast<float4 *>(mine)[lane] = acc;
      if (lane == 0) { mine[kHeadDim] = mx; mine[kHeadDim + 1] = den; }
      __syncthreads();
      if (sub != 0) return;
      float m_all = -INFINITY;
#pragma unroll
      for (int j = 0; j < kWph; ++j) m_all = fmaxf(m_all, mine[j * kCombStride + kHeadDim]);
      acc = make_float4(0.f, 0.f, 0.f, 0.f);
      den = 0.f;
#pragma unroll
      for (int j = 0; j < kWph; ++j) {
        const float *o = mine + j * kCombStride;
        const float a = o[kHeadDim] == -INFINITY ? 0.f : exp2f(o[kHeadDim] - m_all);
        const float4 x = reinterpret_cast<const float4 *>(o)[lane];
        acc.x = fmaf(x.x, a, acc.x); acc.y = fmaf(x.y, a, acc.y); acc.z = fmaf(x.z, a, acc.z); acc.w = fmaf(x.w, a, acc.w);
        den = fmaf(o[kHeadDim + 1], a, den);
      }
    }
    store_out(out_rows + (size_t)g * kHeadDim + 4 * lane, normalised(acc, den));
  }
}

// CTAs that share a list of np pages.  As a rule the set's part of the GPU; a list that would leave more than
// `share` pages to each of those gets more, up to the grid's rows.
__device__ __forceinline__ int attn_rows_of(const Batch &bt, int np, int share, int max_rows) {
  const int most = min(max_rows, (np + bt.attn_least - 1) / bt.attn_least);
  return min(most, max(bt.attn_rows, (np + share - 1) / share));
}

// Lists whose lengths only the device knows (a set per request): every CTA takes the average from all
// counts.  With half as much again as the average for a share, the further rows of all long lists
// together are at most two thirds of the sets' own, and the grid has that many CTAs behind those,
// which look up what is theirs.
__device__ __forceinline__ int count_of(const DevCtx &c, int i) { return max(0, min(c.n_pages[i], c.max_pages)); }
__device__ __forceinline__ int share_by_counts(const DevCtx &c, const Batch &bt, int *s_sum) {
  int sum = 0;
#pragma unroll 4
  for (int i = threadIdx.x; i < bt.n_req; i += kAttnThreads) sum += count_of(c, i);
  sum = __reduce_add_sync(0xffffffffu, sum);
  if ((threadIdx.x & 31) == 0) s_sum[threadIdx.x >> 5] = sum;
  __syncthreads();
  long long pages = 0;
#pragma unroll
  for (int w = 0; w < kAttnWarps; ++w) pages += s_sum[w];
  return max(bt.attn_share, (int)min(share_of(pages, bt.n_req, bt.attn_rows), 1ll << 30));
}
// The further row that is CTA x's to do, in the order of the sets; false: none.
__device__ __forceinline__ bool further_row(const DevCtx &c, const Batch &bt, int share, int x, int *s_sum, int *s_at, int *b, int *row) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int per = (bt.n_req + kAttnThreads - 1) / kAttnThreads, first = threadIdx.x * per, last = min(bt.n_req, first + per);
  auto further = [&](int i) { return max(0, attn_rows_of(bt, count_of(c, i), share, c.max_chunks) - bt.attn_rows); };
  int mine = 0;
#pragma unroll 4
  for (int i = first; i < last; ++i) mine += further(i);
  int before = mine;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int t = __shfl_up_sync(0xffffffffu, before, o);
    if (lane >= o) before += t;
  }
  __syncthreads();                         // the sums have been read
  if (lane == 31) s_sum[warp] = before;
  if (threadIdx.x == 0) s_at[0] = -1;
  __syncthreads();
  before -= mine;
  for (int w = 0; w < warp; ++w) before += s_sum[w];
  if (x >= before && x < before + mine)
    for (int i = first; i < last; ++i) {
      const int more = further(i);
      if (x < before + more) { s_at[0] = i; s_at[1] = bt.attn_rows + x - before; break; }
      before += more;
    }
  __syncthreads();
  *b = s_at[0]; *row = s_at[1];
  return *b >= 0;
}

// Pages that a list of the request's sets may have.
__device__ __forceinline__ int most_pages(const DevCtx &c, const Batch &bt, int i_req) {
  const int most = c.max_pages + c.tail_cap;
  return c.ready && c.kind != kKindCluster ? min(most, min(c.topk, bt.n_partitions[i_req]) + bt.tail_pages[i_req]) : most;
}

// The part of a set's outputs that a CTA of a cluster has computed, for the other CTAs to read: whether there
// is one, its maxima and sums; the outputs are in the CTA's dynamic shared memory (cluster_outputs).
template <int G> struct ClusterPart { float2 ml[G]; int valid; };
__device__ __forceinline__ float *cluster_outputs(uint8_t *smem) { return reinterpret_cast<float *>(smem + kStageBytes); }   // warp 0's second stage
__device__ __forceinline__ uint32_t remote(uint32_t addr, int rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;\n" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
__device__ __forceinline__ void cluster_meet() {
  asm volatile("barrier.cluster.arrive.release;\nbarrier.cluster.wait.acquire;\n" ::: "memory");
}
// Merge of a set's partials by the cluster that holds all its rows: the first CTA (with eight heads the second too; a thread
// has four outputs of a head) reads the others' partials through distributed shared memory, rows in ascending order, always eight
// of them in flight together, the last row's again where the cluster is smaller.  No partial goes to
// memory, and no fence or counter stands between the rows' ends and the merge.  CTAs that no page of the
// list has reached have left (the cluster's barrier does not wait for those).  The others, the first
// `rows`, all come here, one that has waited for the list in vain too (rows < 0: without a part, and
// it reads none), and none leaves before the last has read.  Where a part is missing nothing is written: the
// outputs of a set whose list has not come to all its rows stay as they were.
// Latency-bound: two cluster barriers and one read of the partials.  Against the merge through memory (write,
// fence, counter, read): 8 lists of up to 40 pages 7.2 -> 6.7 us, decode of one set of 17 pages 22.3 -> 21.2
// (five rows instead of three), of 64 sets of 129 pages 100.9 -> 98.5, of 128 sets of 65 pages 78.1 -> 76.4.
template <int G>
__device__ __forceinline__ void merge_cluster(ClusterPart<G> &part, uint8_t *smem, __nv_bfloat16 *__restrict__ out_rows, int row, int rows) {
  constexpr int kMost = kClusterRows;
  if (threadIdx.x == 0) part.valid = rows > 0;
  cluster_meet();
  const uint32_t ml = smem_u32(&part.ml[0]), ok = smem_u32(&part.valid), outs = smem_u32(cluster_outputs(smem));
#pragma unroll 1
  for (int e = row * kAttnThreads + threadIdx.x; rows > 0 && e < G * (kHeadDim / 4); e += rows * kAttnThreads) {
    const int g = e / (kHeadDim / 4);
    float m[kMost], l[kMost];
    float4 x[kMost];
    int valid[kMost];
#pragma unroll
    for (int r = 0; r < kMost; ++r) {
      const int rank = min(r, rows - 1);
      asm volatile("ld.shared::cluster.s32 %0, [%1];\n" : "=r"(valid[r]) : "r"(remote(ok, rank)));
      asm volatile("ld.shared::cluster.v2.f32 {%0, %1}, [%2];\n" : "=f"(m[r]), "=f"(l[r]) : "r"(remote(ml + g * 8, rank)));
      asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];\n" : "=f"(x[r].x), "=f"(x[r].y), "=f"(x[r].z), "=f"(x[r].w) : "r"(remote(outs + e * 16, rank)));
    }
    float mx = -INFINITY;
    bool whole = true;
#pragma unroll
    for (int r = 0; r < kMost; ++r) {
      whole = whole && valid[r];
      if (r < rows) mx = fmaxf(mx, m[r]);
    }
    float4 o = make_float4(0.f, 0.f, 0.f, 0.f);
    float den = 0.f;
#pragma unroll
    for (int r = 0; r < kMost; ++r)
      if (r < rows) {
        const float a = m[r] == -INFINITY ? 0.f : exp2f(m[r] - mx);
        o.x = fmaf(x[r].x, a, o.x); o.y = fmaf(x[r].y, a, o.y); o.z = fmaf(x[r].z, a, o.z); o.w = fmaf(x[r].w, a, o.w);
        den = fmaf(l[r], a, den);
      }
    if (whole) store_out(out_rows + 4 * e, normalised(o, den));
  }
  cluster_meet();
}

// One row of a set by a CTA of W warps (kAttnWarps; 1 for lists that fit one, which have a single row).
// kTogether: the set has a single row, or its rows are a cluster, which leave their outputs in `part`.  The result says
// how many rows' outputs are there to be merged, 0 if that is settled without this one, -1 if the row has waited for its
// list in vain.
template <int G, int W, bool kTogether, bool kOnce>
__device__ __forceinline__ int attn_row(const DevCtx &c, const Batch &bt, const __nv_bfloat16 *__restrict__ q,
                                         __nv_bfloat16 *__restrict__ out, uint8_t *smem, int b, int row, int max_rows, int share, int counted, ClusterPart<G> *part) {
  __shared__ __align__(8) unsigned long long s_bar[W * kWarpStages];
  __shared__ float s_m[W][G], s_l[W][G];
  __shared__ int sh_ok, sh_np, sh_nm, sh_last;
  const int i_req = b / c.Hkv, head = b % c.Hkv;
  const int np_most = most_pages(c, bt, i_req);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t bar0 = smem_u32(&s_bar[kWarpStages * warp]), stage0 = smem_u32(smem) + (uint32_t)(kWarpStages * warp) * kStageBytes;
  if (lane < kWarpStages) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(bar0 + 8 * lane) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
  }
  int np = 0, nm = 0;                      // pages in the set's list; how many of them are early descriptors
  const size_t pl = (size_t)b * (c.max_pages + c.tail_cap);
  const int mine = row * W + warp;
  PageRef ahead{0, -1, -1, 0u};            // a plain list's first batch, asked for together with the list's length (256 sets of 56 pages: 26.4 -> 25.6 us)
  const bool plain = kTogether && !c.ready;   // (which pages are the row's does not depend on it)
  if (c.ready) {
    // A set raises three flags (the last two are one word).  The first says that its missed pages are listed (the leading
    // descriptors, slot still open): a warp requests its first missed page at once, so the
    // pages cross the host link while the cache manager is still busy.  For the hits a warp waits
    // for the second flag (complete list) and for the tail page, for the slot of a page that has
    // come over the link for the third.
    if (threadIdx.x == 0) {
      uint32_t word = 0;
      sh_ok = first_flag_wait(c, c.ready1 + b, bt.epoch, &word);
      // a count beyond what the set's list can have can neither read past the set's row nor leave
      // the merge waiting for rows that have left
      sh_np = min((int)(word >> 12), np_most);
      sh_nm = (int)(word & 4095u);
    }
    __syncthreads();
    if (!sh_ok) return -1;
    np = sh_np; nm = sh_nm;
    pages_visible();
  } else {
    pdl_wait_prev();
    const int pos = mine + lane * max_rows * W;
    if (plain && pos < c.max_pages) { ahead.src = c.page_src[pl + pos]; ahead.mask = c.page_mask[pl + pos]; }
    np = counted >= 0 ? counted : max(0, min(c.n_pages[b], np_most));
    __syncwarp();
  }
  if (row == 0) dbg_ta(b, 10);
  __nv_bfloat16 *out_rows = out + ((size_t)i_req * c.Hq + head * G) * kHeadDim;
  if (np == 0) {                           // nothing to attend: the set's rows are zero
    if (row == 0)
      for (int e = threadIdx.x; e < G * kHeadDim / 4; e += W * 32) store_out(out_rows + 4 * e, make_uint2(0u, 0u));
    return 0;
  }
  const int n_rows = attn_rows_of(bt, np, share, max_rows);
  if (row >= n_rows) return 0;
  const int stride = n_rows * W;                                   // the warp's pages: mine, mine + stride, ...

  const uint64_t policy = kOnce ? stream_policy(true) : 0ull;
  // Q^T as B-operand fragments: column = lane/4 (query head, zero beyond G), 8 k-steps of 16 channels
  uint32_t qb[8][2];
  WarpAcc acc;
  acc.m[0] = acc.m[1] = -INFINITY;
  acc.l[0] = acc.l[1] = 0.f;
#pragma unroll
  for (int i = 0; i < 8; ++i) { acc.o[i][0] = acc.o[i][1] = acc.o[i][2] = acc.o[i][3] = 0.f; }
  const float scale2 = c.sm_scale * 1.4426950408889634f;

  // The warp's pages in batches of 32, a lane per page (one batch as a rule).  The order in which a
  // warp attends its pages is fixed: the hits of a batch, then its missed pages.
  uint32_t phases = 0;                     // parity of the next wait, a bit per stage
  bool dead = false, listed = c.ready == nullptr, slots_known = listed;    // dead: a wait has run out
  uint32_t issued = 0, on_link = 0;        // stages whose page has been requested and not seen to land; whose page has a turn on the link
#pragma unroll 1
  for (int p0 = mine; p0 < np && !dead; p0 += 32 * stride) {
    const int pos = p0 + lane * stride;
    PageRef ref{0, -1, -1, 0u};
    auto request = [&](int stage, int j) {
      const int src = __shfl_sync(0xffffffffu, ref.src, j), fill = __shfl_sync(0xffffffffu, ref.fill, j);
      request_page<kOnce>(stage0 + stage * kStageBytes, bar0 + 8 * stage, fill >= 0 ? c.host_pages + (size_t)fill * kPageBytes : page_ptr(c, src), lane, policy);
    };
    // a missed page is requested as soon as it is known (early pages lead the list: lane 0's is one of
    // them): its turn, its descriptor and the count of closed turns are asked for together
    const bool early = pos < min(nm, np);
    const bool early0 = p0 < nm && !listed;
    int turn0 = 0, turn1 = 0, closed = 0;  // the stages' turns on the host link (lane 0's)
    if (early0) { turn0 = link_turn(c, lane); closed = link_closed(c); on_link = 1u; }
    if (early) ref = page_ref(c, bt, b, i_req, head, pl, pos);
    if (early0 && link_open(turn0, closed)) { request(0, 0); issued = 1u; }
    if (p0 == mine) {
      const int qr = lane >> 2;
      const uint32_t *qrow = reinterpret_cast<const uint32_t *>(q + ((size_t)i_req * c.Hq + head * G + (qr < G ? qr : 0)) * kHeadDim);
#pragma unroll
      for (int ks = 0; ks < 8; ++ks) {
        qb[ks][0] = qr < G ? qrow[ks * 8 + (lane & 3)] : 0u;
        qb[ks][1] = qr < G ? qrow[ks * 8 + 4 + (lane & 3)] : 0u;
      }
    }
    if (!listed) {
      int ok = 1;
      if (lane == 0) ok = list_wait(c, c.ready + b, c.tail_ready + b, bt.epoch);
      listed = __shfl_sync(0xffffffffu, ok, 0) != 0;
      __syncwarp();                        // lane 0's acquire comes before every lane's reads of the list
      pages_visible();
      if (!listed) { dead = true; break; } // reported by the wait: nothing more is requested
    }
    if (pos < np && !early) ref = plain && p0 == mine ? in_range(c, ahead) : page_ref(c, bt, b, i_req, head, pl, pos);
    const bool from_host = ref.fill >= 0 || ref.src < 0;
    const uint32_t here = __ballot_sync(0xffffffffu, pos < np), host = __ballot_sync(0xffffffffu, from_host) & here;   // (lane 0 is here)
    if (row == 0 && p0 == mine) dbg_ta(b, 11);
    if (host == 0 && !early0) {
      // nothing to bring in (the usual batch): pages 0, 1, 2, ... through the two stages in turn
      const int n = __popc(here);
      request(0, 0);
      if (n > 1) request(1, 1);
#pragma unroll 1
      for (int j = 0; j < n; ++j) {
        const int st = j & 1;
        const uint32_t mask = __shfl_sync(0xffffffffu, ref.mask, j);
        if (!page_landed(bar0 + 8 * st, (phases >> st) & 1u)) {
          if (lane == 0) dev_error(c, kErrTimeout);
          issued = 1u << st | (j + 1 < n ? 2u >> st : 0u);
          dead = true;
          break;
        }
        phases ^= 1u << st;
        attend_page(stage0 + st * kStageBytes, qb, mask, scale2, acc, lane);
        __syncwarp();                      // every lane has read the stage
        if (j + 2 < n) request(st, j + 2);
      }
      if (row == 0 && p0 == mine) dbg_ta(b, 12);
      continue;
    }
    // The first missed page has stage 0 from the start; the hits go through stage 1 meanwhile, then
    // the other missed pages through both.
    const uint32_t hosted = host | (early0 ? 1u : 0u);    // (a dropped early descriptor keeps its turn and is attended with an empty mask)
    uint32_t misses = hosted & here, hits = here & ~hosted;
    auto pop = [](uint32_t &m) { const int j = __ffs(m) - 1; m &= m - 1; return j; };
    auto next = [&]() { return hits ? pop(hits) : misses ? pop(misses) : -1; };
    int in0 = early0 ? 0 : -1, in1 = -1;   // the pages (lanes) that have the two stages
    if (early0) misses &= ~1u;
    else { in0 = pop(misses); turn0 = link_turn(c, lane); on_link = 1u; }
    int hits_in1 = __popc(hits), cur = hits_in1 > 0 ? 1 : 0, polls = 0;     // hits still to come through stage 1
    bool refill1 = true, refill0 = false;
    int slot_page = ref.fill >= 0 ? ref.src : -1;         // where a page that is brought in goes
    if (ref.open_idx >= 0) slot_page = slots_known ? __ldcg(c.page_src + pl + ref.open_idx) : -1;
#pragma unroll 1
    for (;;) {
      // a free stage takes the next page: an HBM page is requested at once, a host page takes a turn on the link
      if (refill1) {
        in1 = next();
        if (in1 >= 0 && ((hosted >> in1) & 1u)) { turn1 = link_turn(c, lane); on_link |= 2u; }
        else if (in1 >= 0) { request(1, in1); issued |= 2u; }
        refill1 = false;
      }
      if (refill0) {                       // (no hits are left by then)
        in0 = next();
        if (in0 >= 0) { turn0 = link_turn(c, lane); on_link |= 1u; }
        refill0 = false;
      }
      const int j = cur ? in1 : in0;
      if (j < 0) break;
      const uint32_t waiting = on_link & ~issued;
      if (waiting) {
        closed = link_closed(c);
        if ((waiting & 1u) && link_open(turn0, closed)) { request(0, in0); issued |= 1u; }
        if ((waiting & 2u) && link_open(turn1, closed)) { request(1, in1); issued |= 2u; }
      }
      // a missed page that has landed behind the hits gives its turn on
      if (hits_in1 > 0 && (on_link & issued & 1u) && page_test(bar0, phases & 1u)) { link_close(c, lane); on_link &= ~1u; }
      if (!((issued >> cur) & 1u)) {
        if (++polls < kLinkPolls) { __nanosleep(100); continue; }
        if (lane == 0) dev_error(c, kErrTimeout);
        dead = true;
        break;
      }
      if (((hosted >> j) & 1u) && !slots_known) {                           // while the page is on its way
        int ok = 1;
        if (lane == 0) ok = flag_wait(c, c.ready + b, slots_ready(bt.epoch));
        slots_known = __shfl_sync(0xffffffffu, ok, 0) != 0;
        if (!slots_known) { dead = true; break; }                           // reported by the wait
        __syncwarp();                                                       // (as above)
        if (ref.open_idx >= 0) slot_page = __ldcg(c.page_src + pl + ref.open_idx);   // negative: bypassed, attended only
      }
      if (!page_landed(bar0 + 8 * cur, (phases >> cur) & 1u)) {
        if (lane == 0) dev_error(c, kErrTimeout);
        dead = true;
        break;
      }
      phases ^= 1u << cur;
      if (row == 0 && p0 == mine) dbg_ta(b, 12);
      if ((on_link >> cur) & 1u) link_close(c, lane);
      on_link &= ~(1u << cur);
      issued &= ~(1u << cur);
      const uint32_t spage = stage0 + cur * kStageBytes;
      attend_page(spage, qb, __shfl_sync(0xffffffffu, ref.mask, j), scale2, acc, lane);
      if ((hosted >> j) & 1u) {
        const int slot = __shfl_sync(0xffffffffu, slot_page, j);
        if (slot >= c.n_gpu_pages) { if (lane == 0) dev_error(c, kErrBounds); }
        else if (slot >= 0) { store_page(spage, c.gpu_pages + (size_t)slot * kPageBytes, lane); stores_read(); }
      }
      __syncwarp();                        // every lane has read the stage
      if (cur) refill1 = true; else refill0 = true;
      if (hits_in1 > 0) { if (--hits_in1 == 0) cur = 0; }
      else cur ^= 1;
    }
  }

  // Every way out of the loops above leads here: the list is done (no copy in flight, no turn open), or
  // a wait has run out, for the list (at most stage 0's early page is in flight), for a turn, for the slots
  // or for a page (one or both stages).  A copy in flight writes to a stage that the outputs are exchanged through
  // below, so it is seen off first.
  if (dead)
    for (int st = 0; st < kWarpStages; ++st) {
      if ((issued >> st) & 1u) page_landed(bar0 + 8 * st, (phases >> st) & 1u, kDrainPolls);
      if ((on_link >> st) & 1u) link_close(c, lane);
    }
  if (row == 0) dbg_ta(b, 13);
  // a head's sum lives in the 8 lanes of its column; the warps meet in their own (now idle) stage 0
  float *comb = reinterpret_cast<float *>(smem);
  constexpr int kWarpComb = kWarpStages * kStageBytes / 4;                  // floats between the warps' areas
  static_assert(G * kCombStride * 4 <= kStageBytes, "a warp's outputs fit its first stage");
#pragma unroll
  for (int h = 0; h < 2; ++h) {
#pragma unroll
    for (int o = 4; o < 32; o <<= 1) acc.l[h] += __shfl_xor_sync(0xffffffffu, acc.l[h], o);
    const int hr = (lane & 3) * 2 + h;
    if (hr < G) {
      float *w = comb + warp * kWarpComb + hr * kCombStride + (lane >> 2);
#pragma unroll
      for (int nt = 0; nt < 8; ++nt) { w[nt * 16] = acc.o[nt][h]; w[nt * 16 + 8] = acc.o[nt][2 + h]; }
      if (lane < 4) { s_m[warp][hr] = acc.m[h]; s_l[warp][hr] = acc.l[h]; }
    }
  }
  __syncthreads();
#pragma unroll 1
  for (int e = threadIdx.x; e < G * (kHeadDim / 4); e += W * 32) {
    const int g = e / (kHeadDim / 4), col = e % (kHeadDim / 4);
    float mn = -INFINITY;
#pragma unroll
    for (int w = 0; w < W; ++w) mn = fmaxf(mn, s_m[w][g]);
    float4 o = make_float4(0.f, 0.f, 0.f, 0.f);
    float l = 0.f;
#pragma unroll
    for (int w = 0; w < W; ++w) {
      const float mw = s_m[w][g], a = mw == -INFINITY ? 0.f : exp2f(mw - mn);
      const float4 x = reinterpret_cast<const float4 *>(comb + w * kWarpComb + g * kCombStride)[col];
      o.x = fmaf(x.x, a, o.x); o.y = fmaf(x.y, a, o.y); o.z = fmaf(x.z, a, o.z); o.w = fmaf(x.w, a, o.w);
      l = fmaf(s_l[w][g], a, l);
    }
    if (n_rows == 1) {                     // the set's only CTA finishes here
      store_out(out_rows + 4 * e, normalised(o, l));
    } else if (kTogether) {
      reinterpret_cast<float4 *>(cluster_outputs(smem))[e] = o;
      if (col == 0) part->ml[g] = make_float2(mn, l);
    } else {
      const size_t at = ((size_t)b * c.max_chunks + row) * G + g;
      reinterpret_cast<float4 *>(c.att_part)[at * (kHeadDim / 4) + col] = o;
      if (col == 0) c.att_ml[at] = make_float2(mn, l);
    }
  }
  if (W < kAttnWarps || n_rows == 1) return 0;
  if (kTogether) return n_rows;
  // the last CTA of the set to get here merges all partials (log-sum-exp)
  __syncthreads();
  if (threadIdx.x == 0) sh_last = last_row(c, b, n_rows);
  __syncthreads();
  if (!sh_last) return 0;
  dbg_ta(b, 14);
  merge_rows<G>(c, b, n_rows, out_rows, comb);
  dbg_ta(b, 15);
  return 0;
}

// The kernel: the CTA's work; one CTA then waits for the kernel before this one.  CTAs that
// go by the per-set flags never wait for the scoring kernel as a whole; with one CTA doing so
// before it exits, this grid cannot complete ahead of that one, and whatever the stream runs
// next (the next step's scoring kernel waits for this grid) comes after all of its writes.
// Three forms, each a kernel of its own, since code for the others costs one that does not need it.  us, in one kernel and
// apart: decode, 8 sets of 65 pages, through memory 24.7 and 24.1, 32 sets 28.2 and 27.6; 104 shapes of plain lists (84 to 148 of 21
// to 44 pages), clusters or through memory, 1 % in all.
enum AttnKernel { kTogether, kByMemory, kByCounts };
template <int G, int W, AttnKernel kKernel, bool kOnce>
__global__ void __launch_bounds__(W * 32, 3 * kAttnWarps / W)
k_attn(DevCtx c, Batch bt, const __nv_bfloat16 *__restrict__ q, __nv_bfloat16 *__restrict__ out) {
  extern __shared__ __align__(128) uint8_t smem[];                // [warps][2] staged pages
  pdl_launch_next();
  if (kKernel != kByCounts) {
    // launch order: row 0 of every set first (the rows that own the first missed pages), or set by set
    const int b = bt.attn_set_major ? blockIdx.y : blockIdx.x, row = bt.attn_set_major ? blockIdx.x : blockIdx.y;
    const int rows = bt.attn_set_major ? gridDim.x : gridDim.y, i_req = b / c.Hkv;
    if (row == 0 || row < attn_rows_of(bt, most_pages(c, bt, i_req), bt.attn_share, rows)) {   // else no list of this set reaches this row
      if (kKernel == kTogether && W == kAttnWarps) {
        __shared__ ClusterPart<G> part;
        const int n = attn_row<G, W, true, kOnce>(c, bt, q, out, smem, b, row, rows, bt.attn_share, -1, &part);
        if (n != 0 && bt.attn_cluster) merge_cluster<G>(part, smem, out + ((size_t)i_req * c.Hq + (b % c.Hkv) * G) * kHeadDim, row, n);
        if (row == 0) dbg_ta(b, 15);
      } else {
        attn_row<G, W, kKernel == kTogether, kOnce>(c, bt, q, out, smem, b, row, rows, bt.attn_share, -1, nullptr);
      }
    }
  } else {
    __shared__ int s_sum[kAttnWarps], s_at[2];
    int b = blockIdx.x % bt.n_req, row = blockIdx.x / bt.n_req;
    pdl_wait_prev();
    int np = count_of(c, b);                                      // (asked for together with the other counts)
    const int share = share_by_counts(c, bt, s_sum), own = bt.n_req * bt.attn_rows;
    bool mine = (int)blockIdx.x < own;
    if (!mine) {
      mine = further_row(c, bt, share, (int)blockIdx.x - own, s_sum, s_at, &b, &row);
      if (mine) np = count_of(c, b);
    }
    if (mine) attn_row<G, W, false, kOnce>(c, bt, q, out, smem, b, row, c.max_chunks, share, np, nullptr);
  }
  if (blockIdx.x == 0 && blockIdx.y == 0) pdl_wait_prev();
}

// Set up and asked for once per device, by the first call that launches there.
template <int G>
const AttnGpu &attn_gpu() {
  static AttnGpu gpus[kMaxDevices] = {};
  static std::once_flag once[kMaxDevices];
  const int slot = current_device_slot();
  std::call_once(once[slot], [slot] {
    for (auto kernel : {k_attn<G, kAttnWarps, kTogether, false>, k_attn<G, kAttnWarps, kByMemory, false>, k_attn<G, kAttnWarps, kByCounts, false>,
                        k_attn<G, 1, kTogether, false>, k_attn<G, kAttnWarps, kTogether, true>, k_attn<G, kAttnWarps, kByMemory, true>,
                        k_attn<G, kAttnWarps, kByCounts, true>, k_attn<G, 1, kTogether, true>}) {
      cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kAttnSmem);
      cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
    }
    AttnGpu &gpu = gpus[slot];
    int dev = 0, sms = 0, per_sm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_attn<G, kAttnWarps, kByMemory, false>, kAttnThreads, kAttnSmem);
    for (int r = 2; r <= kClusterRows; ++r) {
      cudaLaunchAttribute attr[1];
      attr[0].id = cudaLaunchAttributeClusterDimension;
      attr[0].val.clusterDim.x = 1;
      attr[0].val.clusterDim.y = r;
      attr[0].val.clusterDim.z = 1;
      cudaLaunchConfig_t cfg = {};
      cfg.gridDim = dim3(1, r);
      cfg.blockDim = dim3(kAttnThreads);
      cfg.dynamicSmemBytes = kAttnSmem;
      cfg.attrs = attr;
      cfg.numAttrs = 1;
      int n = 0;
      if (cudaOccupancyMaxActiveClusters(&n, k_attn<G, kAttnWarps, kTogether, false>, &cfg) != cudaSuccess) { cudaGetLastError(); n = 0; }
      gpu.clusters[r] = n;
    }
    gpu.resident = sms * per_sm > 0 ? sms * per_sm : 148;
  });
  return gpus[slot];
}

template <int G, bool kOnce>
void launch_plan(const DevCtx &c, const Batch &b, const AttnPlan &p, const __nv_bfloat16 *q, __nv_bfloat16 *out, int n_sets, cudaStream_t st) {
  const dim3 grid = b.attn_set_major ? dim3(p.rows, n_sets) : dim3(n_sets, p.rows);
  if (p.form == kAttnWarp) {
    launch_pdl(k_attn<G, 1, kTogether, kOnce>, grid, dim3(32), (size_t)kAttnSmem / kAttnWarps, st, 1, c, b, q, out);
  } else if (p.form == kAttnCounted) {
    launch_pdl(k_attn<G, kAttnWarps, kByCounts, kOnce>, dim3(p.rows), dim3(kAttnThreads), (size_t)kAttnSmem, st, 1, c, b, q, out);
  } else if (p.rows > 1 && !p.cluster) {
    launch_pdl(k_attn<G, kAttnWarps, kByMemory, kOnce>, grid, dim3(kAttnThreads), (size_t)kAttnSmem, st, 1, c, b, q, out);
  } else {
    launch_pdl(k_attn<G, kAttnWarps, kTogether, kOnce>, grid, dim3(kAttnThreads), (size_t)kAttnSmem, st,
               p.cluster ? b.attn_set_major ? dim3(p.rows, 1) : dim3(1, p.rows) : dim3(1), c, b, q, out);
  }
}

template <int G>
void launch_attn_g(const DevCtx &c, Batch b, const __nv_bfloat16 *q, __nv_bfloat16 *out, int n_sets, int max_pages, long long est_pages, cudaStream_t st) {
  const AttnPlan p = attn_plan(attn_gpu<G>(), c.ready != nullptr, b.attn_set_major != 0, n_sets, max_pages, est_pages, c.max_chunks);
  b.attn_rows = p.own;
  b.attn_least = p.least;
  b.attn_share = p.share;
  b.attn_cluster = p.cluster;
  if (b.read_once & kOncePages) launch_plan<G, true>(c, b, p, q, out, n_sets, st);
  else launch_plan<G, false>(c, b, p, q, out, n_sets, st);
}

}  // namespace

int launch_attention(const DevCtx &c, const Batch &b, const __nv_bfloat16 *q,
                     __nv_bfloat16 *out, int max_pages_hint, long long est_pages, cudaStream_t st, Prof *prof) {
  const int n_sets = b.n_req * c.Hkv;
  switch (c.G) {
    case 1: launch_attn_g<1>(c, b, q, out, n_sets, max_pages_hint, est_pages, st); break;
    case 2: launch_attn_g<2>(c, b, q, out, n_sets, max_pages_hint, est_pages, st); break;
    case 4: launch_attn_g<4>(c, b, q, out, n_sets, max_pages_hint, est_pages, st); break;
    default: launch_attn_g<8>(c, b, q, out, n_sets, max_pages_hint, est_pages, st); break;
  }
  prof_mark(prof, st, kProfAttnSplit);
  return 1;
}

}  // namespace spin

// ---------------------------------------------------------------------------------------
// Allocation-free paged attention (see spin_paged_attention_static in spin.h).
//
// The split-K partials and arrival counters of this variant live in a fixed array that is part of the library
// image, so a caller that must not (or cannot) allocate device memory -- code running inside
// someone else's memory budget, a latency-critical loop that may not touch the allocator, a
// plug-in that is only handed its input and output buffers -- can still run the split + merge
// pair.  Every GPU that loads the library carries these 8 MiB until the process exits.
namespace spin {
namespace {
constexpr size_t kStaticPartialFloats = (size_t)2 << 20;                  // 8 MiB of fp32
__device__ __align__(256) static float g_static_partials[kStaticPartialFloats];
// Arrival words, one per set: the size limit admits fewer sets than this (130 floats and a counter each).
constexpr int kStaticSets = (int)(kStaticPartialFloats / (kHeadDim + 2 + 1)) + 1;
__device__ static unsigned long long g_static_words[kStaticSets];         // zero between calls (see last_row)
std::atomic<float *> g_static_partials_addr[kMaxDevices] = {};            // per device, set up by the first call that finds one missing
std::atomic<unsigned long long *> g_static_words_addr[kMaxDevices] = {};
std::atomic<uint32_t> g_static_calls{0};
}  // namespace
}  // namespace spin

extern "C" int spin_paged_attention_static(const void *q, const void *page_pool,
                                           const int32_t *page_ids, const uint32_t *page_masks,
                                           const int32_t *n_pages, int32_t n_sets,
                                           int32_t list_stride, int32_t group, float sm_scale,
                                           void *out, void *cuda_stream) {
  using namespace spin;
  if (!q || !page_pool || !page_ids || !page_masks || !n_pages || !out || n_sets < 1 || list_stride < 1) {
    fprintf(stderr, "spin_paged_attention_static: null pointer or non-positive size\n");
    return SPIN_ERR_INVALID;
  }
  if (group != 1 && group != 2 && group != 4 && group != 8) {
    fprintf(stderr, "spin_paged_attention_static: group must be 1, 2, 4 or 8 (got %d)\n", group);
    return SPIN_ERR_INVALID;
  }
  const int chunks = (list_stride + kChunkPages - 1) / kChunkPages;
  // room in the built-in array for one partial per 8 pages of every list (and, as ever, a word per
  // set): more than the call uses, since a CTA writes one partial for all its pages
  const size_t counter_floats = ((size_t)n_sets + 63) / 64 * 64;
  const size_t need = counter_floats + (size_t)n_sets * chunks * group * (kHeadDim + 2);
  if (need > kStaticPartialFloats) {
    fprintf(stderr,
            "spin_paged_attention_static: n_sets (%d) x ceil(list_stride/8) (%d) x group (%d) x 130 partial "
            "floats + %zu counters = %zu exceed the built-in %zu; use fewer sets per call or the context API\n",
            n_sets, chunks, group, counter_floats, need, kStaticPartialFloats);
    return SPIN_ERR_INVALID;
  }
  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) {
    fprintf(stderr, "spin_paged_attention_static: no usable current CUDA device\n");
    return SPIN_ERR_CUDA;
  }
  float *p = g_static_partials_addr[dev].load(std::memory_order_relaxed);
  unsigned long long *w = g_static_words_addr[dev].load(std::memory_order_relaxed);
  if (!p || !w) {
    // In host code the arrays' names are only stand-ins for the symbols: the addresses the
    // kernels can use have to be asked for, once per device, with that device current (several
    // threads that do so at once get the same ones).
    cudaError_t e = cudaGetSymbolAddress(reinterpret_cast<void **>(&p), g_static_partials);
    if (e == cudaSuccess) e = cudaGetSymbolAddress(reinterpret_cast<void **>(&w), g_static_words);
    if (e != cudaSuccess || !p || !w) {
      fprintf(stderr, "spin_paged_attention_static: cudaGetSymbolAddress failed: %s\n", cudaGetErrorString(e));
      return SPIN_ERR_CUDA;
    }
    g_static_words_addr[dev].store(w, std::memory_order_relaxed);
    g_static_partials_addr[dev].store(p, std::memory_order_relaxed);
  }
  DevCtx c{};
  c.num_layers = 1; c.Hq = group; c.Hkv = 1; c.G = group;
  c.max_pages = list_stride; c.tail_cap = 0; c.max_chunks = chunks;
  c.sm_scale = sm_scale != 0.f ? sm_scale : 0.08838834764831845f;
  c.gpu_pages = const_cast<uint8_t *>(reinterpret_cast<const uint8_t *>(page_pool));
  c.host_pages = nullptr;
  c.n_gpu_pages = 0x7fffffff;                               // the caller vouches for the ids
  c.n_host_pages = 0;
  c.page_src = const_cast<int32_t *>(page_ids);
  c.page_mask = const_cast<uint32_t *>(page_masks);
  c.n_pages = const_cast<int32_t *>(n_pages);
  c.page_fill = nullptr;                                    // every listed page is already in the pool
  c.page_desc = nullptr;                                    // the lists are attended in the order given
  c.ready = nullptr;                                        // plain stream order: no per-set flags
  c.tail_ready = nullptr;
  c.ready1 = nullptr;
  c.att_part = p;
  c.att_ml = reinterpret_cast<float2 *>(c.att_part + (size_t)n_sets * chunks * group * kHeadDim);
  c.att_words = w;
  c.att_call = g_static_calls.fetch_add(1u, std::memory_order_relaxed) + 1u;
  cudaStream_t st = reinterpret_cast<cudaStream_t>(cuda_stream);
  Batch b{};
  b.n_req = n_sets;
  b.read_once = lists_read_once((double)n_sets * list_stride * kPageBytes);
  launch_attention(c, b, reinterpret_cast<const __nv_bfloat16 *>(q), reinterpret_cast<__nv_bfloat16 *>(out),
                   list_stride, 0, st, nullptr);
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) {
    fprintf(stderr, "spin_paged_attention_static: launch failed: %s\n", cudaGetErrorString(e));
    return SPIN_ERR_CUDA;
  }
  return SPIN_OK;
}

#ifdef SPIN_TIMING
extern "C" __attribute__((visibility("default"))) int spin_debug_timestamps_attn(unsigned long long *out) {
  cudaDeviceSynchronize();
  return (int)cudaMemcpyFromSymbol(out, spin::g_dbg_ta, sizeof(unsigned long long) * 256 * 16);
}
#endif
