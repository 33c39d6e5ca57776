// Decode-time / edge append of one set, shared by the stand-alone append kernel and by the
// scoring kernel's in-grid append CTAs (Index + Offload, Section 4.1).
#pragma once
#include "spin_dev.cuh"

namespace spin {

// The append body is run by 256 threads that may be part of a larger CTA (the streaming scoring
// kernel has a producer warp besides them): they meet at a named barrier of their own.
__device__ __forceinline__ void sync_256() { asm volatile("bar.sync 1, 256;\n" ::: "memory"); }

// 256 threads; thread t moves the 16-byte piece (t & 15) of row (t >> 4).
__device__ __forceinline__ uint4 ld16(const void *p) { return *reinterpret_cast<const uint4 *>(p); }
__device__ __forceinline__ void st16(void *p, uint4 v) { *reinterpret_cast<uint4 *>(p) = v; }

// Where the index entries of a partition go.  Looked up before the rows are there: the directory
// reads are in flight together with everything else an append reads.
struct IndexPlace { uint8_t *summary; MetaEntry *meta; };
__device__ __forceinline__ IndexPlace index_place(const DevCtx &c, int set, int part) {
  return IndexPlace{summary_at(c, set, c.kind == kKindToken ? part * kPageTokens : part), meta_at(c, set, part)};
}

// min / max over the 16 key rows held in shared memory, per channel; bf16 compares are done
// in fp32 (exact).  Thread c < 128 handles channel c.
__device__ __forceinline__ void write_minmax(uint8_t *s, const __nv_bfloat16 (*krows)[kHeadDim], int tid) {
  if (tid < kHeadDim) {
    float mn = __bfloat162float(krows[0][tid]), mx = mn;
#pragma unroll
    for (int r = 1; r < kPageTokens; ++r) {
      float x = __bfloat162float(krows[r][tid]);
      mn = fminf(mn, x);
      mx = fmaxf(mx, x);
    }
    __nv_bfloat16 *o = reinterpret_cast<__nv_bfloat16 *>(s);
    o[tid] = __float2bfloat16(mn);            // exact: mn is one of the bf16 inputs
    o[kHeadDim + tid] = __float2bfloat16(mx);
  }
}

// Landmark summary (Table 1, ShadowKV's Index: mean(paged_key, dim=dim_page)): per channel the
// 16 keys are added in token order in fp32, scaled by 1/16 (exact) and rounded to bf16
// (nearest even) -- the order and rounding the CPU oracle uses.
__device__ __forceinline__ void write_mean(uint8_t *dst, const __nv_bfloat16 (*krows)[kHeadDim], int tid) {
  if (tid < kHeadDim) {
    float s = __bfloat162float(krows[0][tid]);
#pragma unroll
    for (int r = 1; r < kPageTokens; ++r) s = s + __bfloat162float(krows[r][tid]);
    reinterpret_cast<__nv_bfloat16 *>(dst)[tid] = __float2bfloat16_rn(s * 0.0625f);
  }
}

__device__ __forceinline__ void write_token_summaries(uint8_t *s, const __nv_bfloat16 (*krows)[kHeadDim], int tid) {
  int r = tid >> 4, piece = tid & 15;
  st16(s + r * kRowBytes + piece * 16, ld16(reinterpret_cast<const uint8_t *>(krows[r]) + piece * 16));
}

__device__ __forceinline__ void index_page(const DevCtx &c, int set, int part, const IndexPlace &at,
                                           const __nv_bfloat16 (*krows)[kHeadDim], int tid) {
  if (!at.summary) { dev_error(c, 1u); }
  else if (c.kind == kKindPage) write_minmax(at.summary, krows, tid);
  else if (c.kind == kKindPageMean) write_mean(at.summary, krows, tid);
  else write_token_summaries(at.summary, krows, tid);
  if (tid == 0) {
    if (at.meta) { at.meta->tokens = kPageTokens; at.meta->resident = 0; } else dev_error(c, 1u);
    off_mirror_set(c, set, part, part);          // page-sized kinds: partition p starts at page p
  }
}

// The pages at the edges of an append for one set, run by a 256-thread CTA: (1) the old tail
// page, if this call completes it and moves on, is indexed from its HBM copy plus the new rows;
// (2) the newest page receives its new rows in the host tier and in the HBM tail page.  Also
// the only form needed for single-token decode appends.  k, v: [n_req][n_new][Hkv][d]; `i` is
// the request's position in that array.  krows: 16 x 128 bf16 of shared memory.
__device__ __forceinline__ void append_edge_body(const DevCtx &c, int set, int i, int head,
                                                 const __nv_bfloat16 *__restrict__ k,
                                                 const __nv_bfloat16 *__restrict__ v, int n_new,
                                                 int n0_host, int epoch, __nv_bfloat16 (*krows)[kHeadDim]) {
  const int tid = threadIdx.x;
  const int r = tid >> 4, piece = tid & 15;
  SetState st = c.state[set];
  // the host has counted every append; its count is the one used, and a device word that
  // disagrees is reported (it is rewritten below)
  if (threadIdx.x == 0 && st.n_tokens != n0_host) {
    dev_error(c, kErrState);
    if (atomicCAS(&c.counters->dbg[0], 0u, (unsigned)set + 1u) == 0u) {
      c.counters->dbg[1] = (unsigned)st.n_tokens; c.counters->dbg[2] = (unsigned)n0_host; c.counters->dbg[3] = (unsigned)epoch;
    }
  }
  const int n0 = n0_host, n1 = n0 + n_new;
  const uint8_t *kin = reinterpret_cast<const uint8_t *>(k) + (size_t)i * n_new * c.Hkv * kRowBytes;
  const uint8_t *vin = reinterpret_cast<const uint8_t *>(v) + (size_t)i * n_new * c.Hkv * kRowBytes;
  auto in_off = [&](int tok) { return ((size_t)(tok - n0) * c.Hkv + head) * kRowBytes + piece * 16; };

  if (c.kind == kKindCluster) {
    sync_256();          // every thread has read the state before thread 0 rewrites it at the end (the other kinds' threads go by the host's counts)
    // decode tokens of a clustered set only extend the always-attended tail
    int tail_pages = st.tail_pages, tail_len = st.tail_len;
    for (int tok = n0; tok < n1; ++tok) {
      if (tail_pages == 0 || tail_len == kPageTokens) { ++tail_pages; tail_len = 0; }
      if (tail_pages > c.tail_cap) { if (tid == 0) dev_error(c, 1u); break; }
      if (tid < 16) {
        const int32_t *hp = cpt_at(c, set, st.tail_first + tail_pages - 1);
        if (!hp) { dev_error(c, 1u); }
        else {
          uint4 kk = ld16(kin + in_off(tok)), vv = ld16(vin + in_off(tok));
          size_t o = (size_t)tail_len * kRowBytes + piece * 16;
          uint8_t *h = c.host_pages + (size_t)(*hp) * kPageBytes + o;
          uint8_t *g = c.gpu_pages + (size_t)c.tail_phys[(size_t)set * c.tail_cap + tail_pages - 1] * kPageBytes + o;
          st16(h, kk); st16(h + kHalfPageBytes, vv);
          st16(g, kk); st16(g + kHalfPageBytes, vv);
        }
      }
      ++tail_len;
    }
    if (tid == 0) {
      SetState *s = &c.state[set];
      s->n_tokens = n1;
      s->tail_pages = tail_pages;
      s->tail_len = tail_len;
      s->n_host_pages = st.tail_first + tail_pages;
    }
    return;
  }

  const int j0 = n0 > 0 ? (n0 - 1) / kPageTokens : -1;      // old tail page
  const int j_end = (n1 - 1) / kPageTokens;                 // newest page after the call
  // Everything the body reads is asked for here, before any of it is used: the table entries of the
  // pages involved (the newest page's host id comes over the host link), the rows that are already
  // in the HBM tail page and the new ones, the places of the index entries.  (Read where they are
  // used, those trips follow one another: the launch took 7 us of the step instead of 4.)
  uint8_t *tail = c.gpu_pages + (size_t)c.tail_phys[(size_t)set * c.tail_cap] * kPageBytes;
  const int lo = max(n0, j_end * kPageTokens) - j_end * kPageTokens, hi = n1 - j_end * kPageTokens;   // the newest page's new rows: [lo, hi)
  const bool mine = r >= lo && r < hi, closes = j0 >= 0 && j0 < j_end;
  const int32_t *hp = mine ? cpt_at(c, set, j_end) : nullptr;
  const int have = n0 - j0 * kPageTokens;                   // rows of the old tail page already in its HBM copy
  const bool late = closes && r >= have;                    // ... and those that this call adds to it
  const int32_t *hp0 = late ? cpt_at(c, set, j0) : nullptr;
  const IndexPlace at = closes ? index_place(c, set, j0) : IndexPlace{nullptr, nullptr};
  const uint4 zero = make_uint4(0, 0, 0, 0);
  const size_t o = mine ? in_off(j_end * kPageTokens + r) : 0, o0 = late ? in_off(j0 * kPageTokens + r) : 0;
  const uint4 kk = mine ? ld16(kin + o) : zero, vv = mine ? ld16(vin + o) : zero;
  const uint4 kk0 = !closes ? zero : late ? ld16(kin + o0) : ld16(tail + r * kRowBytes + piece * 16), vv0 = late ? ld16(vin + o0) : zero;
  const int32_t host_page = hp ? *hp : -1, host_page0 = hp0 ? *hp0 : -1;
  if (closes) {
    // the old tail page is complete after this call (or was already) and stops being the tail
    if (late) {
      if (hp0) {
        uint8_t *dst = c.host_pages + (size_t)host_page0 * kPageBytes + r * kRowBytes + piece * 16;
        st16(dst, kk0);
        st16(dst + kHalfPageBytes, vv0);
      } else if (piece == 0) dev_error(c, 1u);
    }
    st16(reinterpret_cast<uint8_t *>(krows[r]) + piece * 16, kk0);
    sync_256();                                             // (tail rows have been read before they are rewritten below)
    index_page(c, set, j0, at, krows, tid);
  }
  if (mine) {
    if (hp) {
      uint8_t *dst = c.host_pages + (size_t)host_page * kPageBytes + r * kRowBytes + piece * 16;
      st16(dst, kk);
      st16(dst + kHalfPageBytes, vv);
      if (piece == 0 && r == lo) cpt_mirror_set(c, set, j_end, host_page);
    } else if (piece == 0) dev_error(c, 1u);
    st16(tail + r * kRowBytes + piece * 16, kk);
    st16(tail + kHalfPageBytes + r * kRowBytes + piece * 16, vv);
  }
  if (tid == 0) {
    SetState *s = &c.state[set];
    s->n_tokens = n1;
    s->n_partitions = j_end;
    s->n_host_pages = j_end + 1;
    s->tail_first = j_end;
    s->tail_pages = 1;
    s->tail_len = n1 - j_end * kPageTokens;
  }
}

}  // namespace spin
