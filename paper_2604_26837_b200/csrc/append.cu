// Index + Offload (Section 4.1): write appended K/V rows through to the pinned host tier,
// keep the newest page in an HBM tail page, and turn a completed page into a candidate
// partition with its summary (per-channel min/max of the keys, or the key rows themselves
// for token-granular selection).  The host runtime has already mapped the segments and
// filled the host-side tables (Partition Offset, CPU page table) for the pages touched here.
#define SPIN_FILE_ID 1
#include "append_body.cuh"

namespace spin {

namespace {

// The HBM copies of the CPU page table entries of pages [first_page, first_page + n), from the pinned originals, in
// front of the kernel below: its own small reads of those would cross the link against its writes, and wait
// behind them.  32768 tokens of 8 heads: 3001 -> 2864 us with the first step; calls of 512 tokens 622 -> 603 for
// 4100.  Short calls would pay more for the launch than it gives (128 tokens of 8 heads, 56 pages: 924 -> 1000;
// 256 tokens, 120 pages: no difference), so it is for kMirrorPages of all heads together: 65536 rows in calls of 192 and of 256
// pages of all heads, with it and without, one head 1339, 1324 and 934, 1138; two 1317, 1314 and 967, 1213; four 1385,
// 1380 and 955, 1165; eight 1289, 1288 and 921, 1178.
constexpr int kMirrorPages = 192;
__global__ void __launch_bounds__(256)
k_mirror_pages(DevCtx c, int req, int layer, int first_page, int n) {
  const int e = blockIdx.x * 256 + threadIdx.x, set = set_index(c, req, layer, blockIdx.y);
  if (e >= n) return;
  const int32_t *hp = cpt_at(c, set, first_page + e);
  if (hp) cpt_mirror_set(c, set, first_page + e, *hp); else dev_error(c, kErrBounds);
}

// Pages completely covered by this call's tokens that are not the newest page: all 16 rows
// come from the input; the page is written to the host tier and indexed.
__global__ void __launch_bounds__(256)
k_append_bulk(DevCtx c, int req, int layer, const __nv_bfloat16 *__restrict__ k,
              const __nv_bfloat16 *__restrict__ v, int first_page, int first_token_of_call,
              uint8_t *__restrict__ stage, const int32_t *__restrict__ stage_hp, int mirrored) {
  __shared__ __align__(16) __nv_bfloat16 krows[kPageTokens][kHeadDim];
  const int head = blockIdx.y, page = first_page + blockIdx.x, tid = threadIdx.x;
  const int set = set_index(c, req, layer, head);
  const int r = tid >> 4, piece = tid & 15;
  const size_t tok = (size_t)page * kPageTokens + r - first_token_of_call;
  const size_t in_off = (tok * c.Hkv + head) * kHeadDim * 2 + piece * 16;
  uint4 kk = ld16(reinterpret_cast<const uint8_t *>(k) + in_off);
  uint4 vv = ld16(reinterpret_cast<const uint8_t *>(v) + in_off);
  const IndexPlace at = index_place(c, set, page);
  const size_t unit = (size_t)head * gridDim.x + blockIdx.x;        // head-major, as host pages are handed out
  const bool ahead = !stage && mirrored;
  int32_t host_page;
  if (stage) {
    host_page = stage_hp[unit];
  } else {
    const int32_t *hp = ahead ? cpt_lookup(c, set, page) : cpt_at(c, set, page);
    if (!hp) { if (tid == 0) dev_error(c, 1u); return; }
    host_page = *hp;
  }
  if (!ahead && tid == 0) cpt_mirror_set(c, set, page, host_page);
  // Offload: straight to the page's place in pinned host memory, or -- asynchronous offload --
  // into an HBM staging slot from which copy-engine transfers move it on the library's own stream
  uint8_t *dst = c.host_pages + (size_t)host_page * kPageBytes + r * kRowBytes + piece * 16;
  if (stage) dst = stage + unit * kPageBytes + r * kRowBytes + piece * 16;
  st16(dst, kk);
  st16(dst + kHalfPageBytes, vv);
  st16(reinterpret_cast<uint8_t *>(krows[r]) + piece * 16, kk);
  __syncthreads();
  index_page(c, set, page, at, krows, tid);
}

// Stand-alone edge append: one CTA per (kv head, request).  The rows of CTAs beyond the requests
// bring in the step's queries where they live in pinned host memory (nq pieces of 16 bytes), beside
// the append instead of in a launch in front of it; the new K/V rows are read where they are.
__global__ void __launch_bounds__(256)
k_append_edge(DevCtx c, AppendEdgeArgs a, const __nv_bfloat16 *__restrict__ k,
              const __nv_bfloat16 *__restrict__ v, int n_new, uint4 *dq, const uint4 *sq, int nq) {
  __shared__ __align__(16) __nv_bfloat16 krows[kPageTokens][kHeadDim];
  const int head = blockIdx.x, i = blockIdx.y;
  pdl_launch_next();
  pdl_wait_prev();
  if (i >= a.n_req) {
    const int first = ((i - a.n_req) * (int)gridDim.x + head) * 256 + threadIdx.x, step = ((int)gridDim.y - a.n_req) * (int)gridDim.x * 256;
    for (int e = first; e < nq; e += step) dq[e] = sq[e];
    return;
  }
  append_edge_body(c, set_index(c, a.req[i], a.layer, head), i, head, k, v, n_new, a.n_tokens[i], -1, krows);
}

// ---- cluster prefill ------------------------------------------------------------------------
// token_partition [n_tokens][Hkv] from entry `first` on -> tokens per (head, cluster), for the clusters
// [c0, c0 + nc); bad = the first entry that names no cluster (all ones if none does).
__global__ void __launch_bounds__(256)
k_cluster_count(const int32_t *__restrict__ tp, size_t first, size_t rows, int H, int C, int c0, int nc, int32_t *__restrict__ count,
                unsigned long long *bad) {
  for (size_t i = (size_t)blockIdx.x * 256 + threadIdx.x; i < rows; i += (size_t)gridDim.x * 256) {
    const int32_t cl = tp[i];
    if (cl < 0 || cl >= C) atomicMin(bad, (unsigned long long)(first + i));
    else if (cl >= c0 && cl < c0 + nc) atomicAdd(count + (size_t)(i % H) * nc + (cl - c0), 1);
  }
}

// A row's place in its set's logical page order: (first page of its cluster) * 16 + its rank among
// the cluster's tokens (arrival order).  One CTA per kv head, a warp per run of consecutive tokens
// with counters of its own in shared memory, which hold the cluster's next place: count, prefix over the
// warps, then 32 tokens at a time, the lanes of a cluster ranked by match_any.  Where even one warp's
// counters exceed shared memory a single warp counts in the clusters' residency words (zero until the
// prefill is done); these also carry the counts from one chunk of tokens to the next.  tp and place may be
// the same array: an entry is read by the thread that overwrites it, after every count has been taken.
// Latency-bound (a warp's steps follow one another): ~30 us for 32768 tokens and 512 clusters,
// beside 2.6 ms for their rows on the host link.
constexpr int kPlaceWarps = 16, kPlaceSmem = 160 * 1024;
__global__ void __launch_bounds__(kPlaceWarps * 32)
k_cluster_place(DevCtx c, int req, int layer, const int32_t *tp, int64_t n, int C, int n_warps, int in_smem, int first_chunk, int last_chunk,
                int32_t *place) {
  extern __shared__ int32_t s_run[];
  const int head = blockIdx.x, H = c.Hkv, set = set_index(c, req, layer, head), warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  int32_t *cnt = s_run + (size_t)warp * C;
  const int64_t per = (n + n_warps - 1) / n_warps, lo = warp < n_warps ? min(n, warp * per) : n, hi = warp < n_warps ? min(n, lo + per) : n;
  const int32_t *mine = tp + head;
  // the cluster's next place before this chunk (every entry is mapped: the tables have been laid out)
  auto next_of = [&](int cl) {
    const MetaEntry *m = first_chunk ? nullptr : meta_at(c, set, cl);
    const int32_t *o = first_chunk ? off_lookup(c, set, cl) : nullptr;
    return m ? m->resident : o ? *o * kPageTokens : 0;
  };
  auto keep = [&](int cl, int32_t next) { MetaEntry *m = meta_at(c, set, cl); if (m) m->resident = next; else dev_error(c, kErrBounds); };
  if (in_smem) {
    for (int i = threadIdx.x; i < n_warps * C; i += blockDim.x) s_run[i] = 0;
    __syncthreads();
#pragma unroll 4
    for (int64_t t = lo + lane; t < hi; t += 32) atomicAdd(cnt + mine[(size_t)t * H], 1);
    __syncthreads();
    for (int cl = threadIdx.x; cl < C; cl += blockDim.x) {
      int32_t sum = next_of(cl);
      for (int w = 0; w < n_warps; ++w) { const int32_t x = s_run[(size_t)w * C + cl]; s_run[(size_t)w * C + cl] = sum; sum += x; }
      if (!first_chunk || !last_chunk) keep(cl, last_chunk ? 0 : sum);
    }
    __syncthreads();
  } else {
    if (first_chunk)
      for (int cl = threadIdx.x; cl < C; cl += blockDim.x) keep(cl, next_of(cl));
    __syncthreads();
  }
  int64_t t = lo + lane;
  int cl = t < hi ? mine[(size_t)t * H] : -1;
#pragma unroll 1
  for (int64_t t0 = lo; t0 < hi; t0 += 32) {
    const int64_t t_next = t + 32;
    const int cl_next = t_next < hi ? mine[(size_t)t_next * H] : -1;       // in flight while these 32 are ranked
    const uint32_t same = __match_any_sync(0xffffffffu, cl);
    MetaEntry *m = in_smem || cl < 0 ? nullptr : meta_at(c, set, cl);
    const int32_t next = cl < 0 ? 0 : in_smem ? cnt[cl] : m ? m->resident : 0;
    __syncwarp();
    if (cl >= 0) {
      place[(size_t)t * H + head] = next + __popc(same & ((1u << lane) - 1u));
      if ((same >> lane) == 1u) {                                          // the cluster's last lane
        if (in_smem) cnt[cl] = next + __popc(same); else if (m) m->resident = next + __popc(same);
      }
    }
    __syncwarp();
    t = t_next;
    cl = cl_next;
  }
  if (!in_smem && last_chunk) {
    __syncthreads();
    for (int cl = threadIdx.x; cl < C; cl += blockDim.x) keep(cl, 0);
  }
}

// What follows from the layout, for every kv head's set: Meta-partition entries of the clusters
// [c0, c0 + nc), whose counts these are, and with the first of them the HBM copies of the Partition
// Offset and CPU page tables (read from the pinned originals) and the set's scalars.
__global__ void __launch_bounds__(256)
k_cluster_tables(DevCtx c, int req, int layer, int C, int c0, int nc, int n_pages, int n_tokens, const int32_t *__restrict__ count, int slots) {
  const int head = blockIdx.y, set = set_index(c, req, layer, head), e = blockIdx.x * 256 + threadIdx.x;
  if (e < nc) {
    MetaEntry *m = meta_at(c, set, c0 + e);
    if (m) *m = MetaEntry{count[(size_t)head * nc + e], 0}; else dev_error(c, kErrBounds);
  }
  if (c0 > 0) return;
  mirror_tables(c, set, e, C, n_pages);
  if (e == 0) {
    SetState *s = c.state + set;
    s->n_tokens = n_tokens;
    s->n_partitions = C;
    s->n_host_pages = n_pages;
    s->tail_first = n_pages;
    s->tail_pages = 0;
    s->tail_len = 0;
    s->slots = slots;
  }
}

// Row (token, head) -> its place in the host tier.
__global__ void __launch_bounds__(256)
k_cluster_scatter(DevCtx c, int req, int layer, const __nv_bfloat16 *__restrict__ k, const __nv_bfloat16 *__restrict__ v,
                  const int32_t *__restrict__ place, size_t rows) {
  const int piece = threadIdx.x & 15;
  for (size_t row = (size_t)blockIdx.x * 16 + (threadIdx.x >> 4); row < rows; row += (size_t)gridDim.x * 16) {
    const int32_t d = place[row];
    const int32_t *hp = cpt_lookup(c, set_index(c, req, layer, (int)(row % c.Hkv)), d >> 4);
    const int32_t host_page = hp ? *hp : -1;
    if (host_page < 0 || host_page >= c.n_host_pages) { if (piece == 0) dev_error(c, kErrBounds); continue; }
    uint8_t *dst = c.host_pages + (size_t)host_page * kPageBytes + (size_t)(d & 15) * kRowBytes + piece * 16;
    st16(dst, ld16(reinterpret_cast<const uint8_t *>(k) + row * kRowBytes + piece * 16));
    st16(dst + kHalfPageBytes, ld16(reinterpret_cast<const uint8_t *>(v) + row * kRowBytes + piece * 16));
  }
}

// The same through a staging slot in HBM (asynchronous offload): the rows whose page
// lies in [p0, p0 + m) go to the slot, laid out head-major ([head][page - p0], the order in
// which copy-engine transfers then move the pages to host memory), the others are left for
// another pass.
__global__ void __launch_bounds__(256)
k_cluster_scatter_staged(DevCtx c, const __nv_bfloat16 *__restrict__ k, const __nv_bfloat16 *__restrict__ v,
                         const int32_t *__restrict__ place, int n_tokens, int p0, int m, uint8_t *__restrict__ stage) {
  const int piece = threadIdx.x & 15;
  const size_t rows = (size_t)n_tokens * c.Hkv;
  for (size_t row = (size_t)blockIdx.x * 16 + (threadIdx.x >> 4); row < rows; row += (size_t)gridDim.x * 16) {
    const int32_t d = place[row];
    const int lp = d >> 4;
    if (lp < p0 || lp >= p0 + m) continue;
    const int head = (int)(row % c.Hkv);
    uint8_t *dst = stage + ((size_t)head * m + (lp - p0)) * kPageBytes + (size_t)(d & 15) * kRowBytes + piece * 16;
    st16(dst, ld16(reinterpret_cast<const uint8_t *>(k) + row * kRowBytes + piece * 16));
    st16(dst + kHalfPageBytes, ld16(reinterpret_cast<const uint8_t *>(v) + row * kRowBytes + piece * 16));
  }
}

// Centroids [C][Hkv][d] -> the summary rows of each head's set.
__global__ void __launch_bounds__(256)
k_copy_centroids(DevCtx c, int req, int layer, const __nv_bfloat16 *__restrict__ cen, int n_clusters) {
  const int piece = threadIdx.x & 15;
  const size_t rows = (size_t)n_clusters * c.Hkv;
  for (size_t row = (size_t)blockIdx.x * 16 + (threadIdx.x >> 4); row < rows; row += (size_t)gridDim.x * 16) {
    const int cl = (int)(row / c.Hkv), head = (int)(row % c.Hkv);
    uint8_t *s = summary_at(c, set_index(c, req, layer, head), cl);
    if (!s) { if (piece == 0) dev_error(c, 1u); continue; }
    st16(s + piece * 16, ld16(reinterpret_cast<const uint8_t *>(cen) + row * kRowBytes + piece * 16));
  }
}

// Directory entries, carried in the kernel's parameters.
constexpr int kDirBatch = 336;                       // 4 KB of parameters
struct DirBatch { int64_t at[kDirBatch]; int32_t value[kDirBatch]; int32_t n; };
__global__ void __launch_bounds__(256)
k_dir_update(int32_t *__restrict__ dirs, const __grid_constant__ DirBatch a) {
  for (int i = threadIdx.x; i < a.n; i += 256) dirs[a.at[i]] = a.value[i];
}

// A step's queries that live in pinned host memory are brought into the staging buffer by a small
// kernel of zero-copy reads instead of a copy-engine transfer.
__global__ void __launch_bounds__(256)
k_stage_in(uint4 *dq, const uint4 *sq, int nq) {
  pdl_launch_next();
  pdl_wait_prev();
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < nq; i += gridDim.x * blockDim.x) dq[i] = sq[i];
}

}  // namespace

int launch_stage_in(void *dq, const void *sq, size_t q_bytes, cudaStream_t st) {
  const int nq = (int)(q_bytes / 16);
  const int grid = (nq + 255) / 256 < 64 ? (nq + 255) / 256 : 64;
  launch_pdl(k_stage_in, dim3(grid), dim3(256), 0, st, 1, reinterpret_cast<uint4 *>(dq), reinterpret_cast<const uint4 *>(sq), nq);
  return 1;
}

int launch_dir_update(const DevCtx &c, const DirUpdate *u, int n, cudaStream_t st) {
  int launched = 0;
  for (int i = 0; i < n; i += kDirBatch, ++launched) {
    DirBatch a;
    a.n = n - i < kDirBatch ? n - i : kDirBatch;
    for (int j = 0; j < a.n; ++j) { a.at[j] = u[i + j].at; a.value[j] = u[i + j].value; }
    k_dir_update<<<1, 256, 0, st>>>(c.dir_meta, a);
  }
  return launched;
}

int launch_append_bulk(const DevCtx &c, int req, int layer, const __nv_bfloat16 *k,
                       const __nv_bfloat16 *v, int first_page, int n_pages, int first_token_of_call,
                       cudaStream_t st, Prof *prof, uint8_t *stage, const int32_t *stage_hp) {
  if (n_pages <= 0) return 0;
  const bool mirrored = !stage && c.cpt_mirror && n_pages * c.Hkv >= kMirrorPages;
  if (mirrored) k_mirror_pages<<<dim3((n_pages + 255) / 256, c.Hkv), 256, 0, st>>>(c, req, layer, first_page, n_pages);
  k_append_bulk<<<dim3(n_pages, c.Hkv), 256, 0, st>>>(c, req, layer, k, v, first_page, first_token_of_call, stage, stage_hp, mirrored);
  prof_mark(prof, st, kProfAppend);
  return mirrored ? 2 : 1;
}

int launch_append_edge(const DevCtx &c, const AppendEdgeArgs &a, const __nv_bfloat16 *k,
                       const __nv_bfloat16 *v, int n_new, cudaStream_t st, Prof *prof, void *dq, const void *sq, size_t q_bytes) {
  const int nq = sq ? (int)(q_bytes / 16) : 0;
  int q_ctas = (nq + 255) / 256 < 64 ? (nq + 255) / 256 : 64;
  launch_pdl(k_append_edge, dim3(c.Hkv, a.n_req + (q_ctas + c.Hkv - 1) / c.Hkv), dim3(256), 0, st, 1, c, a, k, v, n_new,
             reinterpret_cast<uint4 *>(dq), reinterpret_cast<const uint4 *>(sq), nq);
  prof_mark(prof, st, kProfAppend);
  return 1;
}

int launch_cluster_count(const int32_t *tp, size_t first, size_t rows, int H, int C, int c0, int nc, int32_t *count, unsigned long long *bad,
                         cudaStream_t st) {
  const size_t want = (rows + 255) / 256;
  k_cluster_count<<<(int)(want < 148 * 8 ? want : 148 * 8), 256, 0, st>>>(tp, first, rows, H, C, c0, nc, count, bad);
  return 1;
}

int launch_cluster_place(const DevCtx &c, int req, int layer, const int32_t *tp, int64_t n, int C, bool first_chunk, bool last_chunk, int32_t *place,
                         cudaStream_t st) {
  // as many warps as have room for their counters; one, counting in global memory, where none has
  int warps = kPlaceSmem / 4 / C;
  const int in_smem = warps >= 1;
  warps = warps < 1 ? 1 : warps > kPlaceWarps ? kPlaceWarps : warps;
  const size_t smem = in_smem ? (size_t)warps * C * 4 : 0;
  static bool configured_dev[kMaxDevices] = {};
  bool &configured = configured_dev[current_device_slot()];
  if (!configured) { cudaFuncSetAttribute(k_cluster_place, cudaFuncAttributeMaxDynamicSharedMemorySize, kPlaceSmem); configured = true; }
  k_cluster_place<<<c.Hkv, kPlaceWarps * 32, smem, st>>>(c, req, layer, tp, n, C, warps, in_smem, first_chunk, last_chunk, place);
  return 1;
}

int launch_cluster_tables(const DevCtx &c, int req, int layer, int C, int c0, int nc, int n_pages, int n_tokens, const int32_t *count, int slots,
                          cudaStream_t st) {
  int n = nc;
  if (c0 == 0) { n = C > n_pages ? C : n_pages; }
  k_cluster_tables<<<dim3((n + 255) / 256, c.Hkv), 256, 0, st>>>(c, req, layer, C, c0, nc, n_pages, n_tokens, count, slots);
  return 1;
}

int launch_cluster_scatter(const DevCtx &c, int req, int layer, const __nv_bfloat16 *k,
                           const __nv_bfloat16 *v, const int32_t *place, int64_t n_tokens,
                           cudaStream_t st) {
  const size_t rows = (size_t)n_tokens * c.Hkv;
  int grid = (int)((rows + 15) / 16 < 148 * 16 ? (rows + 15) / 16 : 148 * 16);
  if (grid < 1) grid = 1;
  k_cluster_scatter<<<grid, 256, 0, st>>>(c, req, layer, k, v, place, rows);
  return 1;
}

int launch_cluster_scatter_staged(const DevCtx &c, const __nv_bfloat16 *k, const __nv_bfloat16 *v, const int32_t *place,
                                  int n_tokens, int p0, int m, uint8_t *stage, cudaStream_t st) {
  size_t rows = (size_t)n_tokens * c.Hkv;
  int grid = (int)((rows + 15) / 16 < 148 * 16 ? (rows + 15) / 16 : 148 * 16);
  if (grid < 1) grid = 1;
  k_cluster_scatter_staged<<<grid, 256, 0, st>>>(c, k, v, place, n_tokens, p0, m, stage);
  return 1;
}

int launch_copy_centroids(const DevCtx &c, int req, int layer, const __nv_bfloat16 *cen,
                          int n_clusters, cudaStream_t st) {
  size_t rows = (size_t)n_clusters * c.Hkv;
  int grid = (int)((rows + 15) / 16 < 148 * 4 ? (rows + 15) / 16 : 148 * 4);
  if (grid < 1) grid = 1;
  k_copy_centroids<<<grid, 256, 0, st>>>(c, req, layer, cen, n_clusters);
  return 1;
}

}  // namespace spin
