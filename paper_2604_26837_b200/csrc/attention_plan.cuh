// How a launch of the attention kernel deals its sets to CTAs: host code, from what the host knows of the lists and what the
// GPU holds at once.
#pragma once
#include "spin_dev.cuh"

namespace spin {

constexpr int kAttnWarps = 4;              // warps of a CTA
constexpr int kWarpStages = 2;             // pages that a warp has in flight
constexpr int kClusterRows = 8;            // CTAs that a cluster may have everywhere
constexpr int kSharePages = 32, kExtraCtas = 2048;
constexpr int kCtaPages = kChunkPages;     // pages that a CTA has at least where rows merge through memory: at most ceil(n / 8) partials of a set
constexpr int kClusterPages = kCtaPages / 2;   // ... where they are a cluster, which writes no partials to memory
static_assert(kClusterPages == kAttnWarps, "a row short of its warps has one page per warp (see `plain` in attn_row)");

// What the GPU holds at once: CTAs, and clusters of so many CTAs each.
struct AttnGpu { int resident; int clusters[kClusterRows + 1]; };

enum AttnForm { kAttnWarp, kAttnCounted, kAttnRows };
struct AttnPlan {
  AttnForm form;
  int rows;                // CTAs per set in the grid
  int own;                 // CTAs that a set has as a rule
  int least, share;        // pages that a CTA has at least; pages per CTA beyond which a list gets more
  int cluster;             // a set's CTAs are a cluster of so many (0: they are not)
};

// Half as much again as a CTA's part of an average list.
__host__ __device__ inline long long share_of(long long pages, long long n_sets, int rows) {
  return (3 * pages + 2 * n_sets * rows - 1) / (2 * n_sets * rows);
}

// Clusters of r CTAs that the GPU holds without some waiting for room.  What cudaOccupancyMaxActiveClusters says needs every
// GPC packed perfectly, which the hardware does not do: the last few start when others have ended.  Lists of 24
// pages, us: 142 in clusters of three, as many as it says, 11.9, merged through memory 9.0; 138 8.9 and 9.0; 104 in
// clusters of four 9.1 and 9.0, 103 8.6 and 9.0; 82 in clusters of five 10.0 and 8.9, 80 8.5 and 8.8; 71 of six 8.9 and 8.7, 69 7.8
// and 8.7.  Pairs always fit, and clusters of seven and eight leave room in every GPC anyway (56 of seven 7.4 and 8.8, 48
// of eight, 33 pages, 7.9 and 8.7).
inline int clusters_at_once(const AttnGpu &gpu, int r) {
  return r < 2 ? gpu.resident : gpu.clusters[r] - (r > 2 && r < 7 ? gpu.clusters[r] / 32 : 0);
}

// As many CTAs per set as the GPU holds at once (444), and at least 8 pages for each: every CTA is
// resident, its pages stream through its stages, and CTAs share HBM by what they have in flight,
// so equal shares end together.  256 sets of 56 pages, 8 heads: 57.7 us with a CTA per 8 pages
// (four waves), 24 us with one CTA per set; 128 sets of 65 pages: lists complete to merged
// 34 us -> 17 us.
// Lists are not always equal.  One that leaves a CTA more than kSharePages and more than half as much
// again as the average list does is split further (256 lists, one of 500 pages and the rest of 8: 128 us
// without that, 17 with, 31 with a CTA per 8 pages; decode, 32 requests x 8 heads, one of 8192 tokens
// and the rest of 130: 152 us, 46, 74).  Below that a further split only costs: 256 lists of 56 pages, two
// CTAs each: 35 us instead of 25.  In a decode step the average is the host's estimate, and the grid has
// rows for the longest list it may meet, at most kExtraCtas of them, which leave at once where they
// are not needed (~1 ns each).  Where only the device knows the lengths, CTAs take the average from the
// counts, and fewer spare ones find out from them what is theirs.  That costs a call of even lists 1-2 us,
// so it is done where a list may leave a CTA more than 48 pages (72 lists, one of 354 pages and the rest of
// 8: 15 us with, 21 without, 17 with a CTA per 8 pages), or 64 where sets have one CTA each: there are so
// many of them then that looking costs most (256 lists of 56 pages: 25 us without, 27 with) and gains
// least (445 lists, one of 64 and the rest of 8: 19 without, 22 with).
// decode: lists of a decode step (est_pages of all of them together, about), else plain lists of up to max_pages.
// beside_scoring: CTAs move in one by one while a scoring grid still holds the SMs (Batch::attn_set_major).
inline AttnPlan attn_plan(const AttnGpu &gpu, bool decode, bool beside_scoring, int n_sets, int max_pages, long long est_pages, int max_chunks) {
  auto clamp = [](long long x, long long lo, long long hi) { return (int)(x > hi ? hi : x < lo ? lo : x); };
  const int chunks = clamp((max_pages + kCtaPages - 1) / kCtaPages, 1, max_chunks);
  AttnPlan p;
  p.cluster = 0;
  p.least = kCtaPages;
  p.own = clamp(gpu.resident / n_sets, 1, chunks);
  p.share = clamp(share_of(est_pages, n_sets, p.own), kSharePages, 1 << 30);
  p.rows = clamp((max_pages + p.share - 1) / p.share, p.own, chunks);
  // More sets than the GPU holds CTAs, and lists of one page or two per stage: a CTA of one warp each,
  // four times as many at once.  (16000 lists of one page: 134 us with four warps, 41 with one.)
  if (max_pages <= 2 * kWarpStages && n_sets > gpu.resident) { p.form = kAttnWarp; p.rows = 1; return p; }
  if (!decode && max_pages > (p.own > 1 ? 3 : 4) * kSharePages / 2 * p.own) {
    p.form = kAttnCounted;
    const int own = n_sets * p.own;
    p.rows = own + own * 2 / 3;              // (CTAs of the whole grid)
    return p;
  }
  p.form = kAttnRows;
  if (!decode) p.rows = p.own;
  p.rows = clamp(p.rows, p.own, clamp(kExtraCtas / n_sets, p.own, chunks));
  p.share = clamp((max_pages + p.rows - 1) / p.rows, p.share, 1 << 30);
  // Few rows, all resident: a cluster per set, which merges through shared memory (figures at merge_cluster).  The
  // merge costs little, so a row may be left with a page per warp.  As many CTAs as leave all clusters
  // resident at once, and no cluster where that gives a warp over an eighth more pages than it has without
  // one: 16 numbers of lists from 19 to 222 of 17 to 96 pages, the better of both within 4 % (55 lists of 60 pages,
  // seven CTAs in a cluster 9.9 us, eight without 9.0; 64 of 48, six 8.6 and 9.0).  Not where rows exceed what is resident at
  // once: the CTAs of a long list would have to find room together.  Nor beside a scoring grid that leaves room for one
  // CTA here and there: a cluster waits for room for all of its own in one GPC (8 requests of 131072 tokens, 8 heads, 64
  // pages and 163 slots per set: 206 us in clusters of six, 202 without; of 128 pages and 1024 slots 155 and 155).
  const int most = clamp(gpu.resident / n_sets, 1, kClusterRows);
  int fit = clamp((max_pages + kClusterPages - 1) / kClusterPages, 1, most);
  while (fit > 1 && clusters_at_once(gpu, fit) < n_sets) --fit;
  auto warp_pages = [&](int r) { return (max_pages + r * kAttnWarps - 1) / (r * kAttnWarps); };
  if (!beside_scoring && p.rows <= most && 8 * warp_pages(fit) <= 9 * warp_pages(p.rows)) {
    p.least = kClusterPages;
    p.own = p.rows = fit;
    if (p.rows > 1) p.cluster = p.rows;
  }
  return p;
}

}  // namespace spin
