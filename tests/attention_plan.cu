// Prints the plan of a launch of attention for every line "decode beside_scoring sets pages chunks" of standard input; with an argument, checks
// what has to hold for every plan.
#include <cstdio>
#define SPIN_FILE_ID 0
#include "attention_plan.cuh"
using namespace spin;

// what the runtime says of a B200: three CTAs on each of 148 SMs
static const AttnGpu kGpu = {444, {0, 0, 222, 142, 104, 82, 71, 56, 48}};

static int check() {
  int plans = 0;
  for (int decode = 0; decode < 3; ++decode)     // 2: beside a scoring grid
    for (int sets = 1; sets < 3000; sets += sets < 460 ? 1 : 97)
      for (int pages = 1; pages < 3000; pages += pages < 140 ? 1 : 61) {
        const int chunks = (pages + kChunkPages - 1) / kChunkPages;
        const AttnPlan p = attn_plan(kGpu, decode > 0, decode > 1, sets, pages, decode ? (long long)sets * pages : 0, chunks);
        ++plans;
        bool ok = p.rows >= 1 && p.own >= 1 && p.share >= 1;
        if (p.cluster)         // all there at once, with a page for every warp but those of the last row
          ok = ok && decode < 2 && p.form == kAttnRows && p.cluster == p.rows && p.own == p.rows && p.rows > 1 && p.rows <= kClusterRows &&
               p.least == kClusterPages && (p.rows - 1) * kClusterPages < pages && sets <= clusters_at_once(kGpu, p.rows);
        else if (p.form == kAttnRows && p.rows > 1)
          ok = ok && p.least == kCtaPages && p.rows <= chunks;            // a partial for each
        else if (p.form == kAttnCounted)
          ok = ok && !decode && p.least == kCtaPages;
        else if (p.form == kAttnWarp)
          ok = ok && pages <= 2 * kWarpStages && p.rows == 1;
        if (!ok) { printf("decode %d, %d sets of %d pages: form %d, rows %d, own %d, least %d, cluster %d\n", decode, sets, pages, p.form, p.rows, p.own, p.least, p.cluster); return 1; }
      }
  printf("%d plans\n", plans);
  return 0;
}

int main(int argc, char **) {
  if (argc > 1) return check();
  int decode, beside, sets, pages, chunks;
  while (scanf("%d %d %d %d %d", &decode, &beside, &sets, &pages, &chunks) == 5) {
    const AttnPlan p = attn_plan(kGpu, decode, beside, sets, pages, decode ? (long long)sets * pages : 0, chunks);
    printf("%d %d %d\n", p.form, p.rows, p.cluster);
  }
  return 0;
}
