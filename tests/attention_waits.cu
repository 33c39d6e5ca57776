// Runs the attention kernel over hand-made sets whose flags, turns or pages do not come, and checks what it leaves
// behind.  Every wait has a limit, so each scene ends by itself.  Prints one line per scene; exit code 0 if all hold.
// Built twice: as it is, and with SPIN_LANDED_POLLS=0, where a warp gives up on a page at once.
#include <vector>
#include "attention.cu"
using namespace spin;
void Prof::mark(cudaStream_t, int) {}             // timing of launches belongs to the host runtime

namespace {
constexpr int kSets = 6, kList = 40, kMiss = 17, kGpuPages = 256, kHostPages = 256, kG = 4, kEpoch = 5;
constexpr int kStride = kList + 1;               // max_pages + tail_cap
bool ok_all = true;

template <typename T> T *device(size_t n, int fill = 0) {
  T *p = nullptr;
  if (cudaMalloc(&p, n * sizeof(T)) != cudaSuccess || cudaMemset(p, fill, n * sizeof(T)) != cudaSuccess) { printf("no device memory\n"); exit(3); }
  return p;
}
template <typename T> void put(T *d, const std::vector<T> &h) { cudaMemcpy(d, h.data(), h.size() * sizeof(T), cudaMemcpyHostToDevice); }

// list: 1 = the list is complete; slots: 1 = the missed pages have their slots; early: descriptors of the first flag;
// closed: turns closed so far, from which the window counts; timeout, zeros: what is expected
void scene(const char *name, int list, int slots, int early, int n_miss, int closed, bool timeout, bool zeros) {
  DevCtx c{};
  c.num_layers = 1; c.Hkv = 2; c.G = kG; c.Hq = 2 * kG;
  c.max_pages = c.topk = kList; c.tail_cap = 1; c.max_chunks = (kStride + kChunkPages - 1) / kChunkPages;
  c.sm_scale = 0.088f;
  c.n_gpu_pages = kGpuPages; c.n_host_pages = kHostPages;
  c.gpu_pages = device<uint8_t>((size_t)kGpuPages * kPageBytes, 0x3f);          // bf16 0.747
  uint8_t *host = nullptr;
  if (cudaMallocHost(&host, (size_t)kHostPages * kPageBytes) != cudaSuccess) { printf("no pinned memory\n"); exit(3); }
  memset(host, 0x3f, (size_t)kHostPages * kPageBytes);
  c.host_pages = host;
  c.page_desc = device<int4>(kSets * kStride);
  c.page_src = device<int32_t>(kSets * kStride);
  std::vector<int4> desc(kSets * kStride);
  std::vector<int32_t> src(kSets * kStride), ready(kSets, list ? 2 * kEpoch + slots : 0), tails(kSets, kEpoch), link(kLinkDone + 1, 0);
  std::vector<unsigned long long> first(kSets);
  for (int b = 0; b < kSets; ++b) {
    for (int i = 0; i < kList; ++i) {
      const int at = b * kStride + i;
      src[at] = (b * kList + i) % kGpuPages;
      desc[at] = i < n_miss ? make_int4(-3, (b * kList + i) % kHostPages, 0xffff, i) : make_int4(src[at], -1, 0xffff, i);
    }
    first[b] = (unsigned long long)kEpoch << 32 | (unsigned)kList << 12 | (unsigned)early;
  }
  put(c.page_desc, desc); put(c.page_src, src);
  c.ready = device<int32_t>(kSets); c.tail_ready = device<int32_t>(kSets);
  c.ready1 = device<unsigned long long>(kSets);
  put(c.ready, ready); put(c.tail_ready, tails); put(c.ready1, first);
  c.link = device<int32_t>(kLinkDone + 1);
  link[kLinkDone] = closed;
  put(c.link, link);
  c.att_part = device<float>((size_t)kSets * c.max_chunks * kG * (kHeadDim + 2));
  c.att_ml = reinterpret_cast<float2 *>(c.att_part + (size_t)kSets * c.max_chunks * kG * kHeadDim);
  c.att_count = device<int32_t>(kSets);
  c.counters = device<Counters>(1);
  Batch bt{};
  bt.n_req = kSets / c.Hkv; bt.epoch = kEpoch;
  for (int i = 0; i < bt.n_req; ++i) bt.n_partitions[i] = kList;
  __nv_bfloat16 *q = device<__nv_bfloat16>(kSets * kG * kHeadDim, 0x3c), *out = device<__nv_bfloat16>(kSets * kG * kHeadDim, 0x55);
  for (int call = 0; call < 2; ++call) {                                        // the second meets what the first has left
    cudaMemset(c.att_count, 0, kSets * 4);
    launch_attention(c, bt, q, out, kList, (long long)kSets * kList, nullptr, nullptr);
    cudaDeviceSynchronize();
  }
  const cudaError_t e = cudaDeviceSynchronize();
  Counters k{};
  cudaMemcpy(&k, c.counters, sizeof k, cudaMemcpyDeviceToHost);
  cudaMemcpy(link.data(), c.link, link.size() * 4, cudaMemcpyDeviceToHost);
  std::vector<uint16_t> o(kSets * kG * kHeadDim);
  cudaMemcpy(o.data(), out, o.size() * 2, cudaMemcpyDeviceToHost);
  int nonzero = 0, untouched = 0;
  for (uint16_t x : o) { nonzero += x != 0; untouched += x == 0x5555; }
  const bool good = e == cudaSuccess && ((k.error_bits & kErrTimeout) != 0) == timeout && link[0] == link[kLinkDone] - closed &&
                    untouched == 0 && (!zeros || nonzero == 0) && (timeout || (nonzero == (int)o.size() && link[0] == 2 * kSets * n_miss && !k.error_bits));
  printf("%-40s %s: cuda %d, error bits %u, turns taken %d, closed %d, outputs not zero %d, not written %d\n", name, good ? "ok" : "WRONG", (int)e,
         k.error_bits, link[0], link[kLinkDone] - closed, nonzero, untouched);
  ok_all = ok_all && good;
  for (void *p : {(void *)c.gpu_pages, (void *)c.page_desc, (void *)c.page_src, (void *)c.ready, (void *)c.tail_ready, (void *)c.ready1,
                  (void *)c.link, (void *)c.att_part, (void *)c.att_count, (void *)c.counters, (void *)q, (void *)out})
    cudaFree(p);
  cudaFreeHost(host);
}
}  // namespace

int main() {
  if (kLandedPolls > 0) {
    scene("everything comes", 1, 1, kMiss, kMiss, 0, false, false);
    scene("no list, nothing missed", 0, 0, 0, 0, 0, true, true);
    scene("no list, missed pages on their way", 0, 0, kMiss, kMiss, 0, true, true);
    scene("no slots for the missed pages", 1, 0, kMiss, kMiss, 0, true, false);
    scene("no turn on the link, early pages", 1, 1, kMiss, kMiss, -(1 << 20), true, false);
    scene("no turn on the link, late pages", 1, 1, 0, kMiss, -(1 << 20), true, false);
  } else {
    scene("no hit ever lands", 1, 1, 0, 0, 0, true, true);
    scene("no page ever lands, early misses", 1, 1, kMiss, kMiss, 0, true, true);
    scene("no page ever lands, late misses", 1, 1, 0, kMiss, 0, true, true);
    scene("no page ever lands, one miss", 1, 1, 1, 1, 0, true, true);
  }
  return ok_all ? 0 : 1;
}
