// Runs the attention kernel over hand-made sets whose flags, turns or pages do not come, and checks what it leaves
// behind.  Every wait has a limit, so each scene ends by itself.  Prints one line per scene; exit code 0 if all hold.
// Built twice: as it is, and with SPIN_LANDED_POLLS=0, where a warp gives up on a page at once.
#include <vector>
#include "attention.cu"
using namespace spin;
void Prof::mark(cudaStream_t, int) {}             // timing of launches belongs to the host runtime

namespace waits {
constexpr int kSets = 6, kMiss = 17, kGpuPages = 256, kHostPages = 256, kG = 4, kEpoch = 5;
bool ok_all = true;

template <typename T> T *device(size_t n, int fill = 0) {
  T *p = nullptr;
  if (cudaMalloc(&p, n * sizeof(T)) != cudaSuccess || cudaMemset(p, fill, n * sizeof(T)) != cudaSuccess) { printf("no device memory\n"); exit(3); }
  return p;
}
template <typename T> void put(T *d, const std::vector<T> &h) { cudaMemcpy(d, h.data(), h.size() * sizeof(T), cudaMemcpyHostToDevice); }

// Lists of 40 pages go to clusters of eight CTAs, which merge through shared memory; those of 80 pages to ten CTAs, which
// merge through memory.
// list: 1 = the list is complete; slots: 1 = the missed pages have their slots; early: descriptors of the first flag (negative:
// the flag does not come); closed: turns closed so far, from which the window counts; timeout, zeros: what is expected
void scene(int kList, const char *name, int list, int slots, int early, int n_miss, int closed, bool timeout, bool zeros) {
  const int kStride = kList + 1;                 // max_pages + tail_cap
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
    first[b] = (unsigned long long)(early < 0 ? kEpoch - 1 : kEpoch) << 32 | (unsigned)kList << 12 | (unsigned)max(early, 0);
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
                    untouched == (early < 0 ? (int)o.size() : 0) && (!zeros || nonzero == 0) && (timeout || (nonzero == (int)o.size() && link[0] == 2 * kSets * n_miss && !k.error_bits));
  printf("%d pages: %-40s %s: cuda %d, error bits %u, turns taken %d, closed %d, outputs not zero %d, not written %d\n", kList, name, good ? "ok" : "WRONG", (int)e,
         k.error_bits, link[0], link[kLinkDone] - closed, nonzero, untouched);
  ok_all = ok_all && good;
  for (void *p : {(void *)c.gpu_pages, (void *)c.page_desc, (void *)c.page_src, (void *)c.ready, (void *)c.tail_ready, (void *)c.ready1,
                  (void *)c.link, (void *)c.att_part, (void *)c.att_count, (void *)c.counters, (void *)q, (void *)out})
    cudaFree(p);
  cudaFreeHost(host);
}

// The merge by a cluster of `rows` CTAs, of which one (missing >= 0) has waited for its list in vain: the outputs are
// the rows' average, or stay as they are.
template <int G> __global__ void k_meet(__nv_bfloat16 *out, int rows, int missing) {
  extern __shared__ __align__(128) uint8_t smem[];
  __shared__ ClusterPart<G> part;
  const int row = blockIdx.y;
  for (int e = threadIdx.x; e < G * kHeadDim; e += kAttnThreads) cluster_outputs(smem)[e] = (float)(row + 1);
  for (int g = threadIdx.x; g < G; g += kAttnThreads) part.ml[g] = make_float2(0.f, 1.f);
  __syncthreads();
  merge_cluster<G>(part, smem, out, row, row == missing ? -1 : rows);
}
template <int G> void meeting(int rows, int missing) {
  __nv_bfloat16 *out = device<__nv_bfloat16>(G * kHeadDim, 0x55);
  cudaFuncSetAttribute(k_meet<G>, cudaFuncAttributeMaxDynamicSharedMemorySize, kAttnSmem);
  launch_pdl(k_meet<G>, dim3(1, rows), dim3(kAttnThreads), (size_t)kAttnSmem, nullptr, dim3(1, rows), out, rows, missing);
  const cudaError_t e = cudaDeviceSynchronize();
  std::vector<__nv_bfloat16> o(G * kHeadDim);
  cudaMemcpy(o.data(), out, o.size() * 2, cudaMemcpyDeviceToHost);
  int right = 0;
  for (const __nv_bfloat16 &x : o) {
    uint16_t bits;
    memcpy(&bits, &x, 2);
    right += missing >= 0 ? bits == 0x5555 : __bfloat162float(x) == 0.5f * (float)(rows + 1);
  }
  const bool good = e == cudaSuccess && right == (int)o.size();
  printf("%d heads, %d rows, %2d missing: %s: cuda %d, outputs right %d of %d\n", G, rows, missing, good ? "ok" : "WRONG", (int)e, right, (int)o.size());
  ok_all = ok_all && good;
  cudaFree(out);
}
template <int G> void meetings() {
  for (int rows = 2; rows <= kClusterRows; ++rows)
    for (int missing = -1; missing < rows; ++missing) meeting<G>(rows, missing);
}
}  // namespace waits

int main() {
  using namespace waits;
  for (int pages : {40, 80}) {
    if (kLandedPolls > 0) {
      scene(pages, "everything comes", 1, 1, kMiss, kMiss, 0, false, false);
      scene(pages, "no first flag", 0, 0, -1, kMiss, 0, true, false);
      scene(pages, "no list, nothing missed", 0, 0, 0, 0, 0, true, true);
      scene(pages, "no list, missed pages on their way", 0, 0, kMiss, kMiss, 0, true, true);
      scene(pages, "no slots for the missed pages", 1, 0, kMiss, kMiss, 0, true, false);
      scene(pages, "no turn on the link, early pages", 1, 1, kMiss, kMiss, -(1 << 20), true, false);
      scene(pages, "no turn on the link, late pages", 1, 1, 0, kMiss, -(1 << 20), true, false);
    } else {
      scene(pages, "no hit ever lands", 1, 1, 0, 0, 0, true, true);
      scene(pages, "no page ever lands, early misses", 1, 1, kMiss, kMiss, 0, true, true);
      scene(pages, "no page ever lands, late misses", 1, 1, 0, kMiss, 0, true, true);
      scene(pages, "no page ever lands, one miss", 1, 1, 1, 1, 0, true, true);
    }
  }
  if (kLandedPolls > 0) { meetings<1>(); meetings<4>(); meetings<8>(); }
  return ok_all ? 0 : 1;
}
