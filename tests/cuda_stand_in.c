/* A CUDA runtime without a device, for the host side of the library: host memory is real, device memory an
 * address range that nothing touches, kernels do not run.  It notes the device each kernel was launched on, keeps the
 * runtime's last error as the real one does, and makes the launch, asynchronous copy or fill fail whose turn the test says. */
#include <stddef.h>
#include <stdlib.h>
#include <string.h>

#define API __attribute__((visibility("default")))
typedef int err;
enum { kDevices = 2, kLaunchFailed = 719, kBadDevice = 101 };
static int current, last, fail_in = -1, on_device[kDevices], synced_device[kDevices];

static err status(err e) { if (e) last = e; return e; }
API err cudaGetLastError(void) { err e = last; last = 0; return e; }
API err cudaPeekAtLastError(void) { return last; }
API const char *cudaGetErrorString(err e) { return e ? "stand-in error" : "no error"; }
API err cudaGetDevice(int *d) { *d = current; return 0; }
API err cudaSetDevice(int d) { if (d < 0 || d >= kDevices) return status(kBadDevice); current = d; return 0; }
API err cudaDeviceGetAttribute(int *v, int a, int d) { (void)a; (void)d; *v = 148; return 0; }
API err cudaDeviceSynchronize(void) { ++synced_device[current]; return 0; }
API err cudaStreamSynchronize(void *s) { (void)s; return 0; }
API err cudaStreamCreateWithFlags(void **s, unsigned f) { (void)f; *s = (void *)64; return 0; }
API err cudaStreamDestroy(void *s) { (void)s; return 0; }
API err cudaStreamWaitEvent(void *s, void *e, unsigned f) { (void)s; (void)e; (void)f; return 0; }
API err cudaEventCreateWithFlags(void **e, unsigned f) { (void)f; *e = (void *)64; return 0; }
API err cudaEventDestroy(void *e) { (void)e; return 0; }
API err cudaEventRecord(void *e, void *s) { (void)e; (void)s; return 0; }
API err cudaHostAlloc(void **p, size_t n, unsigned f) { (void)f; *p = malloc(n); return *p ? 0 : status(2); }
API err cudaFreeHost(void *p) { free(p); return 0; }
API err cudaHostGetDevicePointer(void **d, void *h, unsigned f) { (void)f; *d = h; return 0; }
API err cudaMemset(void *p, int v, size_t n) { (void)p; (void)v; (void)n; return 0; }
/* device to host: zeros */
API err cudaMemcpy(void *d, const void *s, size_t n, int kind) { (void)s; if (kind == 2) memset(d, 0, n); return 0; }
static err turn(void) { return fail_in >= 0 && fail_in-- == 0 ? status(kLaunchFailed) : 0; }
API err cudaMemcpyAsync(void *d, const void *s, size_t n, int kind, void *st) { (void)st; cudaMemcpy(d, s, n, kind); return turn(); }
API err cudaMemsetAsync(void *p, int v, size_t n, void *s) { (void)p; (void)v; (void)n; (void)s; return turn(); }
API err cudaFuncSetAttribute(const void *f, int a, int v) { (void)f; (void)a; (void)v; return 0; }
static err launch(void) {
  ++on_device[current];
  return turn();
}
API err cudaLaunchKernel(const void *f, ...) { (void)f; return launch(); }
API err cudaLaunchKernelExC(const void *c, const void *f, void **a) { (void)c; (void)f; (void)a; return launch(); }

/* for the test */
API void stand_in_fail(int in) { fail_in = in; }             /* the launch, copy or fill after so many more fails */
API void stand_in_stale(int e) { last = e; }                 /* an error that some other call has left behind */
API int stand_in_launches(int device) { return on_device[device]; }
API int stand_in_synced(int device) { return synced_device[device]; }
