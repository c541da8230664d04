/* Stand-ins for the CUDA runtime calls of the library's host side, for tests of
 * it without a GPU: "device" memory is host memory, every call that touches it is
 * recorded, and a launch is recorded instead of run.  Preloaded before libcudart. */
#include <stdlib.h>
#include <string.h>

typedef int cudaError_t;
enum { kMaxCalls = 256 };
static char g_calls[kMaxCalls]; /* m(emcpy), s(et), d(evice synchronise) */
static struct {
  const void* dst;
  size_t n;
} g_copy[kMaxCalls]; /* of the call of the same index, where it is a memcpy */
static int g_n;
static int g_fail_at = -1; /* the recorded call that fails */
static long long g_live;   /* allocations not freed */

static cudaError_t record(char c) {
  if (g_n < kMaxCalls - 1) g_calls[g_n++] = c;
  return g_n - 1 == g_fail_at ? 1 : 0;
}
const char* host_cudart_calls(void) { return g_calls; }
const void* host_cudart_copy_dst(int i) { return g_copy[i].dst; }
size_t host_cudart_copy_bytes(int i) { return g_copy[i].n; }
long long host_cudart_live(void) { return g_live; }
void host_cudart_reset(int fail_at) {
  memset(g_calls, 0, sizeof g_calls);
  g_n = 0;
  g_fail_at = fail_at;
}

cudaError_t cudaGetDevice(int* d) { return *d = 0; }
cudaError_t cudaSetDevice(int d) { return d != 0; }
cudaError_t cudaDeviceGetAttribute(int* v, int attr, int dev) {
  (void)dev;
  /* cudaDevAttrMultiProcessorCount, ComputeCapabilityMajor, ComputeCapabilityMinor */
  *v = attr == 16 ? 152 : attr == 75 ? 10 : attr == 76 ? 3 : 0;
  return 0;
}
cudaError_t cudaMalloc(void** p, size_t n) {
  *p = aligned_alloc(256, (n + 255) / 256 * 256 + 256);
  if (*p) ++g_live;
  return *p ? 0 : 2;
}
cudaError_t cudaFree(void* p) {
  if (p) --g_live;
  free(p);
  return 0;
}
cudaError_t cudaMemcpy(void* dst, const void* src, size_t n, int kind) {
  (void)kind;
  g_copy[g_n].dst = dst, g_copy[g_n].n = n;
  const cudaError_t e = record('m');
  if (!e) memcpy(dst, src, n);
  return e;
}
cudaError_t cudaMemset(void* p, int v, size_t n) {
  const cudaError_t e = record('s');
  if (!e) memset(p, v, n);
  return e;
}
cudaError_t cudaDeviceSynchronize(void) { return record('d'); }
cudaError_t cudaFuncSetAttribute(const void* f, int attr, int v) { return (void)f, (void)attr, (void)v, 0; }
cudaError_t cudaOccupancyMaxActiveClusters(int* n, const void* f, const void* cfg) {
  (void)f, (void)cfg;
  *n = 76;
  return 0;
}

/* Launches: threads per block, and the work list of the CTA-pair kernel (the first
 * member of its sixth parameter; null for the other kernels). */
enum { kMaxLaunches = 64, kPairThreads = 224 };
static struct {
  unsigned threads;
  const void* list;
} g_launch[kMaxLaunches];
static int g_launches;
int host_cudart_launches(void) { return g_launches; }
unsigned host_cudart_threads(int i) { return g_launch[i].threads; }
const void* host_cudart_list(int i) { return g_launch[i].list; }

struct config {
  unsigned grid[3], block[3]; /* the first members of cudaLaunchConfig_t */
};
cudaError_t cudaLaunchKernelExC(const struct config* cfg, const void* f, void** args) {
  (void)f;
  if (cfg->grid[1] > 65535 || cfg->grid[2] > 65535) return 9; /* cudaErrorInvalidConfiguration */
  if (g_launches < kMaxLaunches) {
    g_launch[g_launches].threads = cfg->block[0];
    g_launch[g_launches].list = cfg->block[0] == kPairThreads ? *(const void**)args[5] : NULL;
  }
  ++g_launches;
  return 0;
}
cudaError_t cudaGetLastError(void) { return 0; }
static int encode_tiled(void* map) { return memset(map, 0, 128), 0; }
cudaError_t cudaGetDriverEntryPointByVersion(const char* name, void** p, unsigned version, unsigned long long flags,
                                             int* found) {
  (void)name, (void)version, (void)flags;
  *p = (void*)encode_tiled;
  *found = 0; /* cudaDriverEntryPointSuccess */
  return 0;
}
