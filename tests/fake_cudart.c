/* A stand-in for the CUDA runtime with two devices and no GPU, for the host
 * side of the library: memory is the host's, launches run nothing.  It keeps
 * what the tests look at -- the current device, launches on a stream of
 * another device (refused, as the runtime does), copies, the device on which
 * each kernel attribute was set, captured and launched graphs -- and answers pointer queries from a table
 * that the test fills in. */
#include <stddef.h>
#include <stdint.h>
#include <stdlib.h>
#include <string.h>

typedef struct { unsigned x, y, z; } dim3;

enum { kInvalidValue = 1, kInvalidResourceHandle = 400, kStreamDevice1 = 0x1000 };

int fake_device = 0;          /* the current device of the only thread */
int fake_launches = 0, fake_copies = 0, fake_refused = 0;
int fake_attributes[2] = {0, 0};
static int last_error = 0;
static struct { const char* p; size_t bytes; int type, device; } table[16];
static int entries = 0;

void fake_array(const void* p, size_t bytes, int type, int device) {
  table[entries].p = p;
  table[entries].bytes = bytes;
  table[entries].type = type;
  table[entries++].device = device;
}

int cudaGetDevice(int* d) { *d = fake_device; return 0; }
int cudaSetDevice(int d) { if (d < 0 || d > 1) return 101; fake_device = d; return 0; }
int cudaDeviceGetAttribute(int* v, int attr, int device) {
  (void)device;
  *v = attr == 16 ? 152 : attr == 97 ? 232448 : 0;   /* multiprocessors, opt-in shared memory */
  return 0;
}
int cudaGetLastError(void) { int e = last_error; last_error = 0; return e; }
const char* cudaGetErrorString(int e) { (void)e; return "fake"; }

/* cuPointerGetAttributes, for the five attributes in the order that the library asks for them */
static int pointer_attributes(unsigned n, const int* what, void** data, unsigned long long p) {
  static const int order[] = {2, 8, 9, 11, 12};   /* memory type, managed, device, range start, size */
  if (n != 5 || memcmp(what, order, sizeof order)) return kInvalidValue;
  *(unsigned*)data[0] = 0;
  for (int i = 0; i < entries; ++i)
    if ((const char*)(uintptr_t)p >= table[i].p && (const char*)(uintptr_t)p < table[i].p + table[i].bytes) {
      *(unsigned*)data[0] = table[i].type == 0 ? 0 : 2;
      *(int*)data[1] = table[i].type == 3;
      *(int*)data[2] = table[i].device;
      *(unsigned long long*)data[3] = (unsigned long long)(uintptr_t)table[i].p;
      *(size_t*)data[4] = table[i].bytes;
    }
  return 0;
}
int cudaGetDriverEntryPointByVersion(const char* name, void** fn, unsigned version, unsigned long long flags, int* found) {
  (void)version; (void)flags;
  *fn = strcmp(name, "cuPointerGetAttributes") == 0 ? (void*)pointer_attributes : NULL;
  *found = *fn ? 0 : 1;
  return 0;
}

int cudaMallocAsync(void** p, size_t n, void* s) { (void)s; *p = aligned_alloc(256, (n + 255) & ~(size_t)255); return 0; }
int cudaFreeAsync(void* p, void* s) { (void)s; free(p); return 0; }
int cudaHostAlloc(void** p, size_t n, unsigned f) { (void)f; *p = calloc(1, n); return 0; }
int cudaFreeHost(void* p) { free(p); return 0; }
int cudaMemcpyAsync(void* d, const void* s, size_t n, int kind, void* st) {
  (void)kind; (void)st;
  memmove(d, s, n);
  ++fake_copies;
  return 0;
}
int cudaMemsetAsync(void* d, int v, size_t n, void* s) { (void)s; memset(d, v, n); return 0; }
int cudaStreamCreateWithFlags(void** s, unsigned f) { (void)f; *s = (void*)0x2000; return 0; }
int cudaStreamDestroy(void* s) { (void)s; return 0; }
int cudaStreamSynchronize(void* s) { (void)s; return 0; }

int cudaFuncGetAttributes(void* a, const void* f) { (void)f; memset(a, 0, 4 * sizeof(size_t)); return 0; }
int cudaFuncSetAttribute(const void* f, int attr, int v) {
  (void)f; (void)attr; (void)v;
  ++fake_attributes[fake_device];
  return 0;
}
int cudaGetSymbolAddress(void** p, const void* s) { (void)s; static int word[4]; *p = word; return 0; }
int cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void* f, int t, size_t m, unsigned fl) {
  (void)f; (void)fl;
  const int by_memory = m ? (int)(227u * 1024u / m) : 32, by_registers = 65536 / (80 * t);
  *n = by_memory < by_registers ? by_memory : by_registers;
  return 0;
}
int cudaOccupancyMaxActiveClusters(int* n, const void* f, const void* cfg) { (void)f; (void)cfg; *n = 8; return 0; }

static struct { const void* f; const char* name; int launches; } kernels[256];
static int n_kernels = 0;
const char* fake_last_kernel = "";

static int launch(const void* f, void* stream) {
  if (stream == (void*)kStreamDevice1 && fake_device != 1) {
    ++fake_refused;
    return last_error = kInvalidResourceHandle;
  }
  ++fake_launches;
  for (int i = 0; i < n_kernels; ++i)
    if (kernels[i].f == f) {
      fake_last_kernel = kernels[i].name;
      ++kernels[i].launches;
    }
  return 0;
}
int fake_count(const char* part) {                  /* launches of the kernels with that in their name */
  int n = 0;
  for (int i = 0; i < n_kernels; ++i)
    if (strstr(kernels[i].name, part)) n += kernels[i].launches;
  return n;
}
static void* pushed_stream;
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t m, void* s) {
  (void)g; (void)b; (void)m;
  pushed_stream = s;
  return 0;
}
int __cudaPopCallConfiguration(dim3* g, dim3* b, size_t* m, void** s) {
  g->x = g->y = g->z = b->x = b->y = b->z = 1;
  *m = 0;
  *s = pushed_stream;
  return 0;
}
int __cudaGetKernel(void** k, const void* f) { *k = (void*)f; return 0; }
int __cudaLaunchKernel(void* k, dim3 g, dim3 b, void** a, size_t m, void* s) {
  (void)g; (void)b; (void)a; (void)m;
  return launch(k, s);
}
typedef struct { dim3 grid, block; size_t smem; void* stream; void* attrs; unsigned n; } Config;
int cudaLaunchKernelExC(const Config* c, const void* f, void** a) { (void)a; return launch(f, c->stream); }

void** __cudaRegisterFatBinary(void* p) { (void)p; static void* h; return &h; }
void __cudaRegisterFatBinaryEnd(void** h) { (void)h; }
void __cudaUnregisterFatBinary(void** h) { (void)h; }
void __cudaRegisterFunction(void** h, const char* f, char* device_f, const char* name) {
  (void)h; (void)device_f;
  if (n_kernels < 256) {
    kernels[n_kernels].f = f;
    kernels[n_kernels++].name = name;
  }
}
void __cudaRegisterVar(void) {}

int fake_captures = 0, fake_graph_launches = 0;
int cudaStreamBeginCapture(void* s, int mode) { (void)s; (void)mode; ++fake_captures; return 0; }
int cudaStreamEndCapture(void* s, void** g) { (void)s; *g = (void*)0x3000; return 0; }
int cudaGraphInstantiate(void** x, void* g, unsigned long long f) { (void)g; (void)f; *x = (void*)0x4000; return 0; }
int cudaGraphLaunch(void* x, void* s) { (void)x; (void)s; ++fake_graph_launches; return 0; }

/* not reached by these tests */
int cudaEventCreate(void** e) { *e = NULL; return kInvalidValue; }
int cudaEventDestroy(void* e) { (void)e; return 0; }
int cudaEventElapsedTime(float* t, void* a, void* b) { (void)a; (void)b; *t = 0; return kInvalidValue; }
int cudaEventRecord(void* e, void* s) { (void)e; (void)s; return kInvalidValue; }
int cudaEventSynchronize(void* e) { (void)e; return kInvalidValue; }
int cudaGraphAddKernelNode(void) { return kInvalidValue; }
int cudaGraphAddNode(void) { return kInvalidValue; }
int cudaGraphConditionalHandleCreate(void) { return kInvalidValue; }
int cudaGraphCreate(void) { return kInvalidValue; }
int cudaGraphDestroy(void) { return 0; }
int cudaGraphExecDestroy(void) { return 0; }
int cudaStreamBeginCaptureToGraph(void) { return kInvalidValue; }
