/* A CUDA runtime that launches nothing: the library's objects linked against it run their host
 * code on a machine without a GPU.  It keeps a log of launches and can refuse cooperative ones. */
#include <cuda_runtime_api.h>
#include <stdio.h>
#include <string.h>

static struct { const void* host; const char* name; } kernels[4096];
static int n_kernels;
static char text[1 << 16];
static cudaError_t last;
static int sms = 152, refuse, refusals;

/* the next `n` cooperative launches fail with `error` */
void fake_refuse(int error, int n) { refuse = error, refusals = n; }
void fake_sms(int n) { sms = n; }
int fake_last_error(void) { return last; }
/* the launches since the last call: "name blocks flags" lines, flags c (cooperative), p (launched
 * behind the one before); memsets as "memset bytes" */
const char* fake_log(void) {
  static char out[sizeof text];
  memcpy(out, text, sizeof text);
  text[0] = 0;
  return out;
}

static const char* name_of(const void* f) {
  for (int i = 0; i < n_kernels; ++i)
    if (kernels[i].host == f) return kernels[i].name;
  return "?";
}
static void note(const char* name, unsigned long long n, const char* flags) {
  const size_t at = strlen(text);
  snprintf(text + at, sizeof text - at, "%s %llu %s\n", name, n, flags);
}

void** __cudaRegisterFatBinary(void* p) { static void* h; (void)p; return &h; }
void __cudaRegisterFatBinaryEnd(void** h) { (void)h; }
void __cudaUnregisterFatBinary(void** h) { (void)h; }
void __cudaRegisterFunction(void** h, const char* host, char* dev, const char* name, int n, void* a, void* b, void* c,
                            void* d, int* e) {
  (void)h, (void)dev, (void)n, (void)a, (void)b, (void)c, (void)d, (void)e;
  if (n_kernels < 4096) kernels[n_kernels].host = host, kernels[n_kernels++].name = name;
}
void __cudaRegisterVar(void** h, char* host, char* dev, const char* name, int ext, size_t size, int c, int g) {
  (void)h, (void)host, (void)dev, (void)name, (void)ext, (void)size, (void)c, (void)g;
}

static dim3 grid_, block_;
static size_t smem_;
static void* stream_;
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t m, void* s) {
  grid_ = g, block_ = b, smem_ = m, stream_ = s;
  return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3* g, dim3* b, size_t* m, void* s) {
  *g = grid_, *b = block_, *m = smem_, *(void**)s = stream_;
  return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* f) {
  *k = (cudaKernel_t)f;
  return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3 g, dim3 b, void** args, size_t m, cudaStream_t s) {
  (void)b, (void)args, (void)m, (void)s;
  note(name_of((const void*)k), 1ull * g.x * g.y * g.z, "-");
  return cudaSuccess;
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* f, void** args) {
  int coop = 0, pdl = 0;
  (void)args;
  for (unsigned i = 0; i < c->numAttrs; ++i) {
    coop |= c->attrs[i].id == cudaLaunchAttributeCooperative && c->attrs[i].val.cooperative;
    pdl |= c->attrs[i].id == cudaLaunchAttributeProgrammaticStreamSerialization;
  }
  if (coop && refusals > 0) {
    --refusals;
    return last = (cudaError_t)refuse;
  }
  note(name_of(f), 1ull * c->gridDim.x * c->gridDim.y * c->gridDim.z, coop ? "c" : (pdl ? "p" : "-"));
  return cudaSuccess;
}

cudaError_t cudaGetLastError(void) {
  const cudaError_t e = last;
  last = cudaSuccess;
  return e;
}
const char* cudaGetErrorString(cudaError_t e) { (void)e; return "an error of the fake runtime"; }
cudaError_t cudaGetDevice(int* d) { *d = 0; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, enum cudaDeviceAttr a, int d) {
  (void)d;
  *v = a == cudaDevAttrMultiProcessorCount ? sms : a == cudaDevAttrMaxSharedMemoryPerBlockOptin ? 232448 : 1;
  return cudaSuccess;
}
cudaError_t cudaFuncSetAttribute(const void* f, enum cudaFuncAttribute a, int v) { (void)f, (void)a, (void)v; return cudaSuccess; }
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void* f, int t, size_t m, unsigned fl) {
  (void)f, (void)t, (void)fl;
  *n = m > 116000 ? 1 : 3;
  return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessor(int* n, const void* f, int t, size_t m) {
  return cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(n, f, t, m, 0);
}
cudaError_t cudaOccupancyMaxActiveClusters(int* n, const void* f, const cudaLaunchConfig_t* c) { (void)f, (void)c; *n = sms / 2; return cudaSuccess; }
cudaError_t cudaMemsetAsync(void* p, int v, size_t n, cudaStream_t s) { (void)p, (void)v, (void)s; note("memset", n, "-"); return cudaSuccess; }
cudaError_t cudaMemset2DAsync(void* p, size_t pitch, int v, size_t w, size_t h, cudaStream_t s) { (void)p, (void)pitch, (void)v, (void)s; note("memset", w * h, "-"); return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void* d, const void* p, size_t n, enum cudaMemcpyKind k, cudaStream_t s) { (void)d, (void)p, (void)k, (void)s; note("memcpy", n, "-"); return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t s, cudaEvent_t e, unsigned f) { (void)s, (void)e, (void)f; return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t s) { (void)e, (void)s; return cudaSuccess; }
cudaError_t cudaStreamIsCapturing(cudaStream_t s, enum cudaStreamCaptureStatus* c) { (void)s; *c = cudaStreamCaptureStatusNone; return cudaSuccess; }
cudaError_t cudaGetSymbolAddress(void** p, const void* s) { *p = (void*)s; return cudaSuccess; }
static int encode(void) { return 0; }   /* cuTensorMapEncodeTiled */
cudaError_t cudaGetDriverEntryPointByVersion(const char* n, void** p, unsigned v, unsigned long long f, enum cudaDriverEntryPointQueryResult* r) {
  (void)n, (void)v, (void)f;
  *p = (void*)encode;
  if (r) *r = cudaDriverEntryPointSuccess;
  return cudaSuccess;
}
