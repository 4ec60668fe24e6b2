// A CUDA runtime that runs nothing: it logs every launch, event record, event wait and stream
// synchronisation, and fails the call that the caller names.  Linked with plate.cu's object file and a
// stand-in for the stages of the grid, it shows on the CPU what ibfsa_fsi_step does with its streams.
//
//   fsi_streams FAIL STEPS PRIORITY GREEN
//     FAIL: number of the logged call of ibfsa_fsi_step that fails (from 0; -1: none)
//     PRIORITY: of the caller's stream; GREEN: 1 if it belongs to a green context
#include <cuda.h>
#include <cuda_runtime.h>
#include <stdio.h>
#include <stdlib.h>

#include <string>

#include "ibfsa_internal.h"

namespace {
int g_fail = -1, g_calls = 0, g_priority = 0;
bool g_green = false;
bool g_log = false;
cudaError_t g_error = cudaSuccess;
dim3 g_grid, g_block;
size_t g_smem;
cudaStream_t g_stream;
char g_handles[64];
int g_nhandles = 0;

cudaStream_t const MAIN = (cudaStream_t)0x1000;

void *handle() { return &g_handles[g_nhandles++]; }

std::string name(const void *p) {
  if (p == MAIN) return "main";
  return "h" + std::to_string((int)((const char *)p - g_handles));
}

cudaError_t called(const std::string &what) {
  if (!g_log) return cudaSuccess;
  const bool bad = g_calls++ == g_fail;
  printf("%s%s\n", what.c_str(), bad ? " FAILED" : "");
  if (bad) g_error = cudaErrorUnknown;
  return bad ? cudaErrorUnknown : cudaSuccess;
}
}  // namespace

extern "C" {
void **__cudaRegisterFatBinary(void *) {
  static void *h = nullptr;
  return &h;
}
void __cudaRegisterFatBinaryEnd(void **) {}
void __cudaUnregisterFatBinary(void **) {}
void __cudaRegisterFunction(void **, const char *, char *, const char *, int, uint3 *, uint3 *,
                            dim3 *, dim3 *, int *) {}
void __cudaRegisterVar(void **, char *, char *, const char *, int, size_t, int, int) {}
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t s, struct CUstream_st *st) {
  g_grid = g;
  g_block = b;
  g_smem = s;
  g_stream = st;
  return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3 *g, dim3 *b, size_t *s, void *st) {
  *g = g_grid;
  *b = g_block;
  *s = g_smem;
  *(cudaStream_t *)st = g_stream;
  return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t *k, const void *f) {
  *k = (cudaKernel_t)f;
  return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t, dim3, dim3, void **, size_t, cudaStream_t st) {
  return called("launch " + name(st));
}
cudaError_t cudaGetLastError() {
  const cudaError_t e = g_error;
  g_error = cudaSuccess;
  return e;
}
const char *cudaGetErrorString(cudaError_t) { return "failed on purpose"; }
cudaError_t cudaGetDevice(int *d) {
  *d = 0;
  return cudaSuccess;
}
cudaError_t cudaFuncSetAttribute(const void *, cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t cudaDeviceGetStreamPriorityRange(int *least, int *greatest) {
  *least = 0;
  *greatest = -5;
  return cudaSuccess;
}
cudaError_t cudaStreamCreateWithPriority(cudaStream_t *s, unsigned, int priority) {
  *s = (cudaStream_t)handle();
  printf("stream %s %d\n", name(*s).c_str(), priority);
  return cudaSuccess;
}
cudaError_t cudaStreamGetPriority(cudaStream_t, int *priority) {
  *priority = g_priority;
  return cudaSuccess;
}
static CUresult green_context(CUstream, CUgreenCtx *ctx) {
  *ctx = g_green ? (CUgreenCtx)handle() : nullptr;
  return CUDA_SUCCESS;
}
cudaError_t cudaGetDriverEntryPointByVersion(const char *symbol, void **f, unsigned, unsigned long long,
                                             cudaDriverEntryPointQueryResult *r) {
  *f = std::string(symbol) == "cuStreamGetGreenCtx" ? (void *)green_context : nullptr;
  *r = *f ? cudaDriverEntryPointSuccess : cudaDriverEntryPointSymbolNotFound;
  return cudaSuccess;
}
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned) {
  *e = (cudaEvent_t)handle();
  return cudaSuccess;
}
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t s) {
  return called("record " + name(e) + " " + name(s));
}
cudaError_t cudaStreamWaitEvent(cudaStream_t s, cudaEvent_t e, unsigned) {
  return called("wait " + name(s) + " " + name(e));
}
cudaError_t cudaStreamSynchronize(cudaStream_t s) { return called("sync " + name(s)); }
cudaError_t cudaMemsetAsync(void *, int, size_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void *, const void *, size_t, cudaMemcpyKind, cudaStream_t) {
  return cudaSuccess;
}
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes *, const void *) {
  return cudaErrorInvalidValue;
}
}

namespace ibfsa {
cudaError_t grid_stage(Grid *G, const StageArgs &s) {
  const cudaError_t e = called("launch " + name(G->stream));
  if (e != cudaSuccess) return e;
  return s.forces ? cudaEventRecord(s.forces, G->stream) : cudaSuccess;
}
void prof_begin(Prof *, cudaStream_t) {}
void prof_end(Prof *, int, cudaStream_t) {}
double source_scale(const Grid &, double) { return 0.0; }
int api_fail(int code, const char *) { return code; }
}  // namespace ibfsa

int main(int, char **argv) {
  using namespace ibfsa;
  ibfsa_plate_desc d{};
  d.n_el = 4;
  d.n_markers = 16;
  d.length = d.rho_s = d.K_S = d.K_B = 1.0;
  d.newton_max = 10;
  d.newton_tol = 1e-10;
  size_t bytes = 0;
  if (ibfsa_plate_workspace_bytes(&d, &bytes)) return 2;
  void *ws = aligned_alloc(256, (bytes + 255) / 256 * 256);  // never read
  ibfsa_plate *p = nullptr;
  g_priority = atoi(argv[3]);
  g_green = atoi(argv[4]) != 0;
  if (ibfsa_plate_create(&d, ws, bytes, MAIN, &p)) return 3;
  ibfsa_grid *g = new ibfsa_grid();
  g->g.p.dim = g->g.d.dim = 2;
  g->g.d.max_markers = 16;
  g->g.stream = MAIN;
  g_fail = atoi(argv[1]);
  g_log = true;
  const int rc = ibfsa_fsi_step(g, p, 0.01, atoi(argv[2]));
  printf("returned %d\n", rc);
  return 0;
}
