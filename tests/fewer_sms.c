/* A stand-in for the CUDA runtime with a given number of SMs, and a program that steps through the library on it: no kernel
 * runs, every launch is written down, and a cooperative one of more blocks than SMs is refused as the runtime refuses it.
 *   fewer_sms <SMs of the device> <SMs of the stream's green context, 0: it has none> single|list m n r [count]
 * prints the status and the names of the kernels of one step. */
#include <cuda.h>
#include <cuda_runtime_api.h>
#include <stdio.h>
#include <stdlib.h>
#include <string.h>

#include "fira.h"

static int sms, green_sms, logging;
static struct { const void* host; const char* name; } kernels[512];
static int nkernels;
static struct { dim3 grid, block; size_t smem; cudaStream_t st; } config;
static char memory[1 << 20];

void** __cudaRegisterFatBinary(void* f) { (void)f; static void* h; return &h; }
void __cudaRegisterFatBinaryEnd(void** h) { (void)h; }
void __cudaUnregisterFatBinary(void** h) { (void)h; }
void __cudaRegisterFunction(void** h, const char* host, char* dev, const char* name, int limit, uint3* t, uint3* b, dim3* bd, dim3* gd, int* w) {
  (void)h; (void)dev; (void)limit; (void)t; (void)b; (void)bd; (void)gd; (void)w;
  kernels[nkernels].host = host; kernels[nkernels++].name = name;
}
void __cudaRegisterVar(void** h, char* v, char* a, const char* n, int e, size_t s, int c, int g) { (void)h; (void)v; (void)a; (void)n; (void)e; (void)s; (void)c; (void)g; }
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t m, cudaStream_t s) { config.grid = g; config.block = b; config.smem = m; config.st = s; return 0; }
cudaError_t __cudaPopCallConfiguration(dim3* g, dim3* b, size_t* m, void* s) { *g = config.grid; *b = config.block; *m = config.smem; *(cudaStream_t*)s = config.st; return cudaSuccess; }
static cudaError_t launched(const void* f, unsigned blocks, int cooperative) {
  const int have = green_sms ? green_sms : sms;
  if (cooperative && (int)blocks > have) return cudaErrorCooperativeLaunchTooLarge;
  for (int i = 0; logging && i < nkernels; ++i)
    if (kernels[i].host == f) printf(" %s:%u", kernels[i].name, blocks);
  return cudaSuccess;
}
cudaError_t cudaLaunchKernel(const void* f, dim3 g, dim3 b, void** a, size_t m, cudaStream_t s) { (void)b; (void)a; (void)m; (void)s; return launched(f, g.x * g.y, 0); }
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* f, void** a) {
  int cooperative = 0;
  (void)a;
  for (unsigned i = 0; i < c->numAttrs; ++i) cooperative |= c->attrs[i].id == cudaLaunchAttributeCooperative && c->attrs[i].val.cooperative;
  return launched(f, c->gridDim.x, cooperative);
}
cudaError_t cudaGetDevice(int* d) { *d = 0; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, enum cudaDeviceAttr a, int d) { (void)d; *v = a == cudaDevAttrMultiProcessorCount ? sms : 0; return cudaSuccess; }
cudaError_t cudaFuncSetAttribute(const void* f, enum cudaFuncAttribute a, int v) { (void)f; (void)a; (void)v; return cudaSuccess; }
cudaError_t cudaOccupancyMaxActiveClusters(int* n, const void* f, const cudaLaunchConfig_t* c) { (void)f; (void)c; *n = sms / 2; return cudaSuccess; }
cudaError_t cudaGetSymbolAddress(void** p, const void* s) { (void)s; *p = (void*)(((size_t)memory + 255) / 256 * 256); return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, enum cudaMemcpyKind k, cudaStream_t st) { (void)d; (void)s; (void)n; (void)k; (void)st; return cudaSuccess; }
cudaError_t cudaMemsetAsync(void* d, int v, size_t n, cudaStream_t st) { (void)d; (void)v; (void)n; (void)st; return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t st) { (void)st; return cudaSuccess; }
cudaError_t cudaGetLastError(void) { return cudaSuccess; }
const char* cudaGetErrorString(cudaError_t e) { return e == cudaErrorCooperativeLaunchTooLarge ? "too many blocks in cooperative launch" : "error"; }

static CUresult encode(void) { return CUDA_SUCCESS; }
static CUresult get_current(CUcontext* c) { *c = (CUcontext)memory; return CUDA_SUCCESS; }
static CUresult get_green(CUstream s, CUgreenCtx* g) { (void)s; *g = green_sms ? (CUgreenCtx)memory : NULL; return CUDA_SUCCESS; }
static CUresult context_part(CUcontext c, CUdevResource* r, CUdevResourceType t) { (void)c; r->type = t; r->sm.smCount = sms; return CUDA_SUCCESS; }
static CUresult green_part(CUgreenCtx c, CUdevResource* r, CUdevResourceType t) { (void)c; r->type = t; r->sm.smCount = green_sms; return CUDA_SUCCESS; }
#undef cudaGetDriverEntryPoint
cudaError_t cudaGetDriverEntryPoint(const char* name, void** f, unsigned long long flags, enum cudaDriverEntryPointQueryResult* q) {
  (void)flags;
  *f = !strcmp(name, "cuTensorMapEncodeTiled") ? (void*)encode : !strcmp(name, "cuCtxGetCurrent") ? (void*)get_current : !strcmp(name, "cuStreamGetGreenCtx") ? (void*)get_green :
       !strcmp(name, "cuCtxGetDevResource") ? (void*)context_part : !strcmp(name, "cuGreenCtxGetDevResource") ? (void*)green_part : NULL;
  if (q) *q = *f ? cudaDriverEntryPointSuccess : cudaDriverEntryPointSymbolNotFound;
  return cudaSuccess;
}

int main(int argc, char** argv) {
  if (argc < 7) return 2;
  sms = atoi(argv[1]); green_sms = atoi(argv[2]);
  const int count = argc > 7 ? atoi(argv[7]) : 1;
  fira_hparams hp = {0.9f, 0.999f, 1e-8f, 1e-2f, 0.25f, 1.01f, 0, FIRA_FLAG_FORCE_SIMT};
  fira_matrix_desc* d = calloc(count, sizeof(*d));
  for (int i = 0; i < count; ++i) { d[i].m = atoi(argv[4]); d[i].n = atoi(argv[5]); d[i].r = atoi(argv[6]); d[i].dtype = FIRA_F32; }
  char* at = (char*)(((size_t)memory + 4095) / 4096 * 4096);        /* (an address; nothing is read or written there) */
  fira_status s;
  if (!strcmp(argv[3], "single")) {
    logging = 1;
    s = fira_step_single_noalloc(&hp, d, at, at, at, (float*)at, (float*)at, (float*)at, (int64_t*)at, -1.f, NULL);
  } else {
    size_t state, scratch;
    fira_ctx* c = NULL;
    s = fira_query_workspace(&hp, d, count, &state, &scratch);
    if (s == FIRA_OK) s = fira_init(&c, &hp, d, count, at, state, at, scratch, NULL);
    void** p = calloc(count, sizeof(*p));
    for (int i = 0; i < count; ++i) p[i] = at;
    logging = 1;
    if (s == FIRA_OK) s = fira_step(c, p, (const void* const*)p, -1.f);
    fira_destroy(c);
  }
  printf("\n%d %s\n", (int)s, fira_last_error());
  return 0;
}
