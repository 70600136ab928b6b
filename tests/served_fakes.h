// What api.cu and served.cu call of the CUDA runtime and of the other sources,
// faked for tests on the host: calls succeed, except those a test makes fail.
#pragma once
#include <stdio.h>
#include <stdlib.h>

#include <functional>

#include "pipeline.cuh"
#include "stream.cuh"

static int g_fail_pool = 0;  // the next so many pools cannot be made
static int g_fail_host = 0;  // 1: the next pinned allocation fails, 2: the one after it, ...
static std::function<void(cso_ctx*)> g_pipeline = [](cso_ctx*) {};

static void* fake() { return malloc(1); }
extern "C" {
cudaError_t cudaGetDeviceCount(int* n) { return *n = 1, cudaSuccess; }
cudaError_t cudaGetDevice(int* d) { return *d = 0, cudaSuccess; }
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) { return *v = 152, cudaSuccess; }
const char* cudaGetErrorString(cudaError_t) { return "made to fail"; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) { return *s = (cudaStream_t)fake(), cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t s) { return free((void*)s), cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t* e) { return *e = (cudaEvent_t)fake(), cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { return *e = (cudaEvent_t)fake(), cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t e) { return free((void*)e), cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
cudaError_t cudaMalloc(void** p, size_t) { return *p = fake(), cudaSuccess; }
cudaError_t cudaFree(void* p) { return free(p), cudaSuccess; }
cudaError_t cudaMallocHost(void** p, size_t n) {
  if (g_fail_host && --g_fail_host == 0) return cudaErrorMemoryAllocation;
  return *p = malloc(n), cudaSuccess;
}
cudaError_t cudaFreeHost(void* p) { return free(p), cudaSuccess; }
cudaError_t cudaMemPoolCreate(cudaMemPool_t* p, const cudaMemPoolProps*) {
  if (g_fail_pool && g_fail_pool--) return cudaErrorMemoryAllocation;
  return *p = (cudaMemPool_t)fake(), cudaSuccess;
}
cudaError_t cudaMemPoolDestroy(cudaMemPool_t p) { return free((void*)p), cudaSuccess; }
cudaError_t cudaMemPoolSetAttribute(cudaMemPool_t, cudaMemPoolAttr, void*) { return cudaSuccess; }
cudaError_t cudaMemPoolGetAttribute(cudaMemPool_t, cudaMemPoolAttr, void* v) { return *(uint64_t*)v = 0, cudaSuccess; }
cudaError_t cudaMemPoolTrimTo(cudaMemPool_t, size_t) { return cudaSuccess; }
}
int cells_choose(long long, int* nc) { return *nc = 160, CSO_OK; }
int cells_check_dense(int) { return CSO_OK; }
int pipeline_run(cso_ctx* c, const cso_input*, const cso_params*, cso_output*) { return g_pipeline(c), CSO_OK; }
int stream_begin(StreamState**, uint64_t, const cso_params*, cudaMemPool_t) { return CSO_ERR_STATE; }
int stream_step(cso_ctx*, StreamState&, const cso_input*, cso_output*, ServedRequest*) { return CSO_ERR_STATE; }
void stream_release(StreamState*, cudaStream_t) {}

#define CHECK(x)                                                          \
  do {                                                                    \
    if (!(x)) return fprintf(stderr, "line %d: %s\n", __LINE__, #x), 1;    \
  } while (0)
