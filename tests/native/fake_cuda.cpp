// A CUDA runtime on host memory (test infrastructure): linked in place of cudart with the library's
// own objects, it runs the whole host path -- plans, dispatch rules, launch set-up -- without a GPU.
// Device memory is host memory, kernels do not run, and every launch is recorded with its kernel's
// name, its grid and the table it would read: a strided pass's column blocks, a contiguous one's
// stage table.
#include <cuda.h>
#include <cxxabi.h>

#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <map>
#include <new>
#include <string>

#include "tfft_internal.h"

namespace {
// by host entry point; filled by the objects' own static constructors
std::map<const void*, std::string>& kernels() {
  static std::map<const void*, std::string> m;
  return m;
}
std::string g_log;

std::string demangled(const char* name) {
  int st = 0;
  char* d = abi::__cxa_demangle(name, nullptr, nullptr, &st);
  std::string s = st == 0 && d ? d : name;
  std::free(d);
  return s;
}

bool g_graphs = false, g_capturing = false;  // captures refused, unless asked for
int g_fail = 0;                              // launches until one runs out of host memory

cudaError_t record(const void* func, dim3 grid, dim3 block, void** args) {
  if (g_fail > 0 && --g_fail == 0) throw std::bad_alloc();
  const std::string& name = kernels()[func];
  char line[256];
  unsigned long long cb = 0;
  long long ncb = -1, merged = 0;
  if (name.find("strided") != std::string::npos) {
    const auto& a = *static_cast<const tfft::StridedArgs*>(args[0]);
    cb = reinterpret_cast<unsigned long long>(a.colblocks);
    ncb = a.ncolblocks;
    merged = a.merged_blocks;
  } else if (name.find("k_contig_spec") != std::string::npos) {
    cb = reinterpret_cast<unsigned long long>(static_cast<const tfft::ContigArgs*>(args[0])->tws);
  }
  std::snprintf(line, sizeof line, "%u|%u|%u|%llu|%lld|%lld|", grid.x, grid.y, block.x * block.y, cb, ncb, merged);
  g_log += line + name + "\n";
  return cudaSuccess;
}

CUresult encode(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle, CUtensorMapL2promotion,
                CUtensorMapFloatOOBfill) {
  return CUDA_SUCCESS;
}
struct {
  dim3 grid, block;
} g_call;
int g_token;
}  // namespace

extern "C" {
// The launches since the last call, one per line: grid x|grid y|threads|table|column blocks|merged blocks|kernel.
int fake_launches(char* out, int n) {
  const int len = (int)g_log.size();
  if (len < n) std::memcpy(out, g_log.c_str(), len + 1);
  g_log.clear();
  return len;
}

void fake_graphs(int on) { g_graphs = on != 0; }
int fake_capturing() { return g_capturing; }
void fake_fail_launch(int n) { g_fail = n; }

void** __cudaRegisterFatBinary(void*) { return reinterpret_cast<void**>(&g_token); }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
void __cudaRegisterFunction(void**, const char* host, char*, const char* name, int, uint3*, uint3*, dim3*, dim3*, int*) {
  kernels()[host] = demangled(name);
}
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t, void*) {
  g_call = {g, b};
  return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3* g, dim3* b, size_t* s, void* st) {
  *g = g_call.grid;
  *b = g_call.block;
  *s = 0;
  *static_cast<void**>(st) = nullptr;
  return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* f) {
  *k = reinterpret_cast<cudaKernel_t>(const_cast<void*>(f));
  return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3 g, dim3 b, void** args, size_t, cudaStream_t) {
  return record(k, g, b, args);
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* f, void** args) {
  return record(f, c->gridDim, c->blockDim, args);
}
cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void*, int, size_t, unsigned) {
  *n = 2;
  return cudaSuccess;
}
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) {
  *v = 152;
  return cudaSuccess;
}
cudaError_t cudaGetDevice(int* d) {
  *d = 0;
  return cudaSuccess;
}
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
const char* cudaGetErrorString(cudaError_t) { return "fake"; }
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t) {
  std::memcpy(d, s, n);
  return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void* d, int v, size_t n, cudaStream_t) {
  std::memset(d, v, n);
  return cudaSuccess;
}
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) {
  *s = reinterpret_cast<cudaStream_t>(&g_token);
  return cudaSuccess;
}
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus* s) {
  // a caller's capture: launches go directly, not through the graph cache
  *s = g_graphs ? cudaStreamCaptureStatusNone : cudaStreamCaptureStatusActive;
  return cudaSuccess;
}
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) {
  if (g_capturing) return cudaErrorIllegalState;
  g_capturing = true;
  return cudaSuccess;
}
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t* g) {
  *g = g_capturing ? reinterpret_cast<cudaGraph_t>(&g_token) : nullptr;
  g_capturing = false;
  return cudaSuccess;
}
cudaError_t cudaGraphInstantiate(cudaGraphExec_t* x, cudaGraph_t, unsigned long long) {
  *x = reinterpret_cast<cudaGraphExec_t>(&g_token);
  return cudaSuccess;
}
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) {
  g_log += "0|0|0|0|-1|0|graph\n";
  return cudaSuccess;
}
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t*) { return cudaErrorNotSupported; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t*, unsigned) { return cudaErrorNotSupported; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float*, cudaEvent_t, cudaEvent_t) { return cudaErrorNotSupported; }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes*, const void*) { return cudaErrorNotSupported; }
cudaError_t cudaGetSymbolAddress(void**, const void*) { return cudaErrorNotSupported; }
cudaError_t cudaGetDriverEntryPointByVersion(const char*, void** f, unsigned, unsigned long long,
                                             cudaDriverEntryPointQueryResult* q) {
  *f = reinterpret_cast<void*>(&encode);
  *q = cudaDriverEntryPointSuccess;
  return cudaSuccess;
}
}
