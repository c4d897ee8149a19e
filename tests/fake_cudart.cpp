// A stand-in for the CUDA runtime, linked with libmw's objects into a library whose
// host code runs without a GPU: it keeps the current device, what each device was
// told about a kernel's shared memory, and a list of the launches, and refuses a
// launch that asks for more dynamic shared memory than its device has granted (48 KB
// without the attribute), as the runtime does.  Two devices of 152 SMs.
#include <cuda.h>
#include <cuda_runtime.h>

#include <cstdio>
#include <cstring>
#include <map>
#include <string>
#include <utility>
#include <vector>

namespace {

int g_device = 0;
cudaError_t g_last = cudaSuccess;
std::map<const void *, std::string> &names() {
  static std::map<const void *, std::string> n;
  return n;
}
std::map<std::pair<int, const void *>, int> g_granted;
struct Launch {
  int device;
  std::string name;
  unsigned grid, block;
  size_t smem;
  cudaStream_t stream;
};
std::vector<Launch> g_launches;
struct Config {
  dim3 grid, block;
  size_t smem;
  cudaStream_t stream;
};
std::vector<Config> g_config;
uintptr_t g_next_handle = 0x1000;
alignas(256) char g_symbol[256];

CUresult encode_tiled(CUtensorMap *map, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                      const cuuint64_t *, const cuuint32_t *, const cuuint32_t *,
                      CUtensorMapInterleave, CUtensorMapSwizzle, CUtensorMapL2promotion,
                      CUtensorMapFloatOOBfill) {
  memset(map, 0, sizeof *map);
  return CUDA_SUCCESS;
}

}  // namespace

extern "C" {

// ---- for the tests -------------------------------------------------------------
void fake_set_device(int dev) { g_device = dev; }
void fake_clear(void) { g_launches.clear(); }
int fake_launches(void) { return (int)g_launches.size(); }
// "device name grid block shared-memory stream" of launch i
const char *fake_launch(int i) {
  static std::string s;
  const Launch &l = g_launches.at(i);
  char b[128];
  snprintf(b, sizeof b, " %u %u %zu %zu", l.grid, l.block, l.smem, (size_t)l.stream);
  s = std::to_string(l.device) + " " + l.name + b;
  return s.c_str();
}

// ---- registration and launches ---------------------------------------------------
void **__cudaRegisterFatBinary(void *) {
  static void *handle[1];
  return handle;
}
void __cudaRegisterFatBinaryEnd(void **) {}
void __cudaUnregisterFatBinary(void **) {}
void __cudaRegisterFunction(void **, const char *host, char *, const char *name, int, uint3 *,
                            uint3 *, dim3 *, dim3 *, int *) {
  names()[host] = name;
}
void __cudaRegisterVar(void **, char *, char *, const char *, int, size_t, int, int) {}
unsigned __cudaPushCallConfiguration(dim3 grid, dim3 block, size_t smem, CUstream_st *stream) {
  g_config.push_back({grid, block, smem, stream});
  return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3 *grid, dim3 *block, size_t *smem, void *stream) {
  const Config c = g_config.back();
  g_config.pop_back();
  *grid = c.grid;
  *block = c.block;
  *smem = c.smem;
  *static_cast<cudaStream_t *>(stream) = c.stream;
  return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t *k, const void *host) {
  *k = reinterpret_cast<cudaKernel_t>(const_cast<void *>(host));
  return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3 grid, dim3 block, void **, size_t smem,
                               cudaStream_t stream) {
  const void *f = k;
  const auto it = g_granted.find({g_device, f});
  if (smem > (size_t)(it == g_granted.end() ? 49152 : it->second)) return g_last = cudaErrorInvalidValue;
  g_launches.push_back({g_device, names()[f], grid.x * grid.y * grid.z, block.x * block.y * block.z,
                        smem, stream});
  return cudaSuccess;
}
cudaError_t cudaFuncSetAttribute(const void *f, cudaFuncAttribute attr, int value) {
  if (attr == cudaFuncAttributeMaxDynamicSharedMemorySize) g_granted[{g_device, f}] = value;
  return cudaSuccess;
}
cudaError_t cudaFuncGetAttributes(cudaFuncAttributes *a, const void *) {
  memset(a, 0, sizeof *a);
  a->numRegs = 64;
  return cudaSuccess;
}

// ---- device, streams, copies -----------------------------------------------------
cudaError_t cudaGetDevice(int *dev) {
  *dev = g_device;
  return cudaSuccess;
}
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr attr, int) {
  *v = attr == cudaDevAttrMultiProcessorCount ? 152 : 233472;
  return cudaSuccess;
}
cudaError_t cudaGetLastError(void) {
  const cudaError_t e = g_last;
  g_last = cudaSuccess;
  return e;
}
const char *cudaGetErrorString(cudaError_t e) { return e == cudaSuccess ? "no error" : "invalid argument"; }
cudaError_t cudaGetSymbolAddress(void **p, const void *) {
  *p = g_symbol;
  return cudaSuccess;
}
cudaError_t cudaDeviceSynchronize(void) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned) {
  *s = reinterpret_cast<cudaStream_t>(g_next_handle += 16);
  return cudaSuccess;
}
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus *c) {
  *c = cudaStreamCaptureStatusNone;
  return cudaSuccess;
}
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned) {
  *e = reinterpret_cast<cudaEvent_t>(g_next_handle += 16);
  return cudaSuccess;
}
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaMemset(void *, int, size_t) { return cudaSuccess; }
cudaError_t cudaMemsetAsync(void *, int, size_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaMemcpy(void *dst, const void *, size_t n, cudaMemcpyKind kind) {
  if (kind == cudaMemcpyDeviceToHost) memset(dst, 0, n);
  return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void *dst, const void *src, size_t n, cudaMemcpyKind kind, cudaStream_t) {
  return cudaMemcpy(dst, src, n, kind);
}
cudaError_t cudaGetDriverEntryPointByVersion(const char *, void **p, unsigned, unsigned long long,
                                             cudaDriverEntryPointQueryResult *q) {
  *p = reinterpret_cast<void *>(encode_tiled);
  *q = cudaDriverEntryPointSuccess;
  return cudaSuccess;
}

}  // extern "C"
