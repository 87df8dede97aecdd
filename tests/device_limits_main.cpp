// The launch functions of the kernels that take more shared memory than a
// device allows by default, linked against a stand-in for the CUDA runtime with
// two devices.  The stand-in keeps a kernel's limit per device, as CUDA does, and
// refuses a launch beyond it.  Prints one line per launch: name, device, status.
#include <cstdio>
#include <cstring>
#include <map>
#include <utility>

#include "../paper_2512_12094_gb300/csrc/pp_internal.h"

namespace {
int device = 0;
int refuse = 0;  // attribute calls still to be refused
std::map<std::pair<int, const void*>, size_t> limit;
cudaError_t last = cudaSuccess;
dim3 grid_, block_;
size_t smem_;
cudaStream_t stream_;

cudaError_t launched(const void* f, size_t smem) {
  const auto it = limit.find({device, f});
  const size_t allowed = it == limit.end() ? 48 * 1024 : it->second;
  return last = smem > allowed ? cudaErrorInvalidValue : cudaSuccess;
}
}  // namespace

extern "C" {
void** __cudaRegisterFatBinary(void*) { static void* h; return &h; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char*, char*, const char*, int, uint3*, uint3*, dim3*, dim3*,
                            int*) {}
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t smem, cudaStream_t s) {
  grid_ = g, block_ = b, smem_ = smem, stream_ = s;
  return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3* g, dim3* b, size_t* smem, void* s) {
  *g = grid_, *b = block_, *smem = smem_;
  memcpy(s, &stream_, sizeof(stream_));
  return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* f) {
  *k = (cudaKernel_t)f;
  return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3, dim3, void**, size_t smem, cudaStream_t) {
  return launched(k, smem);
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* f, void**) {
  return launched(f, c->dynamicSmemBytes);
}
cudaError_t cudaFuncSetAttribute(const void* f, cudaFuncAttribute, int v) {
  if (refuse > 0) {
    --refuse;
    return last = cudaErrorUnknown;
  }
  limit[{device, f}] = (size_t)v;
  return cudaSuccess;
}
cudaError_t cudaGetDevice(int* d) {
  *d = device;
  return cudaSuccess;
}
cudaError_t cudaSetDevice(int d) {
  device = d;
  return cudaSuccess;
}
cudaError_t cudaGetLastError() {
  const cudaError_t e = last;
  last = cudaSuccess;
  return e;
}
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) {
  *v = 152;
  return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void*, int, size_t,
                                                                   unsigned) {
  *n = 1;
  return cudaSuccess;
}
}

using namespace ppk;

int main(int argc, char** argv) {
  // devices to launch on, in order; "x" before one: its first attribute call is refused
  for (int a = 1; a < argc; ++a) {
    refuse = argv[a][0] == 'x';
    cudaSetDevice(argv[a][refuse] - '0');
    auto say = [](const char* name, int i, cudaError_t e) { printf("%s%d %d %d\n", name, i, device, (int)e); };
    DevTable t = {};
    PhaseAcc acc = {};
    PhaseBuckets b = {};
    PhaseRule rule = {};
    PhaseDesc d = {}, last_phase = {};
    d.count = 1;
    for (int P : {1, 2, 4, 6, 8})
      say("phase", P, launch_phase(P, 12, nullptr, b, b, d, last_phase, nullptr, rule, t, nullptr, acc));
    d.dense = 1;
    for (int P : {1, 2}) {
      say("dense", P, launch_phase(P, 12, nullptr, b, b, d, last_phase, nullptr, rule, t, nullptr, acc));
      for (int f32 = 0; f32 < 2; ++f32) {
        t.B = 256;
        t.f32 = f32;
        const RowsLaunch L = rows_launch(P, t.B, f32 ? 4 : 8, 152);
        say(f32 ? "rows32_" : "rows64_", P,
            launch_rows_phase(P, L, nullptr, b, b, d, last_phase, nullptr, rule, nullptr, nullptr, 1,
                              nullptr, nullptr, t, nullptr, acc));
      }
    }
    MergeBuckets m = {};
    m.nb = 1;
    m.cg = 8;
    for (int n : {32, 64, 128, 192, 256})
      for (int group : {0, 1, 3, 4 | (8 << 8)})
        say("merge", n * 10 + (group & 0xFF),
            launch_merge_buckets(m, n, group, nullptr, t, 1, nullptr, 0, 0.0, t, nullptr, 152, 0));
    for (int W : {1, 2}) say("layer1024_", W, launch_layer(W, 1024, 1, nullptr, nullptr, nullptr, nullptr, 1));
    for (int W : {1, 2, 3, 4}) say("layer256_", W, launch_layer(W, 256, 1, nullptr, nullptr, nullptr, nullptr, 1));
  }
  return 0;
}
