"""The server's pinned buffers against copies still in flight, on the CPU: csrc/server.cu is linked
against a stand-in for the CUDA runtime that makes an asynchronous copy at the wait that follows it
and compares the source then with what it was when the copy was enqueued."""
import os
import subprocess

from paper_1208_1157_gb300 import build as B

FAKE = r"""
#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <vector>
#include "swarm.h"
struct Copy { void *dst; const void *src, *stream; std::vector<char> then; };
static std::vector<Copy> flying;
static size_t fail_bytes = 0;  // the next device allocation of this size fails
static int races = 0;
extern "C" {
int cudaMalloc(void **p, size_t n) {
  if (n == fail_bytes) { fail_bytes = 0; return 2; }
  *p = calloc(1, n);
  return 0;
}
int cudaFree(void *p) { free(p); return 0; }
int cudaHostAlloc(void **p, size_t n, unsigned) { *p = calloc(1, n); return 0; }
int cudaMallocHost(void **p, size_t n) { *p = calloc(1, n); return 0; }
int cudaFreeHost(void *p) { free(p); return 0; }
int cudaMemcpyAsync(void *d, const void *s, size_t n, int, void *st) {
  flying.push_back({d, s, st, std::vector<char>((const char *)s, (const char *)s + n)});
  return 0;
}
int cudaMemsetAsync(void *p, int v, size_t n, void *) { memset(p, v, n); return 0; }
int cudaStreamSynchronize(void *st) {
  for (size_t i = 0; i < flying.size();) {
    Copy &c = flying[i];
    if (c.stream != st) { i++; continue; }
    races += memcmp(c.src, c.then.data(), c.then.size()) != 0;
    memcpy(c.dst, c.src, c.then.size());
    flying.erase(flying.begin() + i);
  }
  return 0;
}
int cudaDeviceSynchronize() { return 0; }
int cudaStreamCreateWithFlags(void **p, unsigned) { *p = malloc(1); return 0; }
int cudaStreamDestroy(void *p) { free(p); return 0; }
int cudaStreamWaitEvent(void *, void *, unsigned) { return 0; }
int cudaEventCreate(void **p) { *p = malloc(1); return 0; }
int cudaEventCreateWithFlags(void **p, unsigned) { *p = malloc(1); return 0; }
int cudaEventDestroy(void *p) { free(p); return 0; }
int cudaEventRecord(void *, void *) { return 0; }
int cudaEventElapsedTime(float *f, void *, void *) { *f = 0; return 0; }
int cudaGetDevice(int *d) { *d = 0; return 0; }
int cudaDeviceGetAttribute(int *v, int, int) { *v = 4; return 0; }
int cudaGetLastError() { return 0; }
const char *cudaGetErrorString(int) { return "error"; }
// kernels are not run
int __cudaPushCallConfiguration() { return 0; }
int __cudaPopCallConfiguration() { return 0; }
int __cudaGetKernel() { return 0; }
int __cudaLaunchKernel() { return 0; }
int cudaLaunchKernel() { return 0; }
void **__cudaRegisterFatBinary() { static void *h; return &h; }
void __cudaRegisterFatBinaryEnd() {}
void __cudaUnregisterFatBinary() {}
void __cudaRegisterFunction() {}
char __cudaInitModule() { return 0; }
}
namespace swarm {
struct BinView;
struct StepParams;
void set_last_error(const char *) {}
}
struct CUstream_st;
extern "C" int one_block(int *blocks) { if (blocks) *blocks = 1; return 0; }
int main() {
  swarm_server_config cfg = {};
  cfg.slots_per_pool = 64;
  cfg.quantum_steps = 10;
  cfg.hermite_dt = cfg.mvs_dt = 0.01;
  swarm_server *sv = nullptr;
  if (swarm_server_create(&cfg, nullptr, &sv)) return 2;
  const double mass[3] = {1, 1e-3, 1e-3}, a[9] = {0, 0, 0, 1, 0, 0, 2, 0, 0}, b[9] = {0, 0, 0, 0, 3, 0, 0, 5, 0};
  int64_t id;
  int32_t done;
  if (swarm_server_submit(sv, 1, 3, mass, a, a, 0, 1, SWARM_HERMITE4, &id)) return 3;
  fail_bytes = 64 * sizeof(int32_t);  // the list of the round's slots
  if (swarm_server_step(sv, &done) == SWARM_OK || fail_bytes) return 4;
  if (swarm_server_submit(sv, 1, 3, mass, b, b, 0, 1, SWARM_HERMITE4, &id)) return 5;
  if (swarm_server_step(sv, &done) != SWARM_OK) return 6;
  swarm_server_destroy(sv);
  printf("races %d left %zu\n", races, flying.size());
  return races != 0;
}
"""
# the launchers, with the library's own types
LAUNCH = r"""
#include "kernels.h"
extern "C" int one_block(int *blocks);
namespace swarm {
cudaError_t launch_hermite_uniform(int, const BinView &, int, const StepParams &, int, cudaStream_t, int *b) { return (cudaError_t)one_block(b); }
cudaError_t launch_mvs_uniform(bool, const BinView &, int, const StepParams &, int, cudaStream_t, int *b) { return (cudaError_t)one_block(b); }
}
"""


def test_a_round_that_fails_leaves_no_copy_behind(tmp_path):
    csrc = os.path.join(os.path.dirname(os.path.abspath(B.__file__)), "csrc")
    (tmp_path / "fake.cpp").write_text(FAKE)
    (tmp_path / "launch.cu").write_text(LAUNCH)
    nvcc = [B.nvcc()] + B.ARCH + ["-std=c++17", "-I", csrc, "-I", B.INCLUDE, "-c"]
    for src, obj in ((os.path.join(csrc, "server.cu"), "server.o"), (str(tmp_path / "launch.cu"), "launch.o")):
        subprocess.run(nvcc + [src, "-o", str(tmp_path / obj)], check=True)
    subprocess.run(["g++", "-std=c++17", "-I", B.INCLUDE, "-o", str(tmp_path / "t"), str(tmp_path / "fake.cpp"),
                    str(tmp_path / "server.o"), str(tmp_path / "launch.o")], check=True)
    r = subprocess.run([str(tmp_path / "t")], capture_output=True, text=True)
    assert r.returncode == 0, (r.returncode, r.stdout)
