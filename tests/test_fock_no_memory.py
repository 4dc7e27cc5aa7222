"""A Fock plan whose convolution finds no room on the device is built on the node walk: the plan's host code compiled on
the CPU against a stand-in for the CUDA runtime whose largest allocation fails."""
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2412_17742_gb300", "csrc")

MAIN = '''
#include <algorithm>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <vector>
#include "gbsbin_fock_conv.h"

static size_t largest = 0, refuse_from = ~(size_t)0;
static int refused = 0, walks = 0, convs = 0, live = 0, calls = 0;

extern "C" {
cudaError_t cudaMalloc(void** p, size_t n) {
  ++calls;
  largest = std::max(largest, n);
  if (n >= refuse_from) {
    ++refused;
    *p = nullptr;
    return cudaErrorMemoryAllocation;
  }
  *p = std::calloc(1, n ? n : 1);
  ++live;
  return cudaSuccess;
}
cudaError_t cudaFree(void* p) { if (p) --live; std::free(p); return cudaSuccess; }
cudaError_t cudaHostAlloc(void** p, size_t n, unsigned) { *p = std::calloc(1, n); return cudaSuccess; }
cudaError_t cudaMallocHost(void** p, size_t n) { return cudaHostAlloc(p, n, 0); }
cudaError_t cudaFreeHost(void* p) { std::free(p); return cudaSuccess; }
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind) { ++calls; std::memcpy(d, s, n); return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t) { std::memcpy(d, s, n); return cudaSuccess; }
cudaError_t cudaMemset(void* d, int v, size_t n) { std::memset(d, v, n); return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaGetDevice(int* d) { *d = 0; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) { *v = 152; return cudaSuccess; }
cudaError_t cudaDeviceSynchronize() { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t*) { return cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) { *ms = 0; return cudaSuccess; }
void gbsbin_default_options(gbsbin_options* o) {
  std::memset(o, 0, sizeof(*o));
  o->oversample = 1;
  o->want_diagnostics = 1;
}
}
namespace gbsbin {
int fock_points_per_thread(bool, long long) { return 1; }
size_t fock_smem_bytes(int, int, int) { return 1024; }
int fock_ctas_per_sm(bool, int, size_t) { return 4; }
cudaError_t launch_fock(const FockArgs& a, bool, int, cudaStream_t) {
  ++walks;
  return a.coef && a.xtw && a.zr && a.parts ? cudaSuccess : cudaErrorInvalidValue;
}
cudaError_t launch_dft_fused(const DftArgs& a, unsigned* bar, int, cudaStream_t) {
  return a.parts && a.tw && a.bufA && a.bufB && bar ? cudaSuccess : cudaErrorInvalidValue;
}
int fock_conv_slots_per_sm(int) { return 5; }
size_t fock_conv_layer_smem(int, int, int) { return 1024; }
cudaError_t launch_fock_conv(const FockConvArgs& a, const FockConvLayer*, int, int, cudaStream_t, int* n) {
  ++convs;
  *n = 3;
  return a.B && a.parts && a.F[0][0] ? cudaSuccess : cudaErrorInvalidValue;
}
}  // namespace gbsbin

int main() {
  constexpr int M = 12, L = 3;
  std::vector<gbsbin_complex> T(M * M);
  for (int i = 0; i < M; ++i) T[i * M + i].re = 0.9;
  std::vector<int> photons(M, 1), bin(M), cut(L, M);
  for (int i = 0; i < M; ++i) bin[i] = i % L;
  gbsbin_fock_problem p{};
  p.M = M;
  p.T = T.data();
  p.photons = photons.data();
  p.bin_of_mode = bin.data();
  p.L = L;
  p.cutoff = cut.data();
  std::vector<double> P(13 * 13 * 13);
  for (int pass = 0; pass < 2; ++pass) {       // with room for everything, then none for the largest block
    gbsbin_fock_plan* h = nullptr;
    walks = convs = refused = calls = 0;
    const int st = gbsbin_fock_plan_create(&p, nullptr, &h);
    const int made = calls;
    const int ex = st ? -1 : gbsbin_fock_execute(h, P.data(), nullptr);
    const int tr = st ? -1 : gbsbin_fock_plan_set_transfer(h, T.data(), nullptr);
    if (h) gbsbin_fock_plan_destroy(h);
    std::printf("%d %d %d %d %d %d %d %d\\n", st, ex, tr, convs, walks, refused, live, made);
    refuse_from = largest;
  }
}
'''


@pytest.fixture(scope="module")
def passes(tmp_path_factory):
    d = tmp_path_factory.mktemp("fock")
    (d / "main.cpp").write_text(MAIN)
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    exe = str(d / "main")
    subprocess.run(["g++", "-O1", "-std=c++17", str(d / "main.cpp"), os.path.join(CSRC, "gbsbin_fock_host.cpp"), "-I", CSRC,
                    "-I", os.path.join(cuda, "include"), "-o", exe], check=True)
    out = subprocess.run([exe], capture_output=True, text=True, check=True).stdout
    return [[int(v) for v in line.split()] for line in out.splitlines()]


def test_convolution_with_room(passes):
    assert passes[0][:7] == [0, 0, 0, 1, 0, 0, 0]


def test_convolution_makes_its_own_arrays_only(passes):
    # one block; one copy of its tables, one of the circuit
    assert passes[0][7] == 3


def test_walk_without_room(passes):
    st, execute, transfer, convs, walks, refused, live, _ = passes[1]
    assert refused == 1 and (st, execute, transfer, convs, walks, live) == (0, 0, 0, 0, 1, 0)
