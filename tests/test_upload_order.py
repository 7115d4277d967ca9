"""Host tables reach the device before anything that reads them is launched: a
plain cudaMemcpy from pageable memory may return before its last bytes have
landed and orders nothing on a non-blocking stream, so tables go up on the stream
that uses them, which is then synchronised.

The host code runs here on a stand-in for the CUDA runtime that takes every
freedom the real one has: work queued on a stream is done when that stream is
synchronised or launches a kernel, and staged copies of the legacy stream land
only when that one is."""
import glob
import os
import platform
import re
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2606_06247_gb300", "csrc")

FAKE = r"""
#include <cstdlib>
#include <cstring>
#include <functional>
#include <map>
#include <vector>
#include "fcsph_internal.h"
using namespace fcsph;

static std::map<cudaStream_t, std::vector<std::function<void()>>> queued;
static void flush(cudaStream_t st) {
  for (auto& f : queued[st]) f();
  queued[st].clear();
}
static int late = 0;  // launches with a table of another stream still on its way
static void launched(cudaStream_t st) {
  flush(st);
  if (!queued[nullptr].empty()) ++late;
}
static cudaError_t copy(void* d, const void* s, size_t n, cudaMemcpyKind k, cudaStream_t st) {
  if (k != cudaMemcpyHostToDevice) {
    flush(st);
    memcpy(d, s, n);
    return cudaSuccess;
  }
  std::vector<char> stage((const char*)s, (const char*)s + n);
  queued[st].push_back([=] { memcpy(d, stage.data(), n); });
  return cudaSuccess;
}
extern "C" {
cudaError_t cudaMalloc(void** p, size_t n) { return (*p = calloc(1, n)) ? cudaSuccess : cudaErrorMemoryAllocation; }
cudaError_t cudaFree(void* p) {  // waits for the device
  for (auto& q : queued) flush(q.first);
  free(p);
  return cudaSuccess;
}
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind k) { return copy(d, s, n, k, nullptr); }
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind k, cudaStream_t st) { return copy(d, s, n, k, st); }
cudaError_t cudaMemset(void* d, int v, size_t n) { queued[nullptr].push_back([=] { memset(d, v, n); }); return cudaSuccess; }
cudaError_t cudaMemsetAsync(void* d, int v, size_t n, cudaStream_t st) { queued[st].push_back([=] { memset(d, v, n); }); return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t st) { flush(st); return cudaSuccess; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) { *s = (cudaStream_t)16; return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
const char* cudaGetErrorString(cudaError_t) { return ""; }
}
cudaError_t init_kernel_attributes() { return cudaSuccess; }
int col_r_split(const fcsph_ctx*) { return 0; }
int col_rb_split(const fcsph_ctx*) { return 0; }
int row_w_m(const fcsph_ctx*) { return 0; }
size_t mean_scratch(const fcsph_ctx*) { return 0; }
void persist_destroy(PersistPlan*) {}
cudaError_t launch_dft_lines(int, int, int, int, const void*, void*, cudaStream_t st, const FftPlan&, const void*) {
  launched(st);
  return cudaSuccess;
}
cudaError_t launch_dft_ip(int, int, int, int, const void*, void*, cudaStream_t st, const FftPlan&, const IpPlan&, const void*) {
  launched(st);
  return cudaSuccess;
}
extern "C" int run(int* late_out) {
  cudaStream_t st = (cudaStream_t)32;  // a non-blocking stream
  double io[2] = {};
  for (int prec : {FCSPH_F64, FCSPH_F32, FCSPH_F32X2})
    for (int n : {12, 89, 179})  // direct, Rader, chirp-z
      if (fcsph_dft(n, 1, -1, prec, io, io, st) != FCSPH_OK) return 2;
  const int dft_late = late;
  for (int prec : {FCSPH_F64, FCSPH_F32, FCSPH_F32X2}) {
    fcsph_grid g = {16, 16, 1.0, 1.0, 0, 1, 1, 0.0};
    fcsph_fc fc = {FCSPH_FC_GRAM, 5, 25, 0};
    fcsph_kernel k = {FCSPH_G4, 1.3};
    fcsph_precision p = {(decltype(p.fft_prec))prec, 0};
    fcsph_ctx* c = nullptr;
    if (fcsph_create(&g, &fc, &k, &p, nullptr, nullptr, st, &c) != FCSPH_OK) return 3;
    launched(st);  // the context's first pass
    fcsph_destroy(c);
  }
  late_out[0] = dft_late;
  late_out[1] = late - dft_late;
  return 0;
}
"""


@pytest.mark.skipif(not os.path.isdir("/usr/local/cuda/include"), reason="no CUDA headers")
def test_tables_land_before_the_launch(tmp_path):
    src, lib = tmp_path / "fake.cpp", tmp_path / "libfake.so"
    src.write_text(FAKE)
    # a library, so that the launchers this path does not reach may stay undefined
    cmd = ["g++", "-O1", "-std=gnu++17", "-fPIC", "-shared", "-Wl,-Bsymbolic", "-Wl,-z,lazy", "-I" + CSRC,
           "-I" + os.path.join(ROOT, "include"), "-I/usr/local/cuda/include", str(src), os.path.join(CSRC, "fcsph_api.cpp"),
           os.path.join(CSRC, "fcsph_tables.cpp"), "-o", str(lib), "-ldl"]
    if platform.machine() == "x86_64":
        cmd.append("-lquadmath")
    subprocess.run(cmd, check=True, capture_output=True, text=True)
    code = "import ctypes, os, sys; n = (ctypes.c_int * 2)(); f = ctypes.CDLL(sys.argv[1], os.RTLD_LAZY).run; print(f(n), *n)"
    r = subprocess.run([sys.executable, "-c", code, str(lib)], capture_output=True, text=True, timeout=120)
    # status, and launches of (fcsph_dft, a new context) before their tables had landed
    assert r.stdout.split() == ["0", "0", "0"], (r.stdout, r.stderr)


def test_no_unordered_table_copies():
    """Also in the persistent plan's work list, whose launcher needs the kernels."""
    for path in glob.glob(os.path.join(CSRC, "*.c*")):
        text = open(path).read()
        for call in re.findall(r"cudaMem(?:cpy|set)\([^;]*;", text):
            assert "DeviceToHost" in call.split(";")[0].split("||")[0], (os.path.basename(path), call)
