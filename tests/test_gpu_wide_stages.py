"""FP64 stages by pairs of outputs (small launches) and by whole butterflies do the
same operations, whichever products the compiler would fuse: the engine's stages
compiled with and without fused multiply-adds give the same bits in both forms."""
import os
import platform
import shutil
import subprocess

import pytest

from gpu_common import torch_cuda

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2606_06247_gb300", "csrc")

SOURCE = r"""
#include <cstdio>
#include <cstring>
#include "fcsph_ip.cuh"
using namespace fcsph;

__global__ void __launch_bounds__(128) k(const __grid_constant__ IpPlan P, const double2* in, double2* out,
                                         const double2* pool, int nl, int ls) {
  extern __shared__ double2 lines[];
  for (int t = threadIdx.x; t < nl * P.n; t += blockDim.x)
    lines[(t / P.n) * ls + in_slot<double>(P, t % P.n)] = in[t];
  __syncthreads();
  fft_ip<double, 17>(lines, nl, ls, P, pool, lines);
  for (int t = threadIdx.x; t < nl * P.n; t += blockDim.x)
    out[t] = lines[(t / P.n) * ls + out_slot<double>(P, t % P.n)];
}

int main() {
  // every butterfly (8, 4, 2, 3, 5, 7, 9, 11, 13, 17), their products, Rader (89 = 1 + 8 11, 281 = 1 + 8 5 7)
  // and chirp-z (94 = 2 47)
  const int lens[] = {8, 16, 32, 64, 6, 15, 63, 72, 66, 78, 136, 96, 89, 281, 94};
  unsigned long long s = 88172645463325252ull, hash = 14695981039346656037ull;
  auto rnd = [&] { s ^= s << 13; s ^= s >> 7; s ^= s << 17; return (double)(s >> 11) / 9007199254740992.0 - 0.5; };
  int bad = 0;
  for (int n : lens) {
    Pool pool;
    std::vector<double> br, bi;
    const FftPlan F = make_plan(n, &pool, &br, &bi);
    if (F.rd || F.bs)  // any filter will do
      for (int j = 0; j < F.sub.n; ++j) pool.re[F.bhat + j] = rnd(), pool.im[F.bhat + j] = rnd();
    std::vector<int> tab;
    IpPlan P = make_ip(F, pool, &tab);
    const int ls = ip_ls<double>(P), nl = 2, np = (int)pool.re.size();
    if (P.big || (size_t)nl * ls * sizeof(double2) > 48 * 1024) return 2;
    std::vector<double2> hp(np), x(nl * n), y[2];
    for (int j = 0; j < np; ++j) hp[j] = make_double2(pool.re[j], pool.im[j]);
    for (auto& v : x) v = make_double2(rnd(), rnd());
    double2 *dp, *dx, *dy;
    int* dt;
    tab.push_back(0);
    if (cudaMalloc(&dp, np * 16) || cudaMalloc(&dx, nl * n * 16) || cudaMalloc(&dy, nl * n * 16) || cudaMalloc(&dt, tab.size() * 4)) return 3;
    cudaMemcpy(dp, hp.data(), np * 16, cudaMemcpyHostToDevice);
    cudaMemcpy(dx, x.data(), nl * n * 16, cudaMemcpyHostToDevice);
    cudaMemcpy(dt, tab.data(), tab.size() * 4, cudaMemcpyHostToDevice);
    P.itab = dt;
    for (int w = 0; w < 2; ++w) {
      P.wide = w;
      k<<<1, 128, nl * ls * sizeof(double2)>>>(P, dx, dy, dp, nl, ls);
      y[w].resize(nl * n);
      if (cudaMemcpy(y[w].data(), dy, nl * n * 16, cudaMemcpyDeviceToHost) != cudaSuccess) return 4;
    }
    if (memcmp(y[0].data(), y[1].data(), nl * n * 16)) printf("%d ", n), ++bad;
    for (int j = 0; j < nl * n * 16; ++j) hash = (hash ^ ((unsigned char*)y[0].data())[j]) * 1099511628211ull;
    cudaFree(dp), cudaFree(dx), cudaFree(dy), cudaFree(dt);
  }
  printf("differ: %d hash: %llx\n", bad, hash);
  return 0;
}
"""


@pytest.mark.gpu
def test_wide_and_whole_stages_agree_under_any_contraction(tmp_path):
    torch_cuda()
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    src = tmp_path / "stages.cu"
    src.write_text(SOURCE)
    libs = ["-lquadmath", "-Xcompiler=-fext-numeric-literals"] if platform.machine() == "x86_64" else []
    jobs = []
    for fmad in ("true", "false"):
        exe = str(tmp_path / f"stages_{fmad}")
        cmd = [nvcc, "-gencode=arch=compute_103a,code=sm_103a", "-O3", "-std=c++17", "-fmad=" + fmad, "-I" + CSRC,
               "-I" + os.path.join(ROOT, "include"), str(src), os.path.join(CSRC, "fcsph_tables.cpp"), "-o", exe] + libs
        jobs.append((exe, subprocess.Popen(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)))
    out = []
    for exe, p in jobs:
        log = p.communicate()[0]
        assert p.returncode == 0, log
        r = subprocess.run([exe], capture_output=True, text=True, timeout=120)
        assert r.returncode == 0, (r.returncode, r.stderr)
        out.append(r.stdout)
    assert out[0].startswith("differ: 0 ") and out[0] == out[1], out
