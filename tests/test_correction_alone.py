"""The correction pass without a transform of the new velocity (no next substep), on
a grid small enough for one CTA per component: an empty grid of instances, so that
only the launcher's arithmetic runs and the launch itself is refused."""
import os
import subprocess

import pytest

from paper_2606_06247_gb300 import build

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
PKG = os.path.join(ROOT, "paper_2606_06247_gb300")

SOURCE = r"""
#include <cstdio>
#include "fcsph_internal.h"
using namespace fcsph;
int main() {
  for (int nz : {1, 16}) {
    fcsph_ctx c;
    c.prec.fft_prec = FCSPH_F64;
    c.gd.nx = c.gd.ny = 16;
    c.gd.nz = nz;
    c.gd.ncol = 16 * nz;
    c.gd.hy = c.gd.rows = 21;
    c.gd.batch = 1;
    c.gd.nb = 0;
    std::vector<double> re, im;
    std::vector<int> tab;
    Pool pool;
    c.plan_y = make_plan(41, &pool, &re, &im);
    c.ip_y = make_ip(c.plan_y, pool, &tab);
    double* v[3] = {};
    printf("%d ", (int)launch_step_corr(&c, StepDev(), nullptr, v, v, nullptr));
  }
  return 0;
}
"""


@pytest.mark.skipif(not os.path.isdir("/usr/local/cuda/include"), reason="no CUDA headers")
def test_correction_without_a_next_transform(tmp_path):
    lib = build.build()
    src, exe = tmp_path / "corr.cpp", tmp_path / "corr"
    src.write_text(SOURCE)
    subprocess.run(["g++", "-O1", "-std=gnu++17", "-I" + os.path.join(PKG, "csrc"), "-I" + os.path.join(ROOT, "include"),
                    "-I/usr/local/cuda/include", str(src), lib, "-o", str(exe), "-Wl,-rpath," + PKG], check=True,
                   capture_output=True, text=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, (r.returncode, r.stdout, r.stderr)
    for code in r.stdout.split():
        assert int(code) not in (0, 1)  # the launch refused, not the arguments (1: invalid value)
