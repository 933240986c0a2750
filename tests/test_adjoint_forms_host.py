"""Both generated forms of the activation adjoint, on the host in double precision, for every compiled channel set: each
is the transpose of the tangent (Eq. 15, <A v, w> = <v, A^T w>), and the convolution of jets that the tensor-core kernel
runs equals the monomial form that the SIMT kernels run.  Sums of at most a few hundred products of values below 30: 1e-12
of their magnitudes."""
import shutil
import subprocess

import pytest

from paper_2606_29702_gb300 import build

HARNESS = r"""
#include <cmath>
#include <cstdio>
#include <random>
#define __device__
#define __host__
#define __forceinline__ inline
#include "jet_closures_gen.h"
using namespace jet;

template <class Cls>
static void run(const char* name) {
  constexpr int C = Cls::C;
  std::mt19937_64 rng(7);
  std::normal_distribution<double> nd;
  double forms = 0.0, inner = 0.0;
  for (int it = 0; it < 400; ++it) {
    double z[C], ab[C], v[C], p[6], da[C], zb[C], zc[C];
    for (int c = 0; c < C; ++c) z[c] = nd(rng), ab[c] = nd(rng), v[c] = nd(rng);
    const double a = std::tanh(z[0]), s = 1 - a * a;
    p[0] = a, p[1] = s, p[2] = -2 * a * s, p[3] = s * (6 * a * a - 2);
    p[4] = 8 * a * s * (2 - 3 * a * a), p[5] = 8 * s * (15 * a * a * a * a - 15 * a * a + 2);
    Cls::tangent(z, p, v, da);
    Cls::adjoint(z, p, ab, zb);
    Cls::adjoint_conv(z, p, ab, zc);
    double lhs = 0, rb = 0, rc = 0, mag = 1, big = 1;
    for (int c = 0; c < C; ++c) {
      lhs += da[c] * ab[c], rb += v[c] * zb[c], rc += v[c] * zc[c];
      mag += std::fabs(da[c] * ab[c]) + std::fabs(v[c] * zb[c]);
      big = std::fmax(big, std::fabs(zb[c]));
    }
    inner = std::fmax(inner, std::fmax(std::fabs(lhs - rb), std::fabs(lhs - rc)) / mag);
    for (int c = 0; c < C; ++c) forms = std::fmax(forms, std::fabs(zb[c] - zc[c]) / big);
  }
  std::printf("%s %.3e %.3e\n", name, forms, inner);
}

int main() {
#define RUN(id, cls) run<cls>(#cls);
  JET_FOR_EACH_CLASS(RUN)
}
"""


@pytest.mark.skipif(shutil.which("g++") is None, reason="no host compiler")
def test_adjoint_forms_agree(tmp_path):
    src, exe = tmp_path / "forms.cpp", str(tmp_path / "forms")
    src.write_text(HARNESS)
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-I" + build.CSRC, str(src), "-o", exe])
    lines = subprocess.check_output([exe], text=True).split("\n")[:-1]
    assert len(lines) == build.n_classes()
    for line in lines:
        name, forms, inner = line.split()
        assert float(forms) < 1e-12 and float(inner) < 1e-12, line
