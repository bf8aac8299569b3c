"""Step weights at the end of the float32 range: a column of 2^127 has D_c^2 below 2^-128, whose
reciprocal is infinite.  A part that does not move adds 0 / weight = 0 to the step rule's sums in
every form of the step kernels."""
import numpy as np
import pytest

import lpgen
from test_gpu_resident import F32, FIXED, P, rel  # noqa: F401  (P: the fixture)

pytestmark = pytest.mark.gpu


def tiny_weights(m, n, seed=1):
    """A random covering LP beside ten rows of one fixed column with entries 2^127."""
    base = lpgen.set_cover(seed, m=m, n=n)
    rows = np.concatenate([np.repeat(np.arange(m), np.diff(base.row_ptr)), m + np.arange(10)])
    cols = np.concatenate([base.col, np.full(10, n)])
    val = np.concatenate([base.val, np.full(10, 2.0 ** 127)])
    z = np.zeros(1)
    return lpgen._lp(m + 10, n + 1, rows, cols, val, np.concatenate([base.b, np.zeros(10)]),
                     np.concatenate([base.sense, np.full(10, lpgen.SENSE_GE)]).astype(base.sense.dtype),
                     np.concatenate([base.c, z]), np.concatenate([base.l, z]),
                     np.concatenate([base.u, z]), np.zeros(n + 1, dtype=np.uint8), "tiny_weights")


@pytest.mark.parametrize("m,n,form", [(40, 160, 3), (300, 1200, 4)])
@pytest.mark.parametrize("adaptive", [0, 1])
def test_weights_below_the_range_of_reciprocals(P, m, n, form, adaptive):  # noqa: F811
    lp = tiny_weights(m, n)
    kw = dict(FIXED, adaptive_step=adaptive, precision="bf16", iter_limit=20)
    x, y, r = P.pdlp_solve(lp, P.default_params(**kw))
    x0, y0, r0 = P.pdlp_solve(lp, P.default_params(lanes_A=2, lanes_AT=2, **kw))
    assert (r["persistent_form"], r0["persistent_form"]) == (form, 0)
    assert r["precision_used"] == P.PDLP_USED_BF16
    assert r["status"] == r0["status"] == P.PDLP_ITER_LIMIT and r["iters"] == 20
    assert rel(x, x0) <= F32 and rel(y, y0) <= F32


PROGRAM = r"""
#include <cmath>
#include <cstdio>
#include <vector>
#include "resident_kernels.cuh"
__global__ void k_div(int count, const float* n, const float* d, float* q, float* plain) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < count) {
    q[i] = pdlp::div_pos(n[i], d[i]);
    plain[i] = n[i] / d[i];
  }
}
int main() {
  const int N = 1 << 22;
  std::vector<float> n(N), d(N), q(N), plain(N);
  unsigned long long s = 12345;
  auto bits = [&s] { return s = s * 6364136223846793005ull + 1442695040888963407ull, (unsigned)(s >> 33); };
  // a random significand (now and then one with all bits set or clear) at a random exponent
  auto number = [&](int lo, int hi) {
    const unsigned k = bits(), f = k % 16 == 0 ? 0u : k % 16 == 1 ? 0x7fffffu : bits() & 0x7fffffu;
    return std::ldexp(1.0f + std::ldexp((float)f, -23), lo + (int)(bits() % (unsigned)(hi - lo)));
  };
  for (int i = 0; i < N; ++i) {
    // (every hundredth divisor subnormal)
    d[i] = i % 100 == 1 ? std::ldexp((float)(1 + bits() % 0x7fffffu), -149) : number(-126, 128);
    do n[i] = i % 100 == 2 || i % 1000 == 1 ? 0.0f : number(-90, 120);
    while (n[i] > 0 && std::fabs(std::log2(n[i]) - std::log2(d[i])) > 120);
  }
  float *dn, *dd, *dq, *dp;
  for (float** p : {&dn, &dd, &dq, &dp})
    if (cudaMalloc(p, 4 * N) != cudaSuccess) return 1;
  cudaMemcpy(dn, n.data(), 4 * N, cudaMemcpyHostToDevice);
  cudaMemcpy(dd, d.data(), 4 * N, cudaMemcpyHostToDevice);
  k_div<<<N / 256, 256>>>(N, dn, dd, dq, dp);
  if (cudaMemcpy(q.data(), dq, 4 * N, cudaMemcpyDeviceToHost) != cudaSuccess) return 1;
  cudaMemcpy(plain.data(), dp, 4 * N, cudaMemcpyDeviceToHost);
  double worst = 0;
  int differ = 0;
  for (int i = 0; i < N; ++i) {
    const double want = (double)n[i] / (double)d[i];
    int e;
    std::frexp(want, &e);
    const double err = want == 0 ? (q[i] == 0 ? 0 : 1e9) : std::fabs(q[i] - want) / std::ldexp(1.0, e - 24);
    worst = err > worst || err != err ? err : worst;
    differ += q[i] != plain[i];
  }
  printf("%.9f %d\n", worst, differ);
  return 0;
}
"""


def test_quotients_of_the_step_rule(tmp_path):
    """n / d over the whole range of weights, subnormal ones among them: half an ulp and 2^-20 of one
    (the derivation stands at div_pos), and 0 for n = 0."""
    import os
    import subprocess
    from paper_2503_10344_gb300 import build as B
    src, exe = tmp_path / "div.cu", tmp_path / "div"
    src.write_text(PROGRAM)
    r = subprocess.run([B._nvcc(), *B.ARCH, "-std=c++17", "-O3", "-I" + os.path.join(B.ROOT, "include"),
                        "-I" + B.CSRC, str(src), "-o", str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    out = subprocess.run([str(exe)], capture_output=True, text=True)
    assert out.returncode == 0, out.stdout
    print(out.stdout)
    assert float(out.stdout.split()[0]) <= 0.5 + 2.0 ** -20, out.stdout
