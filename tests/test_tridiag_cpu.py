"""The tridiagonal solve of the P-space preconditioner (mbe_tridiag.cuh, host
and device code) on the CPU against numpy's eigenvectors: Re (theta - T +
i delta)^{-1} f with theta below the block, inside it and on an eigenvalue.

Its 7 levels make about 32 FP32 roundings of elements below |theta - T| (100
here): relative errors up to 32 * 2^-24 * 100 / d at the distance d of theta from
the nearest eigenvalue, 4e-3 for d >= 0.05; and where theta is on an eigenvalue,
a perturbation of delta = 5e-5 by the roundings of an element (1e-5), so that the
bound 1 / (2 delta) becomes 1.25e4.
"""
import os
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_1905_02786_gb300", "csrc")
MAIN = r"""
#include "mbe_tridiag.cuh"
#include <cstdio>
static TriC s[2][5][TRI_MAX];
int main() {
  int n;
  float th, t[TRI_MAX], e[TRI_MAX], f[TRI_MAX];
  while (std::scanf("%d %f", &n, &th) == 2) {
    for (int i = 0; i < n; i++) if (std::scanf("%f %f %f", t + i, e + i, f + i) != 3) return 1;
    for (int i = 0; i < n; i++) {
      s[0][0][i] = {i > 0 ? -e[i - 1] : 0.f, 0.f};
      s[0][1][i] = {th - t[i], TRI_DELTA};
      s[0][2][i] = {i + 1 < n ? -e[i] : 0.f, 0.f};
      s[0][3][i] = {f[i], 0.f};
      s[0][4][i] = {-2.f * f[i], 0.f};
    }
    int cur = 0;
    for (int st = 1; st < n; st <<= 1, cur ^= 1)
      for (int i = 0; i < n; i++) tri_level(s[cur], s[cur ^ 1], i, st, n);
    for (int i = 0; i < n; i++)
      std::printf("%.9g %.9g\n", tri_div(s[cur][3][i], s[cur][1][i]).re,
                  tri_div(s[cur][4][i], s[cur][1][i]).re);
  }
}
"""


@pytest.fixture(scope="module")
def solve(tmp_path_factory):
    d = tmp_path_factory.mktemp("tri")
    src, exe = d / "tri.cpp", d / "tri"
    src.write_text(MAIN)
    subprocess.run(["g++", "-O1", "-std=c++17", "-I", CSRC, str(src), "-o", str(exe)], check=True)

    def run(t, e, th, f):
        text = f"{len(t)} {th:.9g}\n" + "\n".join("%.9g %.9g %.9g" % r for r in zip(t, [*e, 0.0], f))
        out = subprocess.run([str(exe)], input=text, capture_output=True, text=True, check=True)
        return np.array([[float(v) for v in r.split()] for r in out.stdout.splitlines()]).T

    return run


@pytest.mark.parametrize("n", [2, 3, 5, 64, 127, 128])
@pytest.mark.parametrize("base", [-2.0, -76.0])
@pytest.mark.parametrize("coupling", [0.5, 0.02])
def test_bounded_inverse(solve, n, base, coupling):
    rng = np.random.default_rng(n)
    t = (base + rng.exponential(2.0, n)).astype(np.float32)
    e = (coupling * rng.standard_normal(n - 1)).astype(np.float32)
    f = rng.standard_normal(n).astype(np.float32)
    w, V = np.linalg.eigh(np.diag(t.astype(float)) + np.diag(e.astype(float), 1)
                          + np.diag(e.astype(float), -1))
    for th in [w[0] - 0.3, w[0] - 0.05, 0.5 * (w[0] + w[1]), t[0], w[0], w[n // 2], w[0] + 1e-5,
               w[0] + 1e-4, w[-1] + 0.1]:
        th = np.float32(th)
        x, x2 = solve(t, e, th, f)
        d = float(th) - w
        ref = V @ (V.T @ f * d / (d * d + 2.5e-9))
        assert np.linalg.norm(x) <= 1.25e4 * np.linalg.norm(f)
        assert np.linalg.norm(x2 + 2 * x) <= 1e-5 * np.linalg.norm(x)   # the other right-hand side
        if np.abs(d).min() >= 0.05:
            assert np.linalg.norm(x - ref) <= 4e-3 * np.linalg.norm(ref)
