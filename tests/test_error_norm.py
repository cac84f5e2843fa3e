"""The error norm that accepts a step of the FP64 forms, on the host, against
the plain maximum of the ratios in FP64: near ties (where the choice of the
species in FP32 is not sure), tolerances and errors outside the float range,
values that are not finite."""
import subprocess

import numpy as np

from paper_2311_08927_gb300 import build as B
from paper_2311_08927_gb300 import inputs as I

PROGRAM = r"""
#include <cstdio>
#include "error_norm.cuh"
using namespace chad;
int main() {
  double v[6][NS];
  const double rtol = 1e-6;
  while (std::fread(v, sizeof(v), 1, stdin) == 1) {
    const double r = error_ratio(v[0], v[1], v[2], v[3], v[4], rtol, v[5]);
    std::fwrite(&r, sizeof(r), 1, stdout);
  }
  return 0;
}
"""
RTOL = 1e-6


def _cases():
    """(y, y1, k1, k2, k3, atol) rows, and what they stand for."""
    rng = np.random.default_rng(11)
    NS, out, what = I.NS, [], []

    def add(w, y, y1, e, atol):
        # k1 - 2 k2 + k3 = e exactly
        out.append(np.stack([y, y1, np.zeros(NS), np.zeros(NS), e, atol]))
        what.append(w)

    for k in range(400):
        y = I.x_ss() * np.exp(rng.standard_normal(NS))
        y1 = y * (1 + 0.1 * rng.standard_normal(NS))
        atol = I.atol_vector() * 10.0 ** rng.uniform(-2, 2, NS)
        sc = atol + RTOL * np.maximum(np.abs(y), np.abs(y1))
        ratio = 10.0 ** rng.uniform(-3, 5, NS)
        e = ratio * sc * rng.choice([-1.0, 1.0], NS)
        add("plain", y, y1, e, atol)
        i, j = rng.choice(NS, 2, replace=False)  # two species apart by delta
        for delta in (0.0, 1e-15, 1e-9, 3e-7, 9e-7, 2e-6, 4e-6, 2e-5):
            t = e.copy()
            t[i] = 2e5 * sc[i]
            t[j] = 2e5 * (1 + delta) * sc[j]
            add(f"near tie {delta:g}", y, y1, t, atol)
        for a in (1e-310, 1e-200, 1e-45, 1e-31, 1e35):
            t = atol.copy()
            t[i] = a
            z, z1 = y.copy(), y1.copy()
            z[i] = z1[i] = 0.0
            add(f"atol {a:g}", z, z1, e * (1e30 if a > 1 else 1.0), t)
        add("no error", y, y1, 0.0 * e, atol)
        add("tiny errors", y, y1, 1e-42 * e, atol)
        add("huge errors", y, y1, 1e60 * e, atol)
        for bad in (np.inf, -np.inf, np.nan):
            t = e.copy()
            t[i] = bad
            add("error not finite", y, y1, t, atol)
            t = y1.copy()
            t[i] = bad
            add("state not finite", y, t, e, atol)
    return np.array(out), what


def test_norm_is_the_largest_ratio(tmp_path):
    src, exe = tmp_path / "norm.cu", tmp_path / "norm"
    src.write_text(PROGRAM)
    subprocess.run([B.nvcc(), *B.ARCH, *B.NVCC_FLAGS, "-o", str(exe), str(src)], check=True)
    v, what = _cases()
    r = subprocess.run([str(exe)], input=v.tobytes(), capture_output=True, check=True)
    got = np.frombuffer(r.stdout)
    assert got.size == len(what)
    with np.errstate(all="ignore"):
        e = np.abs(v[:, 4])
        sc = v[:, 5] + RTOL * np.maximum(np.abs(v[:, 0]), np.abs(v[:, 1]))
        ref = np.where(np.isfinite(e).all(1) & np.isfinite(sc).all(1), (e / sc).max(1), np.inf)
    for g, x, w in zip(got, ref, what):
        if np.isinf(x):
            assert np.isinf(g) and g > 0, w
        else:
            # the scale, its reciprocal, the product and the cross products
            # round once each
            assert abs(g - x) <= 8 * 1.2e-16 * x, (w, g, x)
