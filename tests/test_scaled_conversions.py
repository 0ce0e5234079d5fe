"""The scaled binary64 -> int64 and the binary64 -> FP32 conversions on the integer pipe
(paper_1201_3185_gb300/csrc/fixed_conv.h), built for the host and checked against exact references: the product with a
power of two rounded half to even by numpy, and numpy's float32 conversion."""
import os
import shutil
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1201_3185_gb300", "csrc")
DRIVER = r"""
#include <cstdio>
#include <vector>
#include "fixed_conv.h"
int main(int argc, char** argv)
{
    FILE* f = fopen(argv[1], "rb");
    long long n = 0;
    if (fread(&n, 8, 1, f) != 1) return 1;
    std::vector<double> x(n);
    std::vector<int> e(n);
    if (fread(x.data(), 8, n, f) != (size_t)n || fread(e.data(), 4, n, f) != (size_t)n) return 1;
    fclose(f);
    std::vector<long long> q(n);
    std::vector<float> s(n);
    for (long long i = 0; i < n; ++i) q[i] = qumond::f64_to_i64_rn_scaled(x[i], e[i]), s[i] = qumond::f64_to_f32_rn(x[i]);
    FILE* g = fopen(argv[2], "wb");
    fwrite(q.data(), 8, n, g);
    fwrite(s.data(), 4, n, g);
    fclose(g);
    return 0;
}
"""


def test_scaled_and_narrowing_conversions(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no host C++ compiler")
    src, exe = tmp_path / "d.cpp", tmp_path / "d"
    src.write_text(DRIVER)
    subprocess.run([cxx, "-O2", "-std=c++17", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    rng = np.random.default_rng(11)
    e = rng.integers(-60, 101, 300000).astype(np.int32)
    # x 2^e from 2^-4 to 2^61, ties among them; FP32's range, its ends and ties between its values
    x = np.ldexp(rng.random(e.size) + 0.5, rng.integers(-3, 62, e.size) - e) * rng.choice([-1.0, 1.0], e.size)
    x[:1000] = np.ldexp(rng.integers(-(1 << 51), 1 << 51, 1000) + 0.5, -e[:1000])
    x[1000:1500] = 0.0
    x[1500:2000] = -0.0
    f = rng.standard_normal(50000).astype(np.float32)
    mid = 0.5 * (f.astype(np.float64) + np.nextafter(f, np.float32(np.inf)).astype(np.float64))
    ends = np.array([3.4028234663852886e38, 3.4028235677973366e38, 3.5e38, 1.1754943508222875e-38, 1.17549429e-38,
                     1e-40, 1e-45, 7e-46, 1e-300, 5e-324, np.inf, np.nan])
    more = np.concatenate([mid, -mid, ends, -ends])
    x, e = np.concatenate([x, more]), np.concatenate([e, np.zeros(more.size, np.int32)])
    with open(tmp_path / "in", "wb") as out:
        np.array([x.size], dtype=np.int64).tofile(out)
        x.tofile(out)
        e.tofile(out)
    subprocess.run([str(exe), str(tmp_path / "in"), str(tmp_path / "out")], check=True)
    raw = np.fromfile(tmp_path / "out", dtype=np.uint8)
    q, s = raw[:8 * x.size].view(np.int64), raw[8 * x.size:].view(np.float32)
    with np.errstate(over="ignore", invalid="ignore"):
        y = np.ldexp(x, e)
        want = np.where(np.abs(y) < 2.0 ** 62, np.rint(y), 0.0).astype(np.int64)
        want = np.where(np.abs(y) < 2.0 ** 62, want, np.where(np.signbit(x), -(1 << 62), 1 << 62))
        narrow = x.astype(np.float32)
    ok = np.abs(y) != 2.0 ** 62
    assert np.array_equal(q[ok], want[ok])
    assert np.array_equal(s.view(np.uint32)[~np.isnan(x)], narrow.view(np.uint32)[~np.isnan(x)])
    assert np.isnan(s[np.isnan(x)]).all()
