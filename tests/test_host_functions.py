"""Device functions that also compile for the host, checked there value by value
(CPU only; nvcc compiles the file, nothing runs on a GPU): the 32-bit square
root of the node features against the FP64 root rounded to FP32."""
import subprocess

import pytest

from paper_2306_00606_gb300 import _build

ROOT_CHECK = r"""
#include "ef_internal.cuh"
#include <cmath>
#include <cstdio>
int main() {
    long tried = 0, wrong = 0;
    auto check = [&](int64_t x) {
        ++tried;
        wrong += ef::sqrt_exact(x) != (float)std::sqrt((double)x);
    };
    for (int64_t x = 0; x < 1 << 22; ++x) check(x);
    for (int64_t x : {764411958ll, 1474560150ll, (1ll << 46) - 1, 1ll << 46, (1ll << 62) + 12345}) check(x);
    uint64_t z = 88172645463325252ull;
    for (int i = 0; i < 4000000; ++i) {   // over the logarithm of the range
        z ^= z << 13; z ^= z >> 7; z ^= z << 17;
        check((int64_t)(z >> (18 + (z >> 58) % 46)) & ((1ll << 46) - 1));
    }
    for (int i = 0; i < 4000000; ++i) {   // on either side of values halfway between two FP32 numbers
        z ^= z << 13; z ^= z >> 7; z ^= z << 17;
        const double y = std::ldexp(2.0 * ((1u << 23) | (uint32_t)(z & 0x7fffff)) + 1.0, -1 - (int)((z >> 40) % 23));
        if (y * y >= 7e13) continue;
        for (int d = -1; d <= 1; ++d) check((int64_t)std::floor(y * y) + d);
    }
    std::printf("%ld %ld\n", tried, wrong);
    return 0;
}
"""


def test_feature_root_is_the_rounded_fp64_root(tmp_path):
    src, exe = tmp_path / "root.cu", tmp_path / "root"
    src.write_text(ROOT_CHECK)
    try:
        subprocess.run([_build.nvcc(), "-O2", "-std=c++17", "-Xcompiler", "-ffp-contract=off", "-I", _build.CSRC, "-I",
                        _build.INCLUDE, *_build.ARCH, str(src), "-o", str(exe)], check=True, capture_output=True)
    except FileNotFoundError:
        pytest.skip("no nvcc here")
    tried, wrong = map(int, subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split())
    assert tried > 8_000_000 and wrong == 0
