"""df_split (csrc/sg_df.cuh) gives bit for bit the pair of df2's conversion,
hi = fl32(d), lo = fl32(d - hi): random mantissas over all exponents, ties and
their neighbours, the edges of the integer path, zeros, subnormals, infinities
and NaN.  Host build of the device function."""
import os
import shutil
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2111_13655_gb300", "csrc")
DRIVER = r"""
#include <cstdio>
#include "sg_df.cuh"
int main() {
    double d;
    while (std::fread(&d, 8, 1, stdin) == 1) {
        const sg::df2 r = sg::df_split(d), q(d);
        std::fwrite(&r, 8, 1, stdout);
        std::fwrite(&q, 8, 1, stdout);
    }
    return 0;
}
"""


def test_split_equals_the_conversions_bitwise(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no host C++ compiler")
    src, exe = tmp_path / "d.cpp", tmp_path / "d"
    src.write_text(DRIVER)
    subprocess.run([cxx, "-std=c++17", "-O2", "-ffp-contract=off", f"-I{CSRC}", str(src), "-o", str(exe)], check=True)
    g = np.random.Generator(np.random.PCG64(3))
    m, e = g.integers(0, 2 ** 52, 200000, dtype=np.uint64), g.integers(0, 2048, 200000, dtype=np.uint64)
    s = g.integers(0, 2, 200000, dtype=np.uint64)
    near = np.array([(t << 29) + (1 << 28) + d for t in (0, 1, 5, 2 ** 23 - 2, 2 ** 23 - 1) for d in (-1, 0, 1)]
                    + [0, 1, 2 ** 29 - 1, 2 ** 52 - 1], dtype=np.uint64)
    edge = np.array([0, 1, 896, 897, 954, 955, 956, 1022, 1023, 1148, 1149, 1150, 1151, 2046, 2047], dtype=np.uint64)
    M, E, S = (a.ravel() for a in np.meshgrid(near, edge, np.array([0, 1], dtype=np.uint64)))
    bits = np.concatenate([(s << 63) | (e << 52) | m, (s << 63) | ((e % 195 + 955) << 52) | m, (S << 63) | (E << 52) | M])
    out = subprocess.run([str(exe)], input=bits.astype(np.uint64).tobytes(), capture_output=True, check=True).stdout
    r = np.frombuffer(out, np.uint32).reshape(-1, 4)
    nan = np.isnan(r.view(np.float32))
    assert len(r) == len(bits) and (nan[:, :2] == nan[:, 2:]).all()
    assert ((r[:, :2] == r[:, 2:]) | nan[:, :2]).all()
