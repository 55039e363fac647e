"""The FP64 screen's vote bounds a thread's values by the high word of the largest: the
bound holds for every number, and no infinity or NaN passes as a small one."""
import shutil
import struct
import subprocess

import numpy as np
import pytest

from paper_2306_15678_gb300 import build

SRC = r"""
#include <cstdio>
#include "kernels.cuh"
int main() {
    int h;
    while (std::scanf("%d", &h) == 1) std::printf("%d\n", nlse::hi_word_above(h));
}
"""


def test_bound_of_every_kind_of_value(tmp_path):
    try:
        cc = build.nvcc()
    except RuntimeError as e:
        pytest.skip(str(e))
    assert shutil.which("g++")
    (tmp_path / "t.cu").write_text(SRC)
    subprocess.run([cc, *build.ARCH, "-std=c++17", "-I", build.CSRC, str(tmp_path / "t.cu"), "-o", str(tmp_path / "t")],
                   check=True, capture_output=True)
    rng = np.random.default_rng(1)
    finite = np.concatenate([np.exp(rng.uniform(-700, 700, 500)), [0.0, 5e-324, 2.2e-308, 1.0, np.finfo(float).max]])
    words = [struct.unpack("<II", struct.pack("<d", v))[1] for v in finite]
    special = [0x7ff00000, 0x7ff00001, 0x7ff80000, 0x7ffffffe, 0x7fffffff]  # infinity and NaNs
    out = subprocess.run([str(tmp_path / "t")], input=" ".join(str(w) for w in words + special), check=True,
                         capture_output=True, text=True).stdout.split()
    top = [struct.unpack("<d", struct.pack("<Ii", 0, int(w)))[0] for w in out]
    assert all(t > v for t, v in zip(top, finite))
    assert all(t == np.inf for t in top[len(finite):])
