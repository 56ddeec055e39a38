"""The staged FP64 walks leave each warp's extremes in shared memory as 8-byte
pairs.  A shared array is aligned as its element type demands and no more, so
the array's type has to be the one it is accessed with: checked by compiling,
nothing runs."""
import os
import shutil
import subprocess

import pytest

from paper_1701_04329_gb300 import build as B

SRC = r"""
#include "kernels_smooth.cuh"
template <typename R, typename P> constexpr size_t slot_align(R (*)(unsigned, unsigned, P *)) { return alignof(P); }
template <typename P> constexpr size_t slot_align(int (*)(const P *, int)) { return alignof(P); }
static_assert(slot_align(&afg::fx_leave) >= sizeof(int2), "slots a warp writes as one int2");
static_assert(slot_align(&afg::fx_exponent<32, 6>) >= sizeof(int2), "slots a thread reads as one int2");
"""


def test_reduction_slots(tmp_path):
    if not (shutil.which("nvcc") or os.path.exists("/usr/local/cuda/bin/nvcc")):
        pytest.skip("needs nvcc")
    src = tmp_path / "slots.cu"
    src.write_text(SRC)
    r = subprocess.run([B.nvcc()] + B.NVCC_FLAGS + ["-I", B.CSRC, "-c", str(src), "-o", str(tmp_path / "slots.o")],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
