"""The fixed-point transforms of the FP64 products (csrc/fx.cuh), run on the host.

`fx_stages_host.cu` runs the stages and the scale rule of the kernels at every transform
length, forward on half-zero inputs and inverse on full ones, and checks that no value
leaves the range the arithmetic needs (an error of 1e9 is printed if one does).  The bound
is the rounding of an FP64 transform of the same length, 2^-53 per radix-2 level in the
2-norm (Higham, Accuracy and Stability of Numerical Algorithms, Section 24.1, with the
constant of the level taken as 1)."""
import math
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
LENGTHS = (16, 32, 64, 128, 256, 512, 1024, 2048, 4096, 24, 48, 96, 192, 384, 768, 1536, 3072)


@pytest.fixture(scope="module")
def errors(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    exe = str(tmp_path_factory.mktemp("fx") / "fx_stages_host")
    r = subprocess.run([nvcc, "-std=c++17", "-O2", "--expt-relaxed-constexpr", "-x", "cu",
                        os.path.join(HERE, "fx_stages_host.cu"), "-o", exe], capture_output=True, text=True, timeout=900)
    assert r.returncode == 0, r.stderr[-4000:]
    out = subprocess.run([exe], capture_output=True, text=True, timeout=900, check=True).stdout
    return {(int(a), b, int(c)): float(d) for a, b, c, d in (line.split() for line in out.splitlines())}


@pytest.mark.parametrize("L", LENGTHS)
def test_transform_is_as_exact_as_fp64(errors, L):
    got = {k: v for k, v in errors.items() if k[0] == L}
    assert len(got) == 6
    bad = {k: v for k, v in got.items() if not v <= 2.0 ** -53 * math.log2(L)}
    assert not bad, bad
