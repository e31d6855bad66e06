"""The integer conversions between FP64 and FP32 pairs against the conversion instructions, bit
for bit (up to the sign of a zero lo): every exponent of both formats, ties, carries, powers
of two, all-ones mantissas, both signs, subnormals, infinities and NaN, and pairs that are
not normalised."""
import os
import subprocess

import pytest

from paper_2405_12380_gb300 import build
from tests.gpu_common import need_gpu

pytestmark = pytest.mark.gpu


def test_conversions_equal_the_instructions(tmp_path):
    need_gpu()
    exe = str(tmp_path / "pair_conversion")
    src = os.path.join(os.path.dirname(os.path.abspath(__file__)), "pair_conversion.cu")
    include = os.path.join(os.path.dirname(build.HERE), "include")
    r = subprocess.run([build.nvcc(), *build.ARCH, *build.FLAGS, "-I", build.CSRC, "-I", include, src, "-o", exe, "-lcudart"],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-3000:]
    out = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    assert out.returncode == 0, out.stderr[-1000:]
    n, bad, m, bad2 = (int(t) for t in out.stdout.split()[:4])
    assert n > 10 ** 6 and m > 10 ** 6 and bad == 0 and bad2 == 0, out.stdout
