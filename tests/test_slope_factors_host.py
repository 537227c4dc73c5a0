"""The slope factors sin(2 pi k / P) / h of the central column pass carry no more than
the rounding of their table entry in any bin (CPU, compiled from fftconv.cuh)."""
import os
import subprocess

from paper_2001_02765_gb300 import build as b
from tests._lib import ROOT


def test_sines_are_as_good_as_the_table(tmp_path):
    exe = str(tmp_path / "slope_factors_host")
    subprocess.check_call([b._nvcc(), "-gencode", "arch=compute_103a,code=compute_103a", "-O1", "-std=c++17", "-ftz=true",
                           "--expt-relaxed-constexpr", "-I", b.INCLUDE, "-I", b.CSRC,
                           os.path.join(ROOT, "tests", "slope_factors_host.cu"), "-o", exe])
    rows = [l.split() for l in subprocess.check_output([exe], text=True).splitlines()]
    assert len(rows) == 15
    for length, e32, e64 in rows:
        # one rounding in FP32; FP64 entries also carry the sine, the cosine and the quotient
        assert float(e32) <= 1.001, length
        assert float(e64) <= 4.0, length
