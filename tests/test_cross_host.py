"""Host side of the FP32 cross-patch sum on a CPU (cross_host.cu: the launches it
makes, recorded by a fake of the CUDA runtime), and the plan's limit on cells."""
import os
import subprocess

import pytest

from paper_2001_02765_gb300 import build as b
from tests._lib import ROOT, ensure_built


@pytest.fixture(scope="module")
def host(tmp_path_factory):
    exe = str(tmp_path_factory.mktemp("cross_host") / "cross_host")
    subprocess.check_call([b._nvcc(), "-gencode", "arch=compute_103a,code=compute_103a", "-O1", "-std=c++17", "-ftz=true",
                           "--expt-relaxed-constexpr", "-I", b.INCLUDE, "-I", b.CSRC, "-cudart", "shared",
                           os.path.join(ROOT, "tests", "cross_host.cu"), "-o", exe])
    return lambda scenario: subprocess.run([exe, scenario], capture_output=True, text=True, timeout=120)


@pytest.mark.parametrize("scenario", ["clears_every_sum", "empty_patch_adds_no_launch", "unbuilt_tables_are_dropped"])
def test_host_side(host, scenario):
    r = host(scenario)
    assert r.returncode == 0, r.stderr


def test_more_cells_than_32_bit_indexes_are_refused():
    """512 patches of 2048^2 are 2^31 cells: output indexes and target counts are 32-bit."""
    ensure_built()
    from paper_2001_02765_gb300 import sg
    tiles = lambda n: [(0, 2048, 2048, 2048.0 * (k % 32), 2048.0 * (k // 32), 1.0) for k in range(n)]
    with pytest.raises(sg.SgError) as e:
        sg.sg_plan_bytes(tiles(512), sg.SG_FP32)
    assert e.value.status == sg.SG_EINVAL and "cells" in str(e.value)
