"""The request server's admission on a CPU (server_host.cu: server.cu on a fake of the
CUDA runtime whose memory and completions the scenario controls)."""
import os
import subprocess

import pytest

from paper_2001_02765_gb300 import build as b
from tests._lib import ROOT


@pytest.fixture(scope="module")
def host(tmp_path_factory):
    exe = str(tmp_path_factory.mktemp("server_host") / "server_host")
    subprocess.check_call([b._nvcc(), "-gencode", "arch=compute_103a,code=compute_103a", "-O1", "-std=c++17", "-ftz=true",
                           "--expt-relaxed-constexpr", "-I", b.INCLUDE, "-I", b.CSRC, "-cudart", "shared",
                           os.path.join(ROOT, "tests", "server_host.cu"), "-o", exe, "-lpthread"])
    return lambda scenario: subprocess.run([exe, scenario], capture_output=True, text=True, timeout=120)


@pytest.mark.parametrize("scenario", ["failed_group_keeps_arrival_order", "completions_during_a_launch_are_noticed"])
def test_admission(host, scenario):
    r = host(scenario)
    assert r.returncode == 0, r.stderr
