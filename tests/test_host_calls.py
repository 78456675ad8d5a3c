"""The host side of single-key calls on a stand-in for the CUDA runtime
(tests/host_check/tdes_fake_runtime.cpp): what happens to round keys in host
memory, without a GPU."""
import os
import shutil
import subprocess

import pytest

from paper_2007_10752_gb300 import build

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def exe(tmp_path_factory):
    if not os.path.exists(build.nvcc()) and shutil.which("nvcc") is None:
        pytest.skip("nvcc not available")
    d = tmp_path_factory.mktemp("fake")
    srcs = [os.path.join(ROOT, "tests", "host_check", "tdes_fake_runtime.cpp"),
            os.path.join(build.CSRC, "tdes_api.cu"), os.path.join(build.CSRC, "tdes_small.cu")]
    objs = [str(d / (os.path.basename(s) + ".o")) for s in srcs]
    flags = [f for f in build.NVCC_FLAGS if f not in ("-Xptxas", "-v")]  # the library's own optimisation
    procs = [subprocess.Popen([build.nvcc(), *build.ARCH, *flags, "-c", s, "-o", o])
             for s, o in zip(srcs, objs)]
    assert [p.wait() for p in procs] == [0] * len(procs)
    out = str(d / "fake")
    subprocess.check_call(["g++", "-o", out, *objs, "-lpthread"])
    return out


def _case(exe, *args):
    r = subprocess.run([exe, *args], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stderr


@pytest.mark.parametrize("case", ["free", "launch", "sync", "params"])
def test_round_keys_are_cleared(exe, case):
    """Round keys in host memory are overwritten before the memory is freed, on
    the error paths too, and a launch leaves no copy of them on a stack."""
    _case(exe, case)


def test_key_schedule_copies_nothing_back(exe):
    """The host's round keys are those of the kernel's recipe, without a copy
    from the device."""
    _case(exe, "copies")
