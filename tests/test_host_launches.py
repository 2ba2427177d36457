"""What calls launch, looked over without a GPU: the library's objects on a recording runtime (tests/host).  Workspaces have
exactly the queried size; every tensor map, result matrix and slice buffer has to lie inside the buffers of its call."""
import os
import subprocess
import sys

import pytest

from paper_2103_03936_b200 import build as pf_build

HOST = os.path.join(os.path.dirname(os.path.abspath(__file__)), "host")


@pytest.fixture(scope="session")
def host_library(tmp_path_factory):
    d = tmp_path_factory.mktemp("host")
    objects, launches, library = pf_build.objects(), str(d / "launches.o"), str(d / "libpf_host.so")
    include = ["-I", os.path.join(pf_build.ROOT, "include"), "-I", pf_build.CSRC]
    subprocess.check_call([pf_build.nvcc()] + pf_build.NVCC_FLAGS + include + ["-c", "-o", launches, os.path.join(HOST, "launches.cu")])
    cuda = os.path.join(os.path.dirname(os.path.dirname(pf_build.nvcc())), "include")
    subprocess.check_call([os.environ.get("CXX", "g++"), "-std=c++17", "-fPIC", "-shared", "-Wl,-Bsymbolic", "-isystem", cuda, "-o", library,
                           os.path.join(HOST, "runtime.cpp"), launches] + objects)
    return library


@pytest.mark.parametrize("kind", ["linear", "linear_bwd", "linear_f32", "linear_f32_bwd", "grouped", "grouped_bwd", "conv", "conv_bwd",
                                  "conv_f32", "conv_f32_bwd"])
def test_nothing_reaches_outside_the_buffers_of_a_call(host_library, kind):
    """Thousands of drawn calls of every kind; backwards whose reductions over the batch do not fit the machine together
    among them, whose slices once lay behind the workspace."""
    done = subprocess.run([sys.executable, os.path.join(HOST, "calls.py"), host_library, kind, "8000", "1"], capture_output=True, text=True,
                          timeout=300)
    assert done.returncode == 0, done.stderr
    assert done.stdout == "calls reaching outside their buffers: 0\n", done.stdout[:4000]


@pytest.mark.parametrize("kernel", ["tc_conv_dt_dv_kernel", "tc_conv_du_kernel", "tc_conv_dx_kernel"])
def test_a_backward_that_cannot_be_prepared_launches_nothing_of_itself(host_library, kernel):
    """Convolution backward in three launches: what cannot be prepared leaves the call to the products that fetch pixels per
    tap, before x U has been recomputed or U copied for it."""
    code = f"""
import sys
sys.path.insert(0, {HOST!r})
import calls
lib = calls.Library({host_library!r})
lib.L.host_refuse({kernel.encode()!r})
status, faults, launches = calls.conv(lib, 64, 28, 28, 160, 40, 160, 3, 1, 1, calls.BF16, bwd=True, stash=False)
assert status == 0 and not faults, (status, faults)
kernels = launches.split()
named = lambda part: sum(part in k for k in kernels)
assert not named("tc_conv_d") and named("tc_gemm") == 2, launches
assert named("tc_conv_res_kernel") + named("tc_chain") == 1 and named("repack") == 1, launches
"""
    done = subprocess.run([sys.executable, "-c", code], capture_output=True, text=True, timeout=300)
    assert done.returncode == 0, done.stderr
