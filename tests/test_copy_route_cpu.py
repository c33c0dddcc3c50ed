"""Which copies run as kernels: those between memory of the device that the solver's arrays live on, whichever device
is current in the calling thread; and the size of their grid follows that device."""
import ctypes
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2211_05647_gb300", "csrc")
SHIM = """#include "copy_route.cuh"
extern "C" int reaches(int device_memory, int theirs, int home)
{
    return fp::kernel_reaches(device_memory != 0, theirs, fp::CopyHome{home, 1});
}
extern "C" uint32_t blocks(uint32_t units, uint32_t per, int sms) { return fp::copy_blocks(units, per, fp::CopyHome{0, sms}); }
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("route")
    (d / "shim.cpp").write_text(SHIM)
    so = str(d / "shim.so")
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, str(d / "shim.cpp"), "-o", so], check=True)
    return ctypes.CDLL(so)


def test_only_memory_of_the_arrays_device(lib):
    for home in (0, 1, 3):
        for theirs in (0, 1, 3):
            assert lib.reaches(1, theirs, home) == (theirs == home)
            assert lib.reaches(0, theirs, home) == 0      # host, managed or unregistered memory


def test_grid_of_a_linear_copy(lib):
    for sms in (16, 152):
        assert lib.blocks(1, 1024, sms) == 1
        assert lib.blocks(1025, 1024, sms) == 2
        assert lib.blocks(8 * sms * 1024, 1024, sms) == 8 * sms
        assert lib.blocks(2 ** 31, 1024, sms) == 8 * sms


def test_launches_of_a_handle_go_to_its_device():
    """The kernels that took the place of copies and graph launches, neither of which needs the handle's device to be
    current, make it current themselves."""
    rows = open(os.path.join(CSRC, "rows.cu")).read()
    assert rows.count("launch_pdl(") + rows.count("<<<") == 3 and rows.count("DeviceGuard guard(home.dev)") == 2
    capi = open(os.path.join(CSRC, "capi.cu")).read()
    i = capi.index("int fdtd_plasma_step(fdtd_plasma_t h")
    assert "DeviceGuard guard(h->dev)" in capi[i:capi.index("line_step(h, nsteps)", i)]
