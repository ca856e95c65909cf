"""The host-side splits of a step (csrc/plan.h), compiled on their own."""
import ctypes as C
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
WRAP = """
#include "plan.h"
extern "C" int grid(long long N, int sms, int waits) { return ktune::shared_grid(N, sms, waits != 0); }
"""


@pytest.fixture(scope="module")
def plan(tmp_path_factory):
    d = tmp_path_factory.mktemp("plan")
    src, lib = d / "plan.cc", d / "plan.so"
    src.write_text(WRAP)
    subprocess.run(["g++", "-std=c++17", "-O1", "-Wall", "-Werror", "-shared", "-fPIC", "-I",
                    os.path.join(ROOT, "paper_2102_05297_gb300", "csrc"), str(src), "-o", str(lib)], check=True)
    return C.CDLL(str(lib))


@pytest.mark.parametrize("sms", [1, 3, 132, 152])
@pytest.mark.parametrize("waits", [0, 1])
def test_grids_leave_room_for_other_searches(plan, sms, waits):
    """Every grid fits the GPU and takes no more than one chunk of 4,096 per CTA where
    the GPU has the SMs; small spaces leave most of the GPU free."""
    for N in [1, 2, 4097, 5120, 16384, 16385, 40960, 77824, 77825, 155648, 155649, 162816, 204288, 245760, 262143]:
        g = plan.grid(N, sms, waits)
        assert 1 <= g <= sms
        assert -(-N // g) <= 4096 or g == sms
        if sms == 152:
            assert g <= max(16, -(-N // 1024))
            if N > 152 * 1024:
                assert g <= 133            # a step may start while another draws
            if not waits:
                assert g <= max(38, -(-N // 4096))
