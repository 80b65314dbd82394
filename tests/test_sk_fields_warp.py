"""The fields warp of the persistent SK sweep leaves no copy in flight, on the CPU with the code the
kernel runs (csrc/sk_fields_warp.h): neither where one of its own waits gives up nor where none does.
In the second case the other warps of the CTA may still give up after it has issued its last copies, so
they have to have landed by then as well."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_1906_11195_gb300", "csrc")


@pytest.fixture(scope="module")
def fields_warp(tmp_path_factory):
    if shutil.which("g++") is None:
        pytest.skip("g++ not available")
    exe = str(tmp_path_factory.mktemp("fields_warp") / "run")
    subprocess.run(["g++", "-O1", "-std=c++17", "-I", CSRC, "-o", exe,
                    os.path.join(HERE, "sk_fields_warp_harness.cpp")], check=True)
    return lambda *a: [int(x) for x in subprocess.run([exe, *map(str, a)], capture_output=True, text=True,
                                                      check=True).stdout.split()]


@pytest.mark.parametrize("nk,nb,L", [(2, 5, 4), (3, 5, 4), (7, 7, 6), (40, 8, 6), (64, 9, 8)])
def test_no_copy_is_in_flight_when_the_warp_leaves(fields_warp, nk, nb, L):
    waits = max(0, nk - 3) + max(0, nk - L - 1)
    for stop in [-1, *range(waits)]:
        copies, in_flight, bad = fields_warp(nk, nb, L, stop)
        assert copies == nk if stop < 0 else copies < nk
        assert in_flight == 0 and not bad, f"{in_flight} copies in flight, waits that succeed: {stop}"
