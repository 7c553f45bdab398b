"""Shared memory that a launch asks for to hold its blocks per SM down
(csrc/rtlbfs_smem.h), on the CPU: never less than the blocks need, never more
than a block may have, and where it is more than they need, the wanted number
of blocks fits and one more does not.  Blocks per SM from 1 to far beyond the
228 from which an even share is less than the system's part of a block."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2202_13449_gb300", "csrc")
DRIVER = r"""
#include <cstdio>
#include <cstdlib>
#include "rtlbfs_smem.h"
int main(int, char** argv)
{
    const std::size_t need = (std::size_t)std::atoll(argv[1]);
    for (long long b = 1; b <= 2000; ++b) std::printf("%zu\n", rtlbfs::smem_for_blocks(need, b));
    std::printf("%zu\n", rtlbfs::smem_for_blocks(need, 2147483647LL));
    return 0;
}
"""
SM, SYSTEM, MOST = 228 * 1024, 1024, 227 * 1024


@pytest.fixture(scope="module")
def driver(tmp_path_factory):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("g++ not found")
    d = tmp_path_factory.mktemp("smem")
    (d / "drv.cpp").write_text(DRIVER)
    exe = d / "drv"
    subprocess.run([gxx, "-std=c++17", "-O1", "-I", CSRC, str(d / "drv.cpp"), "-o", str(exe)],
                   check=True)
    return str(exe)


@pytest.mark.parametrize("need", [8000, 42464, 76032, 115841, 200000, MOST])
def test_request(driver, need):
    got = [int(x) for x in subprocess.run([driver, str(need)], check=True, capture_output=True,
                                          text=True).stdout.split()]
    for b, ask in zip(list(range(1, 2001)) + [2 ** 31 - 1], got):
        assert need <= ask <= MOST, b
        if ask > need:
            assert b * (ask + SYSTEM) <= SM < (b + 1) * (ask + SYSTEM), b
        else:  # the blocks need more than an even share of one block more
            assert (b + 1) * (need + SYSTEM) > SM - (b + 1) * 128, b
