"""Registers and shared memory of kernels whose launches count on a number of blocks per SM, as ptxas reports them.  An SM has
four schedulers with 16 384 registers each; a block's warps are dealt out to them, each with its registers in units of 256."""
import os
import re
import subprocess

import pytest

from paper_2607_17374_b200 import build as tb_build

QUARTER = 16_384


@pytest.fixture(scope="module")
def kernels():
    """name -> list of (registers, bytes of static shared memory) of its instantiations."""
    tb_build.build()
    srcs = [os.path.join(tb_build.CSRC, n) for n in ("kernels_gemm_tc.cu", "kernels_resident.cu")]
    if not all(os.path.exists(tb_build.resource_log(s)) for s in srcs):
        tb_build.build(force=True)
    found = {}
    for s in srcs:
        text = open(tb_build.resource_log(s)).read()
        for name, used in re.findall(r"Compiling entry function '(\S+)' for.*?\n(?:.*\n)*?.*?(Used \d+ registers.*)", text):
            name = subprocess.run(["c++filt", name], capture_output=True, text=True, check=True).stdout
            name = re.search(r"(\w+)(<[^(]*>)?\(", name.replace("(anonymous namespace)::", "")).group(1)
            smem = re.search(r"(\d+) bytes smem", used)
            found.setdefault(name, []).append((int(re.search(r"Used (\d+)", used).group(1)), int(smem.group(1)) if smem else 0))
    return found


def _quarter(registers, threads):
    """Registers of the scheduler that gets most of a block's warps."""
    return (threads // 32 + 3) // 4 * ((registers * 32 + 255) // 256 * 256)


def test_the_whole_grid_of_store_rows_is_on_the_device_at_once(kernels):
    for registers, _ in kernels["store_rows_kernel"]:   # launched with eight blocks of 256 threads per SM
        assert 8 * _quarter(registers, 256) <= QUARTER


def test_a_block_of_the_accounting_fits_beside_a_projection(kernels):
    """Registers here; shared memory, most of it asked for at the launch, is asserted in the sources."""
    for registers, smem in kernels["project_tc_kernel"]:
        assert smem == 0
        for beside in ("account_kernel", "account_edges_kernel"):
            for r, s in kernels[beside]:
                assert _quarter(registers, 448) + _quarter(r, 256) <= QUARTER and s <= 128
