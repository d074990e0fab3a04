"""What the persistent kernels need of an SM, from the compiler (no GPU): one
block of 1024 threads (k_sweep, k_far_sweep) or 768 (k_power) with its dynamic
shared memory, which the compiler's report leaves out, beside its static one
within 227 KB; and no register spilled in any of them. Where a block did not
fit, a solve would leave the persistent kernel without a word."""
import os
import subprocess

import pytest

from tests.test_kernel_resources import CSRC, NVCC, ROOT, _entries, ptxas_report  # noqa: F401

LIMIT = 227 * 1024


@pytest.fixture(scope="module")
def dynamic(tmp_path_factory):
    if not os.path.exists(NVCC):
        pytest.skip("nvcc not available")
    d = tmp_path_factory.mktemp("sizes")
    src = d / "sizes.cu"
    src.write_text('#include <cstdio>\n#include "rlgl_power.cuh"\nint main() {\n'
                   '    std::printf("%zu %zu %zu %zu\\n", sizeof(rlgl::SweepSmem<float>), sizeof(rlgl::SweepSmem<double>),\n'
                   '                sizeof(rlgl::PowSmem<float>), sizeof(rlgl::PowSmem<double>));\n}\n')
    r = subprocess.run([NVCC, "-gencode", "arch=compute_103a,code=sm_103a", "-std=c++17", "-I", CSRC, "-I",
                        os.path.join(ROOT, "include"), "-o", str(d / "sizes"), str(src)], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-2000:]
    out = subprocess.run([str(d / "sizes")], capture_output=True, text=True, check=True).stdout.split()
    return dict(zip(("sweep_f", "sweep_d", "power_f", "power_d"), map(int, out)))


@pytest.mark.parametrize("prefix,kind,threads", [("_ZN4rlgl7k_sweepI", "sweep", 1024),
                                                 ("_ZN4rlgl11k_far_sweepI", "sweep", 1024),
                                                 ("_ZN4rlgl7k_powerI", "power", 768)])
def test_one_block_fits_an_sm(ptxas_report, dynamic, prefix, kind, threads):  # noqa: F811
    entries = _entries(ptxas_report, prefix)
    assert len(entries) == 4  # {float, double} x {weighted, unit weights}
    for name, regs, spill, smem in entries:
        cash = name[len(prefix)]
        assert regs * threads <= 65536, (name, regs)
        assert smem + dynamic[kind + "_" + cash] + 1024 <= LIMIT, (name, smem, dynamic)  # (1 KB is the system's)
        assert spill == 0, (name, spill)
