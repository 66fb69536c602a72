"""Registers of the point path's search kernels: a lane's adds are long dependent chains, so
the kernel lives on warps in flight, and every instantiation has to leave room for 32 of them
on an SM (65,536 registers, given out 256 at a time to a warp)."""
import os
import re
import subprocess
import tempfile

from paper_2302_01293_gb300 import build


def test_point_kernels_leave_room_for_32_warps():
    nvcc = os.path.join(build._cuda_home(), "bin", "nvcc")
    with tempfile.TemporaryDirectory() as tmp:
        log = subprocess.run([nvcc, *build.ARCH, "-O3", "-std=c++17", "-Xcompiler", "-fPIC", "-Xptxas", "-v",
                              "-I" + os.path.join(build.ROOT, "include"), "-I" + build.CSRC, "-cubin",
                              os.path.join(build.CSRC, "bls_kernels.cu"), "-o", os.path.join(tmp, "k.cubin")],
                             stdout=subprocess.PIPE, stderr=subprocess.STDOUT, check=True).stdout.decode()
    found = re.findall(r"Compiling entry function '\w*bls_kernelILi(\d)ELi(\d)ELi(\d+)E.*?Used (\d+) registers",
                       log, flags=re.S)
    assert len(found) == 24
    for phase, summ, warps, regs in found:
        per_warp = (int(regs) * 32 + 255) // 256 * 256
        blocks = 65536 // (per_warp * int(warps))
        assert blocks * int(warps) >= 32, (phase, summ, warps, regs)
