"""Resident blocks of the moments' kernel, from the compiler's register counts:
the walls' gather of 2-byte storage is bound by latency, and with 122 registers
instead of 80 (two blocks of 256 threads per SM instead of three) it ran a
quarter longer."""
import os
import re
import subprocess

from paper_1411_3133_gb300 import build

SOURCE = '''#include "%s/kernels.cuh"
using namespace lbgm;
#define MACROS(S, R, K) \\
  template __global__ void lbgm::k_macros<S, R, K>(const S* __restrict__, double* __restrict__, double* __restrict__, Dims);
MACROS(__half, float, KELL)
MACROS(__nv_bfloat16, float, KELL)
MACROS(__half, float, KCYL)
MACROS(float, float, KELL)
'''


def test_moments_of_2byte_storage_hold_three_blocks_per_sm(tmp_path):
    src = tmp_path / "macros.cu"
    src.write_text(SOURCE % build.CSRC)
    cmd = [build._nvcc()] + build.ARCH + build.NVCC_FLAGS + ["-I", os.path.join(build.ROOT, "include"), "-c", str(src),
                                                             "-o", str(tmp_path / "macros.o")]
    res = subprocess.run(cmd, capture_output=True, text=True)
    assert res.returncode == 0, res.stderr
    found = re.findall(r"Compiling entry function '(\w*k_macros\w*)'.*?Used (\d+) registers", res.stdout + res.stderr, re.S)
    assert len(found) == 4
    for name, regs in found:
        assert 65536 // (256 * (-(-int(regs) // 8) * 8)) >= 3, (name, regs)
