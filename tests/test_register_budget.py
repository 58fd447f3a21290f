"""Registers that nvcc gives a kernel whose speed rests on two CTAs sharing an SM (no GPU needed)."""
import re
import shutil
import subprocess

import pytest

from paper_2609_32420_b200 import build


@pytest.mark.skipif(shutil.which("nvcc") is None, reason="nvcc is not on PATH")
def test_two_ctas_of_the_selecting_kernel_fit_an_sm(tmp_path):
    """score_select_kernel reads key-block means under another CTA's selection: two CTAs of sixteen rows (512 threads) share 65536
    registers, 64 a thread; rows of 257 to 640 blocks run in two CTAs of eight, 128 a thread.  With 76 instead of 64, rows of 161 to 256
    blocks took 9 to 14 % longer (48 heads of 256 blocks, D = 64, mass 0.5: 101 and 88 us)."""
    forms = [(D, 16, NPL) for D in (64, 128) for NPL in (2, 4, 5, 8)] + [(D, 8, 20) for D in (64, 128)]
    src = tmp_path / "forms.cu"
    src.write_text('#include "common.cuh"\n#include "builder.cuh"\nnamespace carnator {\n' + "".join(
        f"template __global__ void score_select_kernel<{D}, {R}, {NPL}>(const float*, const float*, float*, float, SelectArgs);\n" for D, R, NPL in forms) + "}\n")
    flags = [f for f in build.NVCC_FLAGS if f != "--shared"]
    out = subprocess.run(["nvcc", *flags, "-Xptxas", "-v", "-c", "-o", str(tmp_path / "forms.o"), str(src)], capture_output=True, text=True)
    assert out.returncode == 0, out.stderr
    used = re.findall(r"Compiling entry function '\S*score_select_kernelILi(\d+)ELi(\d+)ELi(\d+)E\S*'.*?Used (\d+) registers", out.stderr, re.S)
    assert sorted((int(D), int(R), int(NPL)) for D, R, NPL, _ in used) == sorted(forms), out.stderr
    assert all(int(n) <= 65536 // (2 * 32 * int(R)) for _, R, _, n in used), used
