"""Registers that nvcc gives a kernel whose speed rests on two CTAs sharing an SM (no GPU needed)."""
import re
import shutil
import subprocess

import pytest

from paper_2609_32420_b200 import build


@pytest.mark.skipif(shutil.which("nvcc") is None, reason="nvcc is not on PATH")
def test_two_ctas_of_sixteen_rows_fit_an_sm(tmp_path):
    """score_select_kernel reads key-block means under another CTA's selection: two CTAs of 512 threads share 65536 registers, 64 a
    thread.  With 76, rows of 161 to 256 blocks took 9 to 14 % longer (48 heads of 256 blocks, D = 64, mass 0.5: 101 and 88 us)."""
    forms = [(D, NPL) for D in (64, 128) for NPL in (2, 4, 5, 8)]
    src = tmp_path / "forms.cu"
    src.write_text('#include "common.cuh"\n#include "builder.cuh"\nnamespace carnator {\n' + "".join(
        f"template __global__ void score_select_kernel<{D}, 16, {NPL}>(const float*, const float*, float*, float, SelectArgs);\n" for D, NPL in forms) + "}\n")
    flags = [f for f in build.NVCC_FLAGS if f != "--shared"]
    out = subprocess.run(["nvcc", *flags, "-Xptxas", "-v", "-c", "-o", str(tmp_path / "forms.o"), str(src)], capture_output=True, text=True)
    assert out.returncode == 0, out.stderr
    used = {m.group(1): int(m.group(2)) for m in re.finditer(r"Compiling entry function '(\S*score_select_kernel\S*)'.*?Used (\d+) registers", out.stderr, re.S)}
    assert len(used) == len(forms), out.stderr
    assert all(n <= 65536 // (2 * 512) for n in used.values()), used
