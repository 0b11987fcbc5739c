"""The potential's form where some coupling A_k is exactly 1 (lambda far below dx):
potential.cu, compiled with the host's undefined-behaviour checks, forms it
without a conversion out of range.
"""
import os
import shutil
import subprocess
import textwrap

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1910_05180_gb300", "csrc")

MAIN = textwrap.dedent("""
    #include "host_internal.h"
    #include <math.h>
    #include <stdio.h>
    int main()
    {
        double A[13], E[13], b[13];
        for (int top = 0; top < 13; ++top)
            for (int fp32 = 0; fp32 < 2; ++fp32) {
                for (int k = 0; k < 13; ++k) {
                    A[k] = k >= top ? 1.0 : 0.2 + 0.05 * k;
                    E[k] = k >= top ? 0x1p-80 : 1.0 - A[k];
                    b[k] = 1.0 / 13;
                }
                spfm_host::Rational r;
                spfm_host::build_rational(A, E, b, 13, fp32 != 0, r);
                for (int i = 0; i <= r.deg; ++i)
                    if (r.deg && !isfinite(r.den[i])) return 1;
            }
        puts("done");
        return 0;
    }
""")


def test_no_conversion_out_of_range(tmp_path):
    gxx, nvcc = shutil.which("g++"), shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not gxx or not os.path.exists(nvcc):
        pytest.skip("no compiler")
    src, exe = tmp_path / "main.cu", str(tmp_path / "main")
    src.write_text(MAIN)
    flags = ["-std=c++17", "-O1", "-I", CSRC, "-I", os.path.join(ROOT, "include")]
    for f in ("undefined", "float-cast-overflow"):
        flags += ["-Xcompiler", "-fsanitize=" + f]
    flags += ["-Xcompiler", "-fno-sanitize-recover=all"]
    subprocess.run([nvcc, *flags, str(src), os.path.join(CSRC, "potential.cu"), "-o", exe], check=True)
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0 and "done" in r.stdout, r.stderr
