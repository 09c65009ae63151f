"""What the compiler gives the kernels that run at the limit of their registers.

The launch-per-class refresh keeps two CTAs of 256 threads on an SM, 128
registers a thread, and its FP32 form needs all of them: with its cluster size a
run-time value it spilled 60 / 80 bytes (stores / loads) instead of 12 / 16 and
took 2.3 % longer per cell.
"""
import os
import re
import subprocess

import pytest

from paper_2312_04998_gb300 import build


@pytest.fixture(scope="module")
def usage(tmp_path_factory):
    """source -> [(mangled kernel name, registers, spill stores, spill loads)]"""
    out = {}

    def of(name):
        if name not in out:
            obj = str(tmp_path_factory.mktemp("ptxas") / "k.cubin")
            cmd = [build._nvcc()] + build.ARCH + build.FLAGS + ["-Xptxas", "-v", "-cubin", "-o", obj,
                                                                os.path.join(build.CSRC, name)]
            log = subprocess.run(cmd, capture_output=True, text=True, check=True).stderr
            out[name] = [(k, int(regs), int(st), int(ld)) for k, st, ld, regs in re.findall(
                r"Compiling entry function '(\S+)'.*?(\d+) bytes spill stores, (\d+) bytes spill loads.*?"
                r"Used (\d+) registers", log, re.S)]
        return out[name]
    return of


def test_fp32_refresh_has_the_registers_it_needs(usage):
    rows = [r for r in usage("integrate.cu") if "refresh_kernel" in r[0]]
    assert len(rows) == 3
    f32 = [r for r in rows if "refresh_kernelIf" in r[0]]
    assert len(f32) == 1   # one CTA a cell: no cluster form
    assert f32[0][1] <= 128 and f32[0][2] <= 16 and f32[0][3] <= 16, f32


def test_sell_gather_has_a_form_for_full_sms(usage):
    """32 registers: 2048 threads on an SM.  (With 72 alone, batches that fill the
    device took up to 11 % longer.)"""
    rows = [r for r in usage("kern_rhs.cu") if "rhs_sell_kernel" in r[0]]
    assert min(r[1] for r in rows) <= 32 and all(r[2] == r[3] == 0 for r in rows), rows
