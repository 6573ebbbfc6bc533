"""The registers that let a decode CTA run beside an append CTA on one SM.

A sub-partition has 512 registers per lane. The append kernel puts three of its
twelve warps on each, the decode kernel one of its four; registers are given to a
warp in steps of eight per lane. No cap in the sources states that sum (a cap of
136 on the append kernel makes the compiler choose a slower schedule of fewer
registers), so it is checked on what the compiler reports."""
import os
import re
import subprocess

import pytest

from paper_2608_22167_gb300 import build

PER_LANE = 512


def _registers(source, kernel, tmp_path):
    """Registers and spilled bytes of every instantiation of `kernel`."""
    cmd = [build.nvcc()] + build._flags(True) + ["-cubin", "-o", str(tmp_path / "x.cubin"),
                                                 os.path.join(build.CSRC, source)]
    log = subprocess.run(cmd, capture_output=True, text=True, check=True).stderr
    found = re.findall(r"Compiling entry function '(\w+)'.*?(\d+) bytes spill stores.*?Used (\d+) registers", log, re.S)
    return {name: (int(regs), int(spilled)) for name, spilled, regs in found if kernel in name}


def test_decode_cta_fits_beside_an_append_cta(tmp_path):
    try:
        build.nvcc()
    except RuntimeError as e:
        pytest.skip(str(e))
    append = _registers("append_tc.cu", "append_tc_kernelILb0", tmp_path)  # not the self-test's form
    decode = _registers("decode.cu", "decode_kernel", tmp_path)
    assert len(append) == 2 and len(decode) == 5, (append, decode)
    decode = {k: v for k, v in decode.items() if not re.search("ILi[67]E", k)}  # wide cascade items: decode steps only
    assert not any(spilled for _, spilled in [*append.values(), *decode.values()]), (append, decode)
    up = lambda regs: -(-regs // 8) * 8  # noqa: E731
    most = 3 * up(max(r for r, _ in append.values())) + up(max(r for r, _ in decode.values()))
    assert most <= PER_LANE, (append, decode)
