"""Rules of the product dispatch (csrc/dispatch.h), compiled for the host: the
sizes where they change, among them sectors whose vectors no test allocates."""
import math
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2105_06806_gb300", "csrc")


def _run(tmp_path, body):
    cc = shutil.which("g++")
    if cc is None:
        pytest.skip("no host C++ compiler")
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text('#include <cstdio>\n#include "dispatch.h"\nint main() {\n%s\n}\n' % body)
    subprocess.run([cc, "-std=c++17", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    return [int(x) for x in subprocess.run([str(exe)], capture_output=True, text=True,
                                           check=True).stdout.split()]


def test_rows_kernel_within_its_32_bit_units(tmp_path):
    """k_hv_rows divides its work unit in 32 bits: it takes FP32 sectors above 2^22
    elements of which every unit is below 2^32, no others (Ns=20 sectors next to
    half filling have 4-6e9 units: their last rows would never be written)."""
    def units(ddw, stride):
        return -(-ddw // 4) * stride

    ns20 = [(math.comb(20, b), -(-math.comb(20, a) // 4) * 4)
            for a in range(7, 12) for b in range(7, 12)]
    shapes = ns20 + [(48620, 48632), (3432, 3432), (2048, 2048), (2048, 2052),
                     (4 * 65536, 65536), (4 * 65536 + 1, 65536), (4 * 65536 - 3, 65536), (1, 64)]
    calls = [(e, d, s) for d, s in shapes for e in (4, 8)]
    got = _run(tmp_path, "\n".join('printf("%%d\\n", (int)ed_takes_rows(%d, %dLL, %dLL));' % c
                                   for c in calls))
    want = [int(e == 4 and d * s > 2 ** 22 and units(d, s) <= 2 ** 32) for e, d, s in calls]
    assert got == want
    assert units(math.comb(20, 9), math.comb(20, 8)) > 2 ** 32
    for (e, d, s), g in zip(calls, got):
        if g:  # the largest unit's row and column survive the 32-bit division
            u = units(d, s) - 1
            assert ((u & 0xffffffff) // s, (u & 0xffffffff) % s) == (u // s, u % s)
