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


def test_sector_order_detour_rule(tmp_path):
    """The sector-order FP32 product goes through block-major order only where that was
    measured faster, never with a scratch above 2 GiB, and follows a pinned kernel."""
    M, G = 1 << 20, 1 << 30
    cases = [  # norb, group, dup, dim, bdim, pinned, want
        (2, 7, 3432, 11778624, 11806080, -1, 0),   # Norb=2 Ns=14 (7,7): slower
        (2, 8, 12870, 165636900, 165791340, -1, 1),  # Norb=2 Ns=16 (8,8)
        (3, 5, 6435, 41409225, 41460705, -1, 1),   # Norb=3 Ns=15 (7,7)
        (3, 5, 5005, 15030015, 15100000, -1, 1),
        (3, 5, 3003, 19324305, 19400000, -1, 0),
        (4, 4, 11440, 91611520, 92000000, -1, 1), (4, 4, 8008, 102951200, 103200000, -1, 0),
        (4, 4, 12870, 7207200, 7300000, -1, 1),
        (5, 3, 6435, 41409225, 41900000, -1, 0),   # five orbitals
        (2, 0, 48620, 200000000, 201000000, -1, 0),  # no factorised product
        (3, 6, 48620, 2363904400, 2364487840, -1, 0),  # Norb=3 Ns=18: 19 GB of scratch
        (3, 6, 48620, 2363904400, 2364487840, 0, 0),
        (2, 8, 8008, G // 4, G // 4, -1, 1), (2, 8, 8008, G // 4, G // 4 + 1, -1, 0),
        (2, 8, 5000, 5 * M, 5 * M, -1, 1), (2, 8, 5000, 5 * M - 1, 5 * M, -1, 0),
        (2, 8, 4999, 5 * M, 5 * M, -1, 0), (2, 8, 11000, M, M, -1, 1),
        (2, 8, 11000, M - 1, M, -1, 0),
        (4, 4, 11000, 32 * M, 32 * M, -1, 1), (4, 4, 11000, 32 * M - 1, 32 * M, -1, 0),
        (4, 4, 12000, 32 * M - 1, 32 * M, -1, 1), (4, 4, 10999, 32 * M, 32 * M, -1, 0),
        (2, 7, 2002, 6012006, 6030000, 0, 1), (2, 7, 2002, M - 1, M, 0, 0),  # tiled pinned
        (5, 3, 3003, M, M, 0, 1), (2, 8, 12870, 165636900, 165791340, 1, 0),  # pinned
    ]
    got = _run(tmp_path, "\n".join(
        'printf("%%d\\n", (int)ed_takes_permuted(%d, %d, %dLL, %dLL, %dLL, %d));' % c[:6]
        for c in cases))
    assert got == [c[6] for c in cases]


def test_size_classes_of_the_autotuner(tmp_path):
    """Three classes in FP32 (up to 2^20 padded elements, up to 13 * 2^20, above), one in
    FP64; the half-filled sector of every Ns shares its class with the neighbours that a
    solve visits (rows padded by at most 1%)."""
    sizes = [2 ** 17 + 4, 2 ** 20 - 1, 2 ** 20, 13 * 2 ** 20 - 1, 13 * 2 ** 20, 2 ** 31, 2 ** 40]
    solves = []
    for n in range(12, 21):
        h = n // 2
        for up, dw in ((h, h), (h + 1, h), (h - 1, h), (h, h + 1), (h, h - 1)):
            d = math.comb(n, up) * math.comb(n, dw)
            solves += [d, d * 101 // 100]
    every = sizes + solves
    got = _run(tmp_path, "\n".join('printf("%%d %%d\\n", ed_tune_class(4, %dLL), ed_tune_class(8, %dLL));'
                                    % (x, x) for x in every))
    f32, f64 = got[::2], got[1::2]
    assert f32[:len(sizes)] == [0, 0, 1, 1, 2, 2, 2]
    assert f64 == [0] * len(every)
    of_solves = f32[len(sizes):]
    for k in range(0, len(of_solves), 10):
        assert len(set(of_solves[k:k + 10])) == 1
