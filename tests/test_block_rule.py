"""The rule that picks the form of the sliced deterministic block, against measured times.

Setup on one GB300 in ms, with the Gram matrix on the orbitals and with the contraction over
the kept pairs (N_aux = 3N); the sizes where the two differ by more than 7%.  Host arithmetic
only."""
import subprocess

from paper_2005_12338_gb300 import build

# n, n_occ, n_tau, kept pairs, orbitals, pairs
MEASURED = [
    (90, 36, 64, 2142, 6.2, 38.4), (110, 61, 8, 1230, 4.28, 7.05), (126, 63, 16, 3088, 7.06, 17.1),
    (129, 52, 64, 3073, 29.3, 84.5), (129, 64, 16, 4643, 11.0, 30.7), (131, 39, 64, 1517, 30.9, 69.5),
    (131, 59, 4, 3203, 7.56, 9.31), (131, 72, 8, 1517, 7.74, 11.99), (160, 48, 64, 1826, 56.0, 80.8),
    (200, 60, 64, 2414, 126.6, 136.5), (200, 80, 64, 7556, 120.1, 230.5),
    (230, 92, 64, 5796, 204.3, 260.7), (230, 115, 16, 5796, 64.9, 74.0),
    (250, 100, 64, 6236, 265.2, 300.3), (257, 103, 64, 9635, 420.1, 576.3),
    (257, 128, 16, 6303, 135.0, 123.0), (270, 148, 32, 6766, 212.9, 228.6),
    (272, 109, 64, 6768, 502.6, 444.1), (272, 109, 64, 10324, 502.9, 584.9),
    (288, 115, 64, 7296, 596.4, 517.2), (288, 136, 16, 7296, 191.6, 145.4),
    (320, 128, 64, 12300, 845.9, 920.0), (320, 128, 64, 8130, 845.8, 708.7),
    (360, 180, 16, 13746, 436.7, 360.0), (400, 160, 16, 15320, 821.3, 534.2),
    (450, 180, 16, 17260, 1328.4, 763.1),
]


def test_the_faster_form_is_taken(tmp_path):
    src, exe = tmp_path / "check.cu", tmp_path / "check"
    calls = "".join(f'  std::printf("%d\\n", (int)rssri::mo_block_pays_sliced({n}, {o}, {3 * n}, {p}, {t}));\n'
                    for n, o, t, p, _, _ in MEASURED)
    src.write_text('#include <cstdio>\n#include "mo.cuh"\nint main() {\n' + calls + "}\n")
    subprocess.run([build.nvcc(), "-std=c++17", "-I", build.CSRC, "-I", build.INCLUDE, str(src),
                    "-o", str(exe)], check=True)
    got = subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout.split()
    for m, g in zip(MEASURED, got, strict=True):
        assert (g == "1") == (m[4] < m[5]), m
