"""The plain-FMA GEMMs' addresses at sizes past 32 bits: one long segment's [T, f] activations may have more than 2^31
elements (T = 800 000 at f = 2752), and a row may be long.  The kernels' own offset functions, compiled for the host."""
import os
import re
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2405_03133_b200", "csrc")
TILES = [(0, 1, 0), (799872, 2752, 2736), ((1 << 30) - 128, 1, 0), ((1 << 30) - 128, 4096, 4032), (48, 1 << 28, 16)]
IN_TILE = [(0, 1, 0), (127, 500, 15), (15, 2752, 127), (127, (1 << 24) - 1, 127), (127, 1 << 24, 127), (127, (1 << 31) - 1, 15)]


@pytest.mark.skipif(shutil.which("nvcc") is None, reason="needs nvcc")
def test_offsets_past_32_bits(tmp_path):
    src = tmp_path / "offset.cu"
    body = "".join(f'printf("%ld\\n", fma_offset<true>({r}, {ld}, {c}));' for r, ld, c in TILES)
    body += "".join(f'printf("%ld\\n", fma_wide({ld}) ? fma_offset<true>({r}, {ld}, {c}) : fma_offset<false>({r}, {ld}, {c}));'
                    for r, ld, c in IN_TILE)
    body += "".join(f'printf("%ld\\n", (long)(fma_row((const float*)0 + {c}, {r}, (size_t){ld} * 4) - (const float*)0));'
                    for r, ld, c in TILES + IN_TILE)
    src.write_text('#include <stdio.h>\n#include "fma_gemm.cuh"\nusing namespace lory;\nint main() {' + body + "}\n")
    exe = tmp_path / "offset"
    subprocess.run(["nvcc", "-std=c++17", "-gencode", "arch=compute_100a,code=sm_100a", "-I" + CSRC,
                    "-I" + os.path.join(ROOT, "include"), str(src), "-o", str(exe)], check=True, capture_output=True, text=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split()
    assert [int(v) for v in out] == [r * ld + c for r, ld, c in 2 * (TILES + IN_TILE)]


def test_kernels_multiply_no_row_by_a_row_length_in_32_bits():
    with open(os.path.join(CSRC, "fma_gemm.cuh")) as f:
        assert not re.search(r"(?<!\(size_t\))\b\w+ \* J\.ld[ab]", f.read())
