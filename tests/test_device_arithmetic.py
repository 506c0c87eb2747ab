"""Index arithmetic that host and kernels share, compiled for the host (nvcc needs no GPU) and checked against Python's integers."""

import os
import random
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2609_07536_b200", "csrc")


def _compiled(tmp_path, body):
    nvcc = next((c for c in (os.environ.get("NVCC"), "/usr/local/cuda/bin/nvcc", shutil.which("nvcc")) if c and os.path.exists(c)), None)
    if nvcc is None:
        pytest.skip("no nvcc")
    src = tmp_path / "arith.cu"
    src.write_text(f'#include <cstdio>\n#include "{CSRC}/moe_internal.h"\nint main()\n{{\n{body}\n}}\n')
    exe = tmp_path / "arith"
    subprocess.run([nvcc, "-std=c++17", "-gencode", "arch=compute_100a,code=sm_100a", "-cudart", "static", "-o", str(exe), str(src)], check=True)
    return exe


def _run(exe, rows):
    text = "\n".join(" ".join(str(v) for v in r) for r in rows) + "\n"
    out = subprocess.run([str(exe)], input=text, check=True, capture_output=True, text=True).stdout.split()
    assert len(out) == len(rows)
    return [int(v) for v in out]


def test_rows_of_y_beyond_32_bits(tmp_path):
    # element offsets of a unit over all that shape_ok lets through (T * k_tot < 2^30, L <= 8): T * L passes 2^31 and 2^32
    exe = _compiled(tmp_path, '    int t, s, c, L, w, k;\n    while (scanf("%d %d %d %d %d %d", &t, &s, &c, &L, &w, &k) == 6)\n'
                              '        printf("%zu\\n", moe::y_unit(t, s, c, L, w, k));\n    return 0;')
    rng = random.Random(1)
    rows = [((1 << 28) - 1, 7, 0, 8, 8, 1), (1 << 28, 0, 0, 8, 8, 1), ((1 << 29) - 1, 7, 0, 8, 8, 1), (1 << 29, 0, 0, 8, 8, 1), ((1 << 30) - 1, 7, 128, 8, 264, 1)]
    for _ in range(500):
        k, L = rng.randint(1, 32), rng.randint(1, 8)
        rows.append((rng.randrange((1 << 30) // k), rng.randrange(L), 128 * rng.randint(0, 60), L, 8 * rng.randint(1, 4000), k))
    assert _run(exe, rows) == [((t * L + s) * w + c) * k for t, s, c, L, w, k in rows]


def test_places_of_the_operand_maps(tmp_path):
    # one launch's maps, and those of buffers a power of two of bytes apart, never share a place (they would be encoded on every call)
    exe = _compiled(tmp_path, '    unsigned long long p; int b;\n    while (scanf("%llu %d", &p, &b) == 2)\n'
                              '        printf("%u\\n", moe::map_place(reinterpret_cast<const void *>(p), b));\n    return 0;')
    rng = random.Random(2)
    boxes, pairs = (32, 64, 96, 128, 256), [(0x7f0000000000 + 256 * rng.randrange(1 << 28), 1 << j) for j in range(8, 35) for _ in range(4)]
    got = _run(exe, [(q, b) for p, d in pairs for q in (p, p + d) for b in boxes])
    assert all(0 <= v < 128 for v in got)
    for i in range(len(pairs)):
        one, other = got[10 * i:10 * i + 5], got[10 * i + 5:10 * i + 10]
        assert len(set(one)) == 5 and not set(one[:4]) & set(other[:4]), (hex(pairs[i][0]), pairs[i][1])
