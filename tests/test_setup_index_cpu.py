"""Sizes and indexes that the setup's kernels compute, on the CPU and at
values that no test problem reaches: the header that holds them is compiled
with the host compiler and called."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def values(tmp_path, *expressions):
    """The integer expressions, evaluated with csrc/setup_index.h."""
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("g++ not found")
    src, exe = tmp_path / "values.cpp", tmp_path / "values"
    src.write_text('#include <cstdio>\n#include "setup_index.h"\nusing namespace airg;\nint main() {\n' +
                   "".join('  std::printf("%%lld\\n", (long long)(%s));\n' % e for e in expressions) + "}\n")
    r = subprocess.run([gxx, "-std=c++17", "-Wall", "-Werror",
                        "-I", os.path.join(ROOT, "paper_2508_17517_gb300", "csrc"), str(src), "-o", str(exe)],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0
    return [int(v) for v in r.stdout.split()]


def test_sparse_product_table_sizes(tmp_path):
    """A table is a power of two, at least twice the columns that the row can
    have (its products or the matrix's columns, whichever are fewer), and the
    size is found for every count: the products saturate at 2^30 - 1."""
    cases = [(769, 10**6), (769, 2600), (10**6, 2600), (2**29, 2**31 - 1), (2**29 + 1, 2**31 - 1),
             (2**30 - 1, 2**31 - 1), (2**30 - 1, 1000), (2**30 - 1, 2**29), (1, 1)]
    got = values(tmp_path, *["gemm_table_slots(%dLL, %dLL)" % c for c in cases])
    for (products, n_cols), size in zip(cases, got):
        most = min(products, n_cols)
        assert size & (size - 1) == 0 and 2 * most <= size < 4 * most, (products, n_cols, size)
    # 32-bit offsets: what is refused, and the bound on a piece
    assert values(tmp_path, "gemm_table_slots(1LL << 29, 2147483647) <= GEMM_MAX_SLOTS",
                  "gemm_table_slots((1LL << 29) + 1, 2147483647) <= GEMM_MAX_SLOTS",
                  "gemm_piece_limit(-5)", "gemm_piece_limit(4096)", "gemm_piece_limit(1LL << 40)") == \
        [1, 0, 1, 4096, 2**30]


def test_warp_per_row_index(tmp_path):
    """Row of a thread where one warp takes a row, up to 2^31 rows: with
    blocks of 256 threads the thread number passes 2^32 at row 2^27."""
    rows = [0, 7, 8, 2**27 - 1, 2**27, 2**27 + 9, 2**31 - 1]
    assert values(tmp_path, *["warp_index(%du, 256u, %du)" % (r // 8, r % 8 * 32 + 31) for r in rows]) == rows
