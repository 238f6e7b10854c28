"""The sum by target rows is taken only where its 32-bit positions hold every row's records.

The check is the library's own host function, called from a small program.
"""
import os
import subprocess

import pytest

from conftest import ROOT

SRC = """
#include <cstdio>
#include "sfci_internal.cuh"
int main() {
    long long n, nd;
    int na, po_a, sb;
    while (std::scanf("%lld %lld %d %d %d", &n, &nd, &na, &po_a, &sb) == 5) {
        sfci::SysDev d{};
        d.na = na, d.po_a = po_a, d.sb = sb;
        std::printf("%d\\n", (int)sfci::gather_numbers(d, n, nd));
    }
    for (int bb = 1; bb <= 26; ++bb) {  // bits of a beta string's number
        sfci::GatherShape p{};
        p.bb = bb;
        const sfci::RowPlanArgs ra = sfci::row_plan_args(sfci::SysDev{}, p, 1000);
        std::printf("%llu %u\\n", ra.half, ra.w_fixed);
    }
}
"""
# sources, distinct beta strings, alpha electrons, their pairs, beta singles
CASES = {
    (1_000_000, 1_184_040, 7, 21, 147): 1,
    (100_000_000, 1_184_040, 7, 21, 147): 1,
    (20_700_000, 20_700_000, 0, 0, 204): 1,
    # one row: 204 beta singles a source fit 32 bits, with its diagonal they do not
    (21_000_000, 21_000_000, 0, 0, 204): 0,
    # many sources listed under a row's pairs, and its own beta singles
    (60_000_000, 20_000_000, 12, 66, 192): 0,
    (200_000_000, 1_000_000, 7, 21, 147): 0,
    (3_000_000_000, 100, 0, 0, 9): 0,
}


def _output(tmp_path, text):
    import importlib
    build = importlib.import_module("paper_2312_01846_gb300.build")
    try:
        lib, nvcc = build.build(), build.nvcc()
    except RuntimeError as e:  # no nvcc on this machine
        pytest.skip(str(e))
    src, exe = tmp_path / "limits.cu", tmp_path / "limits"
    src.write_text(SRC)
    subprocess.run([nvcc, *build.ARCH, *build.FLAGS, "-I", build.CSRC, str(src), lib, "-o", str(exe),
                    "-Xlinker", "-rpath=" + os.path.dirname(lib)], check=True, capture_output=True, cwd=ROOT)
    return subprocess.run([str(exe)], input=text, check=True, capture_output=True, text=True).stdout.splitlines()


def test_records_fit_their_positions(tmp_path):
    out = _output(tmp_path, "\n".join(" ".join(map(str, k)) for k in CASES))
    assert [int(x) for x in out[: len(CASES)]] == list(CASES.values())
    # in numbers: what one row may hold, against 2^32
    for (n, nd, na, po, sb), ok in CASES.items():
        assert ok == (n < 1 << 31 and n * (po + 1) + min(n, nd) * (sb + 1) < 1 << 32)


def test_rows_of_a_group_fit_their_key_bits(tmp_path):
    """A group holds at most 2 half / w_fixed rows: 120 (7 bits), and fewer than its keys can number
    beside the beta string, from one beta string (1 bit) to 2^26."""
    for bb, line in enumerate(_output(tmp_path, ""), start=1):
        half, w_fixed = map(int, line.split())
        rows = 2 * half // w_fixed
        assert w_fixed >= 32 and rows <= min(120, 2 ** (32 - bb) - 2), bb
        assert w_fixed == 32 or rows >= min(120, 2 ** (32 - bb) - 2) // 2, bb
