"""The least that the row lists of a sigma take, known before they are made, against a count of
every row's entries.

The bound is the library's own host function, called from a small program.
"""
import itertools
import math
import os
import subprocess

import numpy as np
import pytest

from conftest import ROOT

SRC = """
#include <cstdio>
#include "sfci_internal.cuh"
int main() {
    int n, na, sa, sb, po_a, bb;
    long long m;
    while (std::scanf("%d %d %d %d %d %d %lld", &n, &na, &sa, &sb, &po_a, &bb, &m) == 7) {
        sfci::SysDev d{};
        sfci::GatherShape p{};
        d.n = n, d.na = na, d.sa = sa, d.sb = sb, d.po_a = po_a, d.ss_any = d.ab_any = 1, p.bb = bb;
        std::printf("%zu\\n", sfci::gather_lists_least(d, p, m));
    }
}
"""
CASES = [(6, 0, 2), (6, 1, 3), (6, 2, 2), (7, 3, 3), (7, 7, 2), (8, 6, 4), (16, 2, 8)]


def _count(n, na, nb, m):
    """Records and one-hop sources of all rows, for m sources of random alpha strings."""
    strings = [sum(1 << o for o in c) for c in itertools.combinations(range(n), na)]
    rng = np.random.default_rng(n)
    src = [strings[i] for i in rng.integers(0, len(strings), m)]
    occ = {s: [o for o in range(n) if s >> o & 1] for s in strings}
    by1, by2 = {}, {}
    for s in src:
        for x in occ[s]:
            by1.setdefault(s ^ 1 << x, []).append(s)
        for x, y in itertools.combinations(occ[s], 2):
            by2.setdefault(s ^ 1 << x ^ 1 << y, []).append(s)
    rec = ab = 0
    for t in strings:
        own = src.count(t)
        hops = sum(len(by1.get(t ^ 1 << x, [])) for x in occ[t]) - na * own
        rec += hops + own * (1 + nb * (n - nb))
        rec += sum(len(by2.get(t ^ 1 << x ^ 1 << y, [])) for x, y in itertools.combinations(occ[t], 2))
        ab += hops
    return rec, ab


def test_least_is_what_all_rows_hold(tmp_path):
    import importlib
    build = importlib.import_module("paper_2312_01846_gb300.build")
    try:
        lib, nvcc = build.build(), build.nvcc()
    except RuntimeError as e:  # no nvcc on this machine
        pytest.skip(str(e))
    src, exe = tmp_path / "lists.cu", tmp_path / "lists"
    src.write_text(SRC)
    subprocess.run([nvcc, *build.ARCH, *build.FLAGS, "-I", build.CSRC, str(src), lib, "-o", str(exe),
                    "-Xlinker", "-rpath=" + os.path.dirname(lib)], check=True, capture_output=True, cwd=ROOT)
    m, lines, want = 50, [], []
    for n, na, nb in CASES:
        bits = max(1, (math.comb(n, nb) - 1).bit_length())
        lines.append(f"{n} {na} {na * (n - na)} {nb * (n - nb)} {na * (na - 1) // 2} {bits} {m}")
        rec, ab = _count(n, na, nb, m)
        want.append(rec * (24 if bits > 12 else 12) + 16 * ab)  # (rows in classes: their records twice)
    out = subprocess.run([str(exe)], input="\n".join(lines), check=True, capture_output=True, text=True).stdout
    assert [int(x) for x in out.split()] == want
