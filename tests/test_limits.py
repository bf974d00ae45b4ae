"""Size rules of the host side at sizes no run here can reach, compiled from
their header alone (CPU only)."""
import os
import shutil
import subprocess

import pytest

from paper_2501_13051_gb300 import build as B


def values(tmp_path, exprs):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    src = tmp_path / "limits.cpp"
    lines = "".join('  std::printf("%%llu\\n", (unsigned long long)(%s));\n' % e for e in exprs)
    src.write_text('#include <cstdio>\n#include "limits.h"\nusing namespace cdl;\nint main() {\n%s}\n' % lines)
    exe = tmp_path / "limits"
    subprocess.run([cxx, "-std=c++17", "-Wall", "-Werror", "-I", B.CSRC, str(src), "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout
    return [int(x) for x in out.split()]


def test_direct_entries(tmp_path):
    cases = [(b, n, lim) for b in (1, 16, 17, 20, 27, 28, 29, 30, 31, 32)
             for n in (0, 1, 1 << 14, (1 << 15) - 1, 1 << 15, 1 << 18, 1 << 25, 1 << 27, 1 << 29, 1 << 30, (1 << 32) - 1)
             for lim in (False, True)]
    got = values(tmp_path, ["direct_entries(%d, %dull, %s)" % (b, n, "true" if lim else "false")
                            for b, n, lim in cases])
    for (b, n, lim), g in zip(cases, got):
        want = 1 << b
        if want > 65536 and (lim or want > 4 * n or 8 * want > 4 << 30):
            want = 0
        assert g == want, (b, n, lim)
        assert g < 1 << 32 and 8 * g <= max(32 * n, 512 << 10)
    # 2^32 keys do not fit the 32-bit number of entries: rows or not, the hash form
    assert [g for (b, n, lim), g in zip(cases, got) if b == 32] == [0] * 22


def test_graph_set_rows(tmp_path):
    cases = [(n, t) for t in (0, 1, 8) for n in (0, 1, 8192, 8193, 1 << 20, (1 << 29) - 1, 1 << 29, (1 << 29) + 1,
                                                 1 << 31, (1 << 32) - 1)]
    got = values(tmp_path, ["graph_set_rows(%dull, %d)" % c for c in cases])
    most = (1 << 32) - 1
    for (n, t), g in zip(cases, got):
        assert g == (most if t == 0 else min(most, max(1 << 16, t * n))), (n, t)
        assert g >= n  # (Full fits when the graph begins)
