"""The host's rules (csrc/rules.h), compiled by themselves."""
import os
import subprocess

import pytest

from paper_2609_00993_b200 import build as build_mod


@pytest.fixture(scope="module")
def rules(tmp_path_factory):
    """rules("expression", ...) -> the expressions' values, as integers."""
    d = tmp_path_factory.mktemp("rules")

    def evaluate(*exprs):
        src, exe = d / "r.cc", d / "r"
        src.write_text('#include <cstdio>\n#include "rules.h"\nint main() {\n' +
                       "".join(f'  printf("%lld\\n", (long long)({e}));\n' for e in exprs) + "}\n")
        subprocess.run(["g++", "-std=c++17", "-Wall", "-Werror", "-I", build_mod.CSRC, str(src), "-o", str(exe)], check=True)
        return [int(v) for v in subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split()]

    return evaluate


def test_layout_reads_stay_linear_in_the_batch(rules):
    """Chunks are whole warp steps, fit the scratch (a row of counts per 256 slots) and are never more than one CTA per SM
    once a chunk has 4096 slots: every CTA reads every chunk's counts, so more of them cost with the square."""
    sizes = [1, 1023, 1024, 1025, 16384, 16385, 65536, 65537, 262144, 262145, 148 * 4096, 148 * 4096 + 1, 1 << 22, (1 << 27) + 5,
             1 << 30]
    cases = [(n, E) for n in sizes for E in (1, 64, 512, 513, 1024)]
    for (n, E), chunk in zip(cases, rules(*[f"moe::layout_chunk_slots({n}LL, {E})" for n, E in cases])):
        chunks = -(-n // chunk)
        assert chunk % 1024 == 0 and chunk < 1 << 31
        assert chunks * E <= max(1, -(-n // 256)) * E
        assert chunks <= 148 or chunk < 4096, (n, E, chunk)
        assert chunks ** 2 * E * 4 <= 148 ** 2 * 1024 * 4
