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


@pytest.mark.parametrize("fp8,gated,K,n_feat,E,R,small", [
    # whole steps of which one side was measured at least 2 % faster, per pass (csrc/rules.h has the times)
    (0, 1, 512, 2048, 8, 1100, 0), (0, 1, 768, 512, 128, 100, 0), (0, 1, 1024, 512, 64, 192, 0), (0, 1, 1024, 512, 64, 400, 0),
    (0, 1, 1024, 512, 512, 24, 1), (0, 1, 1024, 512, 512, 160, 1), (0, 1, 1024, 256, 256, 40, 1), (0, 1, 1024, 256, 256, 300, 1),
    (0, 1, 1280, 768, 128, 160, 1), (0, 1, 1536, 512, 128, 300, 1), (0, 1, 2048, 768, 128, 72, 1), (0, 1, 2048, 768, 128, 144, 1),
    (0, 1, 2048, 768, 512, 24, 1), (0, 1, 2048, 768, 512, 48, 1), (0, 1, 2048, 768, 512, 96, 1), (0, 1, 2048, 768, 512, 160, 1),
    (0, 1, 2048, 768, 4, 2100, 0), (0, 1, 7168, 512, 8, 1100, 0), (0, 1, 7168, 512, 8, 2000, 1),
    (0, 1, 7168, 2048, 256, 750, 1), (0, 1, 7168, 2048, 256, 1500, 1),
    (0, 0, 256, 2048, 128, 160, 0), (0, 0, 512, 1536, 128, 200, 0), (0, 0, 512, 1024, 64, 192, 0), (0, 0, 768, 2048, 128, 144, 1),
    (0, 0, 768, 2048, 512, 48, 1), (0, 0, 768, 2048, 128, 200, 0), (0, 0, 1024, 1792, 128, 160, 1), (0, 0, 1024, 1792, 128, 600, 0),
    (0, 0, 2048, 7168, 256, 256, 1), (0, 0, 2048, 512, 8, 1100, 0),
    (1, 1, 1024, 256, 256, 64, 0), (1, 1, 1536, 512, 128, 72, 0), (1, 1, 2048, 768, 128, 120, 0), (1, 1, 2048, 768, 128, 220, 0),
    (1, 1, 2048, 768, 512, 24, 1), (1, 1, 2048, 768, 512, 48, 1), (1, 1, 2048, 256, 128, 80, 0), (1, 1, 2560, 1536, 128, 250, 1),
    (1, 1, 2560, 1536, 128, 350, 0), (1, 1, 4096, 1536, 128, 600, 1), (1, 1, 7168, 2048, 256, 1024, 1), (1, 1, 3072, 768, 128, 160, 1),
    (1, 1, 2560, 768, 64, 250, 0), (1, 1, 4096, 512, 128, 160, 1), (1, 1, 4096, 512, 32, 800, 0), (1, 1, 7168, 512, 8, 1100, 0),
    (1, 0, 1024, 2560, 512, 140, 1), (1, 0, 1024, 2560, 512, 220, 0), (1, 0, 1536, 2560, 128, 200, 0), (1, 0, 2048, 7168, 256, 750, 0),
])
def test_the_kernel_that_was_measured_faster_is_chosen(rules, fp8, gated, K, n_feat, E, R, small):
    assert rules(f"moe::small_m_is_faster({fp8}, {gated}, {K}, {n_feat}, {R * E}LL, {E}, 148)") == [small]


@pytest.mark.parametrize("H,I,E,k,Is,T,ctas,at_once", [
    # whole steps measured in one launch and in three, at least 2 % apart unless at the edge of a line (csrc/rules.h)
    (256, 512, 8, 2, 0, 64, 148, 1), (256, 128, 8, 2, 0, 64, 148, 1), (64, 64, 32, 16, 0, 64, 148, 1), (448, 320, 16, 10, 0, 47, 148, 0),  # 128 | 144 tiles
    (320, 192, 4, 4, 64, 64, 148, 1), (64, 64, 32, 32, 0, 32, 148, 0), (128, 64, 64, 32, 1024, 12, 148, 0),                             # top-32
    (6592, 128, 128, 12, 0, 1, 148, 1), (6592, 128, 128, 32, 0, 6, 148, 0), (704, 640, 64, 2, 0, 6, 148, 1),                              # 12 slots
    (2048, 768, 128, 8, 0, 3, 148, 1), (1024, 256, 64, 8, 0, 3, 148, 1), (1024, 256, 64, 8, 0, 4, 148, 0), (1024, 960, 64, 2, 0, 14, 148, 0),
    (768, 1792, 128, 4, 64, 7, 148, 0), (4160, 576, 32, 8, 0, 3, 148, 0), (704, 2112, 64, 16, 0, 1, 148, 1), (704, 2112, 64, 16, 0, 2, 148, 0),
    (512, 512, 16, 4, 0, 4, 148, 1), (192, 512, 24, 4, 0, 8, 148, 0), (256, 256, 32, 8, 0, 64, 148, 0), (256, 256, 32, 16, 0, 64, 148, 0),
    (4992, 2048, 4, 4, 2048, 11, 148, 0), (4928, 576, 8, 8, 576, 7, 148, 1), (1024, 2048, 4, 2, 0, 64, 148, 1), (1024, 2048, 8, 8, 0, 64, 148, 0),
    (4096, 256, 16, 4, 0, 32, 148, 1), (4096, 256, 16, 4, 0, 33, 148, 0), (960, 640, 16, 8, 0, 31, 148, 0), (1024, 512, 16, 8, 0, 64, 148, 0),
    (7168, 2048, 256, 8, 2048, 64, 148, 1), (2560, 1024, 512, 8, 0, 64, 148, 1), (4096, 1536, 128, 8, 0, 48, 148, 1),
    (4096, 1536, 128, 8, 0, 49, 148, 0), (2048, 768, 128, 8, 0, 5, 148, 1), (2048, 768, 128, 8, 0, 6, 148, 0), (2048, 768, 128, 8, 0, 37, 148, 0),
    (1536, 1536, 64, 8, 0, 8, 148, 0), (1024, 2048, 64, 8, 0, 16, 148, 0), (7168, 1024, 64, 16, 1024, 12, 148, 1), (7168, 1024, 64, 16, 1024, 13, 148, 0),
    # on part of the SMs: few tiles only
    (7168, 2048, 256, 8, 2048, 64, 100, 0), (7168, 2048, 256, 8, 2048, 1, 100, 0), (256, 512, 8, 2, 0, 64, 100, 1), (1024, 256, 64, 8, 0, 1, 48, 1),
])
def test_the_steps_made_in_one_launch(rules, H, I, E, k, Is, T, ctas, at_once):
    assert rules(f"moe::step_at_once_is_faster({T}, {k}, {E}, {H}, {I}, {Is}, {ctas}, {int(ctas == 148)})") == [at_once]


def test_the_rows_that_the_gated_pass_gathers(rules):
    """Above 8192 rows (up to there moving them hides behind the pass's set-up), below 256 rows an expert, and few feature tiles beside
    what the launch saves."""
    cases = [(8192, 128, 2048, 256, 0), (8193, 128, 2048, 256, 1), (256 * 128 - 1, 128, 2048, 512, 1), (256 * 128, 128, 2048, 512, 0),
             (8447, 33, 512, 512, 1), (8193, 32, 2048, 256, 0), (1531 * 8, 128, 2048, 768, 1), (2300 * 8, 128, 2048, 768, 1),
             (2600 * 8, 128, 2048, 768, 0), (4096 * 8, 512, 2560, 1024, 1), (11000 * 8, 512, 2560, 1024, 0), (3300 * 8, 128, 4096, 1536, 0),
             (1500 * 6, 64, 2048, 1408, 0), (2600 * 6, 64, 2048, 1408, 0), (4096 * 8, 256, 7168, 2048, 1), (6000 * 8, 256, 7168, 2048, 0),
             (200 * 256, 256, 7168, 1792, 1), (100 * 256, 256, 1024, 576, 0)]
    assert rules(*[f"moe::gather_is_faster({rows}LL, {E}, {H}, {I})" for rows, E, H, I, _ in cases]) == [c[-1] for c in cases]
