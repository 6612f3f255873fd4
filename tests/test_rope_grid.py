"""How the rotary append divides its tokens among CTAs (csrc/rope_grid.h), on the CPU."""
import ctypes
import os
import subprocess

import pytest

from paper_2412_07017_b200 import build as lib_build

PROBE = """
#include "rope_grid.h"
extern "C" int tokens(int total, int heads, int d) { return asynclm::rope_tokens(total, heads, d); }
extern "C" int threads(int t, int heads, int d) { return asynclm::rope_threads(t, heads, d); }
extern "C" int smem(int t) { return (int)asynclm::rope_smem(t); }
"""


@pytest.fixture(scope="module")
def grid(tmp_path_factory):
    d = tmp_path_factory.mktemp("rope_grid")
    src, lib = os.path.join(d, "probe.cpp"), os.path.join(d, "probe.so")
    with open(src, "w") as f:
        f.write(PROBE)
    subprocess.run(["g++", "-std=c++17", "-shared", "-fPIC", "-I", lib_build.CSRC, "-o", lib, src], check=True)
    return ctypes.CDLL(lib)


# (tokens, heads that are rotated, head_dim) -> tokens of a CTA, where another choice was measured to be slower
@pytest.mark.parametrize("total,heads,d,want", [
    (1, 40, 128, 1), (444, 40, 128, 1), (445, 40, 128, 2), (1200, 40, 128, 3), (2048, 40, 128, 5), (8192, 40, 128, 19), (8880, 40, 128, 20),
    (520, 40, 64, 1), (520, 18, 128, 1), (520, 8, 128, 1), (520, 4, 64, 1), (520, 10, 64, 2), (592, 40, 64, 1), (593, 40, 64, 2), (700, 40, 64, 2),
    (2000, 8, 64, 4), (2000, 40, 64, 5),
    (8881, 40, 128, 4), (13999, 72, 128, 4), (14000, 72, 128, 8), (65536, 40, 128, 8), (9500, 40, 64, 8), (9500, 8, 64, 4), (65536, 8, 64, 4),
    (65536, 4, 64, 4)])
def test_tokens_of_a_cta(grid, total, heads, d, want):
    assert grid.tokens(total, heads, d) == want


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("heads", [1, 4, 8, 10, 18, 40, 72, 144, 300])
def test_up_to_a_wave_is_one_wave(grid, heads, d):
    """Up to 20 tokens for each CTA of a wave, a grid is about a wave of at least a warp each, and never more tokens than there is room for."""
    for total in list(range(1, 2300)) + list(range(8000, 9000)) + [1 << 20]:
        t = grid.tokens(total, heads, d)
        assert 1 <= t <= 20 and 32 <= grid.threads(t, heads, d) <= 256 and grid.threads(t, heads, d) % 32 == 0
        ctas = -(-total // t)
        if total <= 444 * 20:
            assert ctas <= 444 or (ctas <= 592 and grid.threads(t, heads, d) <= 160)
        assert grid.smem(t) >= t * (64 * 16 + 8) and grid.smem(t) <= 48 << 10
