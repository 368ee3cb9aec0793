"""Which strides the tensor maps over a token grid take: `tok_grid_exists`, as the library has it, against what a map of five dimensions asks for (strides
that do not decrease, below 2^40 bytes; those of single heads and entries are free)."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2312_08874_b200", "csrc")
CUDA = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "include")

PROGRAM = r"""
#include <cstdio>
#include "kernels.h"
using namespace aa;
typedef unsigned long long u64;

static bool map_exists(const TokLayout& l, int batch, int heads, u64 H, u64 W) {
    const bool heads_first = heads > 1 && l.sh < l.st;
    const u64 st = 2 * l.st, row = st * W, slab = row * H;
    u64 sh = 2 * l.sh, sb = 2 * l.sb;
    if (heads == 1 && sh < slab) sh = slab;
    const u64 entry = heads_first ? slab : sh * heads;
    if (batch == 1 && sb < entry) sb = entry;
    const u64 a[4] = {heads_first ? sh : st, heads_first ? st : row, heads_first ? row : sh, sb};
    for (int i = 0; i < 4; ++i)
        if (a[i] >= 1ull << 40 || (i && a[i] < a[i - 1])) return false;
    return true;
}
int main() {
    long long with = 0, without = 0, wrong = 0;
    for (int B = 1; B <= 3; ++B) for (int h = 1; h <= 4; ++h) for (int H = 1; H <= 5; H += 2) for (int W = 1; W <= 9; W += 4) for (int d = 8; d <= 64; d += 56) {
        const long long N = H * W, c[] = {d, 2 * d, h * d, 3 * h * d, N * d, N * h * d, 3 * N * h * d, B * d, B * h * d, N * B * d, N * B * h * d, W * d, W * h * d};
        for (long long sb : c) for (long long sh : c) for (long long st : c) {
            const TokLayout l = {sb, sh, st};
            bool hf;
            unsigned long long n[2], s[3];
            const bool tokens = tok_map_dims(l, B, h, N, &hf, n, s), got = tok_grid_exists(l, B, h, H, W), want = tokens && map_exists(l, B, h, H, W);
            (want ? with : without)++;
            if (got != want && wrong++ < 5) printf("B %d heads %d grid %d x %d d %d strides %lld %lld %lld: %d, want %d\n", B, h, H, W, d, sb, sh, st, got, want);
        }
    }
    printf("with %lld without %lld wrong %lld\n", with, without, wrong);
    return wrong != 0 || with < 1000 || without < 1000;
}
"""


@pytest.mark.skipif(shutil.which("g++") is None or not os.path.isdir(CUDA), reason="needs g++ and the CUDA headers")
def test_grid_maps_are_claimed_where_they_exist(tmp_path):
    src = tmp_path / "maps.cpp"
    src.write_text(PROGRAM)
    exe = tmp_path / "maps"
    subprocess.run(["g++", "-O1", "-std=c++17", "-I", CSRC, "-I", CUDA, str(src), "-o", str(exe)], check=True, timeout=300)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout
