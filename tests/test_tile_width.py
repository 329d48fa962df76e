"""The tile width a dense product takes by default (csrc/tile_width.h), against times measured on GB300 (us per width,
GELU-distributed BF16 operands): at most 6 % over the width with the fewest padded columns, the rule of linear products
before the one by N alone, and at most 16 % over the latter, at the sizes where the two are furthest apart, with
FP32 (linear) and with BF16 GELU outputs. The width changes no output bit."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2312_05800_gb300", "csrc")

# M, N, K, GELU, {width: us}
TIMES = [
    (4096, 176, 1144, 0, {64: 9.6, 128: 12.7, 160: 14.5, 208: 15.6, 256: 16.1}),
    (4096, 352, 1144, 0, {64: 16.6, 128: 13.9, 160: 15.9, 208: 18.6, 256: 21.4}),
    (4096, 1144, 1144, 0, {128: 22.5, 160: 24.4, 208: 28.6, 256: 32.8}),
    (20000, 896, 400, 0, {64: 47.3, 128: 50.9, 160: 53.4, 208: 55.1, 256: 60.8}),
    (126000, 640, 1144, 0, {64: 399.5, 128: 302.6, 160: 286.5, 208: 341.2, 256: 315.9}),
    (126000, 704, 1144, 0, {64: 441.0, 128: 407.3, 160: 395.8, 208: 382.1, 256: 342.5}),
    (126000, 800, 1144, 0, {64: 516.8, 128: 413.7, 160: 358.9, 208: 374.3, 256: 407.4}),
    (126000, 808, 1144, 0, {64: 516.2, 128: 406.4, 160: 429.2, 208: 356.5, 256: 395.1}),
    (126000, 1600, 1144, 0, {128: 767.4, 160: 685.1, 208: 690.5, 256: 673.3}),
    (4096, 176, 1144, 1, {64: 10.0, 128: 11.4, 160: 12.9, 208: 13.3, 256: 13.8}),
    (4096, 1144, 1144, 1, {128: 20.8, 160: 22.2, 208: 25.8, 256: 29.0}),
    (126000, 640, 1144, 1, {64: 366.9, 128: 239.3, 160: 217.4, 208: 263.3, 256: 243.4}),
    (126000, 704, 1144, 1, {64: 405.7, 128: 314.9, 160: 310.4, 208: 289.6, 256: 257.7}),
    (126000, 800, 1600, 1, {64: 681.6, 128: 391.3, 160: 288.9, 208: 248.1, 256: 250.2}),
]

HARNESS = r"""
#include <cstdio>
#include "tile_width.h"
int main() {
    long M;
    int N, K, g;
    while (std::scanf("%ld %d %d %d", &M, &N, &K, &g) == 4)
        std::printf("%d %d %d\n", chemgb::product_tile_width(M, N, K, g, 152), chemgb::padded_tile_width(N),
                    chemgb::default_tile_width(N));
}
"""


def test_default_width_loses_to_neither_rule(tmp_path):
    src, exe = tmp_path / "w.cc", tmp_path / "w"
    src.write_text(HARNESS)
    subprocess.run(["g++", "-std=c++17", "-I" + CSRC, str(src), "-o", str(exe)], check=True)
    text = "\n".join("%d %d %d %d" % c[:4] for c in TIMES)
    out = subprocess.run([str(exe)], input=text, capture_output=True, text=True, check=True).stdout.splitlines()
    assert len(out) == len(TIMES)
    for c, line in zip(TIMES, out):
        pick, padded, by_n = (c[4][int(v)] for v in line.split())
        assert pick <= 1.06 * padded and pick <= 1.16 * by_n, (c, line)
