"""Choice of kernel for calls of at most 16 tokens (zero_filled_first in csrc/gs_plan.cu), compiled
with g++: at measured points over layer counts, sizes, densities and tokens, the kernel chosen is
the faster one or close to it."""
import math
import shutil
import subprocess
from pathlib import Path

import pytest

CSRC = Path(__file__).resolve().parent.parent / "paper_2609_33977_gb300" / "csrc"

DRIVER = r"""
#include "gs_plan.cuh"
#include <cstdio>
int main() {
  int n = 0, kw = 0, T = 0;
  while (std::scanf("%d %d %d", &n, &kw, &T) == 3) {
    std::vector<gs::FewTokenLayer> v(n);
    for (auto& l : v) {
      long long o = 0, i = 0;
      if (std::scanf("%lld %lld %lf %d %d %d", &o, &i, &l.kept_bytes, &l.chunks, &l.cpu, &l.cpu_fine) != 6) return 2;
      l.out = o;
      l.in = i;
    }
    std::printf("%d\n", (int)gs::zero_filled_first(v, kw, T, 152));
  }
  return 0;
}
"""

BLOCK_7B = [(4096, 4096)] * 4 + [(11008, 4096)] * 2 + [(4096, 11008)]
BLOCK_13B = [(5120, 5120)] * 4 + [(13824, 5120)] * 2 + [(5120, 13824)]
BLOCK_60M = [(2048, 2048), (512, 2048), (512, 2048), (2048, 2048), (8192, 2048), (8192, 2048), (2048, 8192)]

# layers, chunk width, kept fraction, tokens, us per eager call on the decode / zero-filled kernel
MEASURED = [
    ([(4096, 4096)], 256, 0.5, 1, 8.0, 9.7),
    ([(5120, 5120)], 256, 0.1, 1, 10.8, 9.8),
    ([(5120, 5120)], 256, 0.5, 16, 20.2, 11.5),
    ([(1024, 20480)], 256, 0.1, 1, 8.9, 11.2),          # few windows: all decode units resident at once
    ([(1024, 20480)], 256, 0.1, 8, 10.5, 12.2),
    ([(1024, 20480)], 256, 0.1, 16, 14.5, 12.7),
    ([(1024, 20480)], 256, 0.5, 8, 21.2, 13.1),
    ([(512, 40960)], 256, 0.05, 2, 9.5, 13.9),
    ([(4096, 5120)], 256, 0.5, 8, 9.9, 10.5),
    ([(4096, 5120)], 256, 1.0, 1, 20.4, 11.4),
    ([(20480, 1024)], 128, 0.5, 4, 19.2, 10.4),
    ([(28672, 8192)], 128, 0.1, 1, 63.9, 38.0),
    ([(1024, 4096)] * 8, 256, 0.1, 8, 16.2, 22.3),      # the host sets the pace
    ([(2048, 2048)] * 8, 256, 0.1, 16, 27.9, 17.8),
    (BLOCK_60M, 256, 0.5, 8, 28.2, 18.0),
    (BLOCK_7B, 256, 0.2, 1, 47.2, 29.7),                # sparse: the decode kernel's walk
    (BLOCK_7B, 256, 0.5, 16, 47.9, 39.6),
    (BLOCK_7B, 128, 0.5, 1, 59.7, 41.6),
    (BLOCK_13B, 256, 0.5, 1, 61.0, 55.6),
    (BLOCK_13B, 256, 0.1, 1, 57.8, 40.4),
    ([(2048, 2048)] * 9, 256, 0.1, 1, 19.1, 29.3),      # a second launch for one layer
    ([(2048, 2048)] * 16, 256, 0.5, 1, 29.9, 38.0),
    ([(1024, 1024)] * 32, 256, 0.5, 8, 53.7, 67.7),
    ([(1024, 1024)] * 32, 128, 0.5, 8, 53.8, 69.0),
    ([(2048, 2048)] * 32, 256, 0.5, 16, 53.8, 73.5),
    ([(1024, 4096)] * 32, 256, 0.5, 1, 54.5, 76.0),
    (BLOCK_7B * 2, 256, 0.1, 1, 63.5, 56.8),
    (BLOCK_7B * 2, 128, 0.5, 4, 114.8, 80.7),
    (BLOCK_60M * 2, 128, 0.2, 1, 66.2, 35.6),
    ([(4096, 4096)] * 16, 256, 0.85, 16, 108.3, 79.3),
]


def plan(out, inp, kw, d):
    """Kept bytes, chunks and the decode kernel's chunks per unit, as packing sets them."""
    chunks, blocks = inp // kw, -(-out // 64)
    kept = round(d * out * chunks)
    splits = math.floor(2.0 * kw * kept / blocks / (224 * 1024) + 0.5)
    splits = min(chunks, max(splits, 1, -(-chunks // 64)))
    cpu = -(-chunks // splits)
    return f"{out} {inp} {2.0 * kw * kept} {chunks} {cpu} {max(1, cpu // 4)}"


@pytest.fixture(scope="module")
def choose(tmp_path_factory):
    gxx = shutil.which("g++")
    if not gxx:
        pytest.skip("g++ not available")
    d = tmp_path_factory.mktemp("rule")
    (d / "main.cpp").write_text(DRIVER)
    exe = d / "rule"
    subprocess.run([gxx, "-std=c++17", "-O2", "-x", "c++", str(CSRC / "gs_plan.cu"), str(d / "main.cpp"), "-x", "none",
                    f"-I{CSRC}", "-o", str(exe)], check=True, capture_output=True)

    def run(layers, kw, density, T):
        inp = f"{len(layers)} {kw} {T}\n" + "\n".join(plan(o, i, kw, density) for o, i in layers) + "\n"
        return int(subprocess.run([str(exe)], input=inp, capture_output=True, text=True, check=True).stdout)
    return run


@pytest.mark.parametrize("case", MEASURED, ids=lambda c: f"{len(c[0])}x{c[0][0][0]}x{c[0][0][1]}-{c[1]}-d{c[2]}-T{c[3]}")
def test_the_faster_kernel_is_chosen(choose, case):
    layers, kw, density, T, decode_us, zero_filled_us = case
    chosen = zero_filled_us if choose(layers, kw, density, T) else decode_us
    assert chosen <= 1.04 * min(decode_us, zero_filled_us)


def test_small_layers_stay_on_the_decode_kernel(choose):
    for T in (1, 8, 16):
        assert not choose([(1024, 1024)], 256, 0.5, T)
        assert not choose([(1024, 1024)] * 9, 128, 0.5, T)
        assert not choose([(4096, 4096)], 128, 1.0, T)
