"""Which form the gate+up projection on bf16 weights takes (host code, no GPU needed): one wave of wide tiles only where that was
measured to be the quicker one."""
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2603_01399_b200", "csrc")

PROGRAM = r'''
#include <stdio.h>
#include "tc_dual.h"
int main() {
  long long m, n, k;
  while (scanf("%lld %lld %lld", &m, &n, &k) == 3) printf("%d\n", quasar::dual_channels(m, n, k));
  return 0;
}
'''


@pytest.fixture(scope="module")
def channels(tmp_path_factory):
    where = tmp_path_factory.mktemp("rule")
    src, exe = where / "rule.cpp", where / "rule"
    src.write_text(PROGRAM)
    subprocess.check_call(["g++", "-std=c++17", "-I", CSRC, str(src), "-o", str(exe)])

    def ask(cases):
        text = "".join("%d %d %d\n" % c for c in cases)
        return [int(x) for x in subprocess.run([str(exe)], input=text, text=True, check=True, capture_output=True).stdout.split()]

    return ask


def test_wide_tiles_where_they_won(channels):
    cases = [(m, 24576, 4096) for m in (1, 2, 4, 6, 8)] + [(8, 19072, 4096), (8, 28672, 4096), (3, 22016, 3584), (8, 24576, 5120)]
    cases += [(m, n, k) for m in (1, 8) for n, k in ((19072, 4096), (22016, 3600), (30784, 4096), (37888, 1024))]   # as the GPU test runs them
    assert channels(cases) == [176] * 5 + [144, 208, 160, 176] + [144, 160, 208, 256] * 2


def test_tiles_of_128_where_wide_ones_lost(channels):
    cases = [(m, 34816, 5120) for m in (1, 2, 4, 6, 8)]                                       # the 14B shape: 240 channels
    cases += [(m, n, k) for m in (1, 8) for n in (34816, 37888) for k in (2048, 4096, 8192)]         # 240 and 256 channels
    cases += [(m, n, 3072) for m in (1, 8) for n in (27648, 30720)] + [(8, 30720, 2560)]             # 192 and 208, shorter contractions
    cases += [(m, 19072, k) for m in (1, 8) for k in (512, 768, 2560)] + [(1, 24576, 512)]
    cases += [(9, 24576, 4096), (64, 24576, 4096), (1, 18944, 4096), (1, 1376, 256), (0, 24576, 4096)]   # rows; tiles of 128 do
    assert channels(cases) == [0] * len(cases)


@pytest.mark.parametrize("k,least,most", [(1024, 160, 256), (2048, 160, 176), (3072, 144, 176), (4096, 144, 208), (8192, 144, 208)])
def test_the_tiles_of_one_wave(channels, k, least, most):
    """Multiples of 16 that cover all channels with at most 148 tiles."""
    cases = [(1, 2 * f, k) for f in range(9000, 20000, 16)]
    for (_, n, _), c in zip(cases, channels(cases)):
        narrowest = -(-n // (148 * 16)) * 16
        assert c == (narrowest if least <= narrowest <= most else 0)
