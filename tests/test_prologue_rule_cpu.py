"""The rule that shapes the prologue launch of the small-batch forward and picks its kernel, compiled for the host and asked over the
range of widths, ranks, token counts and layers of a launch."""
import itertools
import os
import subprocess
from collections import namedtuple

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2601_19675_b200", "csrc")
SMS = 148

PROGRAM = r"""
#include <cstdio>
#include "prologue_rule.h"
int main() {
    int d, r, T, layers, fp8, other, sms;
    while (scanf("%d %d %d %d %d %d %d", &d, &r, &T, &layers, &fp8, &other, &sms) == 7) {
        const lopro::PrologueShape s = lopro::prologue_shape(d, r, T, layers, fp8, other, sms);
        printf("%d %d %d %d %d %d %d %d\n", s.tpr, s.row_ctas, s.rot_ctas, s.groups, s.staged, s.pairs, s.deep, s.common);
    }
}
"""
Ask = namedtuple("Ask", "d_in r_pad T layers fp8 other")
Shape = namedtuple("Shape", "tpr row_ctas rot_ctas groups staged pairs deep common")


@pytest.fixture(scope="module")
def shapes(tmp_path_factory):
    """{Ask: Shape} over the range: the FP8 record and other products run layers alone, group sizes are those of a launch."""
    there = tmp_path_factory.mktemp("rule")
    src, exe = there / "rule.cpp", there / "rule"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    asks = [Ask(*a) for a in itertools.product((64, 512, 1024, 2048, 4096, 8192, 11008, 16384, 28672),
                                               (0, 16, 32, 48, 64, 96, 128, 256), range(1, 33), (1, 2, 3, 4, 8), (0, 1), (0, 1))
            if not (a[3] > 1 and (a[4] or a[5])) and not (a[4] and a[5])]
    text = "\n".join(" ".join(map(str, (*a, SMS))) for a in asks)
    out = subprocess.run([str(exe)], input=text, check=True, capture_output=True, text=True).stdout.split("\n")
    return {a: Shape(*map(int, line.split())) for a, line in zip(asks, out)}


def test_row_ctas_cover_every_row_and_token_once(shapes):
    for a, s in shapes.items():
        rows = 2 if s.pairs else 1
        assert s.groups == -(-a.T // 8) and s.tpr in (1, 2, 4, 8)
        assert s.row_ctas == a.r_pad // rows * -(-min(a.T, 8) // s.tpr)


def test_a_row_cta_has_no_loop_for_tokens_that_are_absent(shapes):
    for a, s in shapes.items():
        assert s.tpr < 2 * min(a.T, 8)
