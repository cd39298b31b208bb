"""The rule that shapes the prologue launch of the small-batch forward and picks its kernel, compiled for the host and asked over the
range of widths, ranks, token counts and layers of a launch."""
import itertools
import os
import re
import subprocess
from collections import namedtuple

import pytest

from paper_2601_19675_b200 import build

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


def test_the_number_of_multiprocessors_counts_from_five_tokens_on(shapes):
    # the launch asks the device for it there only
    assert all(s.tpr < 8 for a, s in shapes.items() if a.T <= 4)


def test_a_row_cta_has_no_loop_for_tokens_that_are_absent(shapes):
    for a, s in shapes.items():
        assert s.tpr < 2 * min(a.T, 8)


def test_the_loop_of_eight_tokens_by_itself_runs_where_every_row_cta_starts_at_once(shapes):
    # (it leaves room for one CTA per multiprocessor); rows come before rotation within a layer and group of eight tokens
    own = {a: s for a, s in shapes.items() if s.tpr == 8 and not s.common}
    assert own
    for a, s in own.items():
        assert (s.row_ctas + s.rot_ctas) * s.groups * a.layers - s.rot_ctas <= SMS
        assert not s.pairs and not s.deep


def test_the_kernel_of_long_rows_does_not_depend_on_how_many_ctas_there_are(shapes):
    for a, s in shapes.items():
        if s.deep and s.tpr < 8 and not a.other:
            assert s.common == bool(a.fp8)


@pytest.fixture(scope="module")
def kernels(tmp_path_factory):
    """{(staged, siblings, kind, tokens of a row CTA): (registers, bytes spilled)} of the prologue kernels, as the assembler reports."""
    obj = tmp_path_factory.mktemp("obj") / "rotate.o"
    run = [build._nvcc(), *build.NVCC_FLAGS, "-Xptxas", "-v", "-I", os.path.join(ROOT, "include"), "-I", CSRC, "-c",
           os.path.join(CSRC, "rotate.cu"), "-o", str(obj)]
    text = subprocess.run(run, check=True, capture_output=True, text=True).stderr
    found = {}
    for name, stores, loads, regs in re.findall(r"entry function '(\S*prologue_kernel\S*)'.*?(\d+) bytes spill stores, (\d+) bytes spill loads"
                                                r".*?Used (\d+) registers", text, re.S):
        staged, none, kind, tpr = re.search(r"prologue_kernelILb([01])E\S*?(No)?PrologueSiblingsELi(\d)ELi(\d)E", name).groups()
        found[int(staged), none is None, ("plain", "paired", "deep")[int(kind)], int(tpr)] = (int(regs), int(stores) + int(loads))
    assert found
    return found


def test_the_common_prologue_kernels_spill_nothing_and_run_two_to_a_multiprocessor(kernels):
    for name, (regs, spilled) in kernels.items():
        if name[3] == 0:
            assert spilled == 0 and regs <= 128, name


def test_every_prologue_kernel_is_reached_and_every_shape_has_one(shapes, kernels):
    # the table of siblings is also what experts alone and layers under the switch for one kernel set carry
    reached = set()
    for a, s in shapes.items():
        kind = "paired" if s.pairs else ("deep" if s.deep else "plain")
        for table in ({True} if a.layers > 1 else {False, True}):
            reached.add((s.staged, table, kind, 0 if s.common else s.tpr))
    assert reached == set(kernels)
