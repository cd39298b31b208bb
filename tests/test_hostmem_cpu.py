"""The rule for host buffers that kernels read and write in place, compiled for the host: the one pinned piece that holds the
first byte has to hold the last one and all between."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include <cstdio>
#include <initializer_list>
#include "hostmem.h"
int main() {
    using lopro::HostRange;
    using lopro::holds_whole_buffer;
    const HostRange cases[] = {
        {0x1000, 0x1000, 0x3000},              // the allocation itself
        {0x1800, 0x1000, 0x3000},              // a part of it
        {0x1000, 0x1000, 0x1000},              // the first of two registered pages, the one between them not registered
        {0, 0, 0},                             // pageable
        {0x1000, 0x1000, 0},                   // a device address, but no range known
        {0x1000, 0x2000, 0x3000},              // addresses of different spaces
        {~0ull - 0xfff, ~0ull - 0xfff, 0x800}  // at the end of the address space
    };
    for (const HostRange& r : cases)
        for (unsigned long long bytes : {0ull, 16ull, 0x1000ull, 0x2800ull, 0x2801ull, 0x3000ull, 0x3010ull, ~0ull})
            printf("%d", (int)holds_whole_buffer(r, bytes));
    printf("\n");
}
"""


def test_only_a_buffer_inside_one_pinned_piece_is_taken_in_place(tmp_path):
    src, exe = tmp_path / "rule.cpp", tmp_path / "rule"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-I", os.path.join(ROOT, "paper_2601_19675_b200", "csrc"), str(src), "-o", str(exe)], check=True)
    got = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.strip()
    assert got == "01111100" "01110000" "01100000" "00000000" "00000000" "00000000" "01000000"
