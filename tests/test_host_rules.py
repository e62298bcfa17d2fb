"""Rules of the kernels that are plain host and device functions, compiled with nvcc and run on
the CPU: the entries of a tile's run labels that the label of a site reads."""
import subprocess

import pytest

from paper_1405_1931_gb300 import build

LABELS = r"""
#include <cstdio>
#include <cstdlib>
#include <vector>
#include "hk_device.cuh"
// a tile's run labels: the entries of one row are [first, first + n); any other read is counted
struct Checked {
    int first, n;
    mutable long outside = 0;
    __host__ __device__ int operator[](int i) const {
        if (i < first || i >= first + n) ++outside;
        return 1000 + i;
    }
};
int main() {
    std::vector<unsigned> words = {0u, ~0u, 1u, 1u << 31, 0x55555555u, 0xaaaaaaaau, 0x7ffffffeu, 0x80000001u};
    srand(7);
    for (int i = 0; i < 5000; ++i) words.push_back(((unsigned)rand() << 17) ^ ((unsigned)rand() << 2) ^ (unsigned)rand());
    long outside = 0, wrong = 0;
    for (unsigned m : words)
        for (int first : {0, 1, 37}) {
            const unsigned rs = m & ~(m << 1);
            const Checked lab{first, __builtin_popcount(rs)};
            int run = first - 1;
            for (int x = 0; x < 32; ++x) {
                if ((rs >> x) & 1u) ++run;
                const int want = (m >> x) & 1u ? 1000 + run : -1;
                if (hk::site_label(m, rs, first, hk::le_mask(x), lab) != want) ++wrong;
            }
            outside += lab.outside;
        }
    printf("%ld %ld\n", outside, wrong);
}
"""


def host_program(tmp_path, source):
    src, exe = tmp_path / "rule.cu", tmp_path / "rule"
    src.write_text(source)
    subprocess.run([build.nvcc(), "-std=c++17", "-O1", *build.ARCH, "-I", build.CSRC, "-o", str(exe), str(src)], check=True)
    return subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout


def test_site_label_reads_its_rows_entries_only(tmp_path):
    assert host_program(tmp_path, LABELS).split() == ["0", "0"]
