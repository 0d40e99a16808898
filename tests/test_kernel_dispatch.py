"""CPU checks of the rules by which a kernel picks one of its compiled loops:
the rule's own source, compiled for the host."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
NVCC = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"

PROGRAM = r"""
#include <cstdio>
#include "sw_warp.cuh"

// The loop over directions of a pass that with_directions has picked, on rows
// that hold 1 where L p has been written, 0 where not and 2 for the row that
// the pass reads in any case; the lowest and the number of those it reads.
struct Pass {
    int nd, km;
    const int *const *row;
    int *low, *read;
    template <class ND> __host__ __device__ void operator()(ND) const
    {
        for (int l = 0; l < km; ++l)
            if (l < (ND::value ? ND::value : nd)) {
                *low = *row[l] < *low ? *row[l] : *low;
                *read += *row[l] == 1;
            }
    }
};

template <int KM, bool ONE>
void all()
{
    for (int nd = 0; nd <= KM; ++nd) {
        int lp[KM], other = 2, low = 9, read = 0;
        const int *row[KM];
        for (int l = 0; l < KM; ++l) {
            lp[l] = l < nd;
            row[l] = ONE ? sw::direction_row<int>(l, nd, &lp[l], &other) : &lp[l];
        }
        sw::with_directions<KM, ONE>(nd, Pass{nd, KM, row, &low, &read});
        std::printf("%d %d\n", low, read);
    }
}

int main()
{
    all<4, false>();
    all<4, true>();
    all<8, false>();
    return 0;
}
"""


@pytest.mark.skipif(not os.path.exists(NVCC), reason="needs nvcc")
def test_a_pass_reads_written_directions_only(tmp_path):
    """L(e) with nd directions reads those nd rows of L p and no other: before
    the first one has been written, none."""
    from paper_2103_16120_gb300 import build
    src, exe = tmp_path / "directions.cu", tmp_path / "directions"
    src.write_text(PROGRAM)
    subprocess.run([NVCC, *build.ARCH, "-std=c++17", "-I", build.INCLUDE, "-I", build.CSRC, str(src), "-o", str(exe)],
                   check=True, capture_output=True, text=True)
    out = subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout.split()
    got = [(int(a), int(b)) for a, b in zip(out[::2], out[1::2])]
    assert len(got) == 5 + 5 + 9
    assert all(low >= 1 for low, _ in got)               # nothing unwritten
    assert [n for _, n in got] == [*range(5), *range(5), *range(9)]
