"""Shared-memory layout of the tensor-core operators, computed on the host: every
warp's slab starts with floats, so its offset has to be a multiple of their size
at every order the operators accept."""
import subprocess

from paper_2608_24348_gb300 import build

SRC = r"""
#include <cstdio>
#include <cuda_runtime.h>
#include "ax_tc.cuh"
template <int NP> static void row()
{
    using A = TcCfg<NP>; using B = TcSplitCfg<NP>;
    printf("%d %d %zu %d %zu\n", NP, (int)A::OK, A::PER_ELEM, (int)B::OK, B::PER_ELEM);
}
int main() { row<2>(); row<3>(); row<4>(); row<5>(); row<6>(); row<7>(); row<8>(); row<9>(); row<10>(); }
"""


def test_warp_slabs_are_aligned_for_their_floats(tmp_path):
    src, exe = tmp_path / "layout.cu", tmp_path / "layout"
    src.write_text(SRC)
    subprocess.run([build.nvcc(), *build.ARCH, "-std=c++17", "--expt-relaxed-constexpr", "-I", build.CSRC,
                    str(src), "-o", str(exe)], check=True, capture_output=True)
    rows = [[int(v) for v in line.split()] for line in
            subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.splitlines()]
    assert [r[0] for r in rows] == list(range(2, 11))
    for n, ok, per, ok_split, per_split in rows:
        if ok:
            assert per % 4 == 0, n
        if ok_split:
            assert per_split % 4 == 0, n
