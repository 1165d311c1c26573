"""The 16-byte records in a CTA's shared memory start on 16-byte boundaries for every number of
pairs, nodes and precision: the bytes in front of them, from the size functions that the launches
use, evaluated on the host (no GPU)."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = r"""
#include <cstdio>
#include "bf_device.cuh"
template <int Q, class P> int bad()
{
    using T2 = bfk::Tile2<Q, P, bfk::KIND_GENRADON, false>;
    int n = 0;
    for (int k = 0; k <= 3; ++k)
        for (int T = 1; T <= 16; T *= 2) {
            const int np = T << (2 * k);
            // column pass: the geometry (two levels, then the switch's) and the parts end the allocation
            n += (T2::col_smem(np, false) - np * (T2::PSTR * sizeof(typename P::R) + 2 * sizeof(typename T2::Geo) + sizeof(int4))) % 16 != 0;
            n += (T2::col_smem(np, true) - np * (2 * sizeof(typename T2::Geo) + sizeof(int4))) % 16 != 0;
            n += (T2::row_smem(np, T, k, true) - 2 * (np >> 2) * sizeof(typename T2::GeoR)) % 16 != 0;
            const size_t boxes = (size_t)T * (((1 << (2 * k)) - 1) / 3);
            n += (T2::row_adj_smem(np, T, k) - k * (np >> 2) * sizeof(typename T2::GeoR) -
                  boxes * T2::RR * sizeof(typename T2::PH::T)) % 16 != 0;
        }
    return n;
}
template <class P> int all() { return bad<2, P>() + bad<3, P>() + bad<4, P>() + bad<5, P>() + bad<6, P>() + bad<8, P>(); }
int main() { std::printf("%d %d\n", all<bfk::PMIX>(), all<bfk::PF64>()); }
"""


def test_records_are_aligned(tmp_path):
    from paper_1305_4650_gb300 import build
    nvcc = build._nvcc()
    if not shutil.which(nvcc):
        pytest.skip("no nvcc")
    src = tmp_path / "layout.cu"
    src.write_text(SRC)
    subprocess.run([nvcc, "-std=c++17", "--expt-relaxed-constexpr", "-I", build.CSRC, "-I", os.path.join(ROOT, "include"),
                    *build.ARCH, str(src), "-o", str(tmp_path / "layout")], check=True)
    out = subprocess.run([str(tmp_path / "layout")], capture_output=True, text=True, check=True).stdout
    assert out.split() == ["0", "0"], out
