"""The launch rules that depend on the device's size, evaluated on the host for made-up numbers of SMs
(no GPU): threads of a single-RHS pass, pairs per thread block in FP64."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = r"""
#include <cstdio>
#include "bf_host.h"
#include "bf_inst.cuh"
static int g_sms;
namespace bfl { int sm_count() { return g_sms; } }
int main()
{
    for (int sms : {1, 76, 152, 200}) {
        g_sms = sms;
        const uint64_t n = (uint64_t)sms;
        // 64 pairs, q = 5: 320 threads, or those of up to three blocks
        std::printf("%d %u %u %u %u\n", sms, bfl::tile_threads<2, 5, bfk::PMIX>(1, 3, n, 3, 5), bfl::tile_threads<2, 5, bfk::PMIX>(1, 3, n + 1, 3, 5),
                    bfl::tile_threads<2, 5, bfk::PMIX>(1, 3, (1ull << 32) + 1, 3, 5), bfl::tile_threads<2, 5, bfk::PMIX>(1, 3, 1, 3, 2));
    }
}
"""


def run(tmp_path, src):
    from paper_1305_4650_gb300 import build
    nvcc = build._nvcc()
    if not shutil.which(nvcc):
        pytest.skip("no nvcc")
    (tmp_path / "shape.cu").write_text(src)
    subprocess.run([nvcc, "-std=c++17", "--expt-relaxed-constexpr", "-I", build.CSRC, "-I", os.path.join(ROOT, "include"),
                    *build.ARCH, str(tmp_path / "shape.cu"), "-o", str(tmp_path / "shape")], check=True)
    return subprocess.run([str(tmp_path / "shape")], capture_output=True, text=True, check=True).stdout


def test_threads_follow_the_number_of_sms(tmp_path):
    for line in run(tmp_path, SRC).splitlines():
        sms, one, more, huge, capped = (int(v) for v in line.split())
        assert (one, more, huge, capped) == (960, 320, 320, 640), line


PAIRS = r"""
#include <cstdio>
#include "bf_host.h"
static int g_sms;
namespace bfl { int sm_count() { return g_sms; } }
int main()
{
    bfl::PassFns two{}, one{};
    two.kmax = 2; two.np = 32;    // FP64 at d = 2: two tiles of 16 pairs
    one.kmax = 3; one.np = 64;    // one tile
    for (int sms : {60, 152}) {
        g_sms = sms;
        for (int L = 1; L <= 8; ++L)
            std::printf("%d %d %d %d\n", sms, L, (int)bfl::single_pairs(&two, 2, 1ll << (2 * L)), (int)bfl::single_pairs(&one, 2, 1ll << (2 * L)));
    }
}
"""


def test_fp64_blocks_hold_one_tile_where_sms_would_idle(tmp_path):
    for line in run(tmp_path, PAIRS).splitlines():
        sms, L, two, one = (int(v) for v in line.split())
        assert one == 64
        assert two == (16 if 4 ** L // 16 <= sms else 32), line
