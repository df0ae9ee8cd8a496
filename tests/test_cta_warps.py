"""The rule that turns a mapping's or a server's warps per CTA into the warps
its CTAs run (cta_warps in csrc/kernels.h), over every population size: what is
accepted follows K sequences, their energies and 256 bytes a word; what is
accepted fits with the search's scratch, in the largest CTA that does."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include <cstdio>
#include "kernels.h"
int main() {
    const int words[] = {2, 3, 4, 5, 6, 8};
    for (int nw : words)
        for (int K = 1; K <= LABS_MAX_K; ++K)
            for (int least = 1; least <= 2; ++least)
                for (int wpb = least; wpb <= 8; wpb *= 2) {
                    const size_t need = (static_cast<size_t>(K) * (nw + 1) * 4 + lgpu::tabu_scratch_bytes(nw) + 15) & ~size_t{15};
                    std::printf("%d %d %d %d %d\n", nw, K, least, wpb,
                                lgpu::cta_warps(wpb, least, lgpu::warp_smem_asked(nw, K), need));
                }
}
"""


@pytest.fixture(scope="module")
def rows(tmp_path_factory):
    from paper_2504_00987_gb300 import _build

    if shutil.which("g++") is None:
        pytest.skip("no g++")
    d = tmp_path_factory.mktemp("cta_warps")
    (d / "main.cpp").write_text(PROGRAM)
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(_build.nvcc_path()))), "include")
    exe = str(d / "main")
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-I", os.path.join(ROOT, "include"), "-I", _build.CSRC,
                           "-I", cuda, str(d / "main.cpp"), "-o", exe])
    out = subprocess.check_output([exe], text=True)
    return [tuple(int(x) for x in line.split()) for line in out.splitlines()]


def test_cta_warps_over_every_population(rows):
    assert len(rows) == 6 * 1024 * (4 + 3)
    halved = 0
    for nw, K, least, wpb, got in rows:
        most = 227 * 1024 - (128 if least == 2 else 0)
        pop = 4 * K * (nw + 1)
        accepted = -(-(pop + 256 * nw) // 16) * 16 * wpb <= most
        assert (got > 0) == accepted, (nw, K, least, wpb, got)
        if not accepted:
            continue
        need = -(-(pop + 608 * nw) // 16) * 16
        assert least <= got <= wpb and need * got <= most, (nw, K, least, wpb, got)
        assert got == wpb or need * 2 * got > most, (nw, K, least, wpb, got)
        halved += got < wpb
    assert halved > 0
