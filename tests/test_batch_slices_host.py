"""The batch kernel's slices of a CTA's shared memory, compiled for the host: groups that can be at
work at the same time never overlap, for every on-chip budget and block size."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_0908_4520_gb300", "csrc")

CHECK = r"""
#include <cstdio>
#include "lb_batch_slices.h"
using namespace lbk;

int main() {
    long long bad = 0;
    for (int nwarp = 2; nwarp <= 16; ++nwarp)
        for (int cap = 0; cap <= 227 * 1024; ++cap) {
            const BatchSlice cta = batch_slice(kBatchCta, 0, cap, nwarp);
            bad += cta.offset != 0 || cta.bytes > cap || cta.bytes < cap - 15;
            int end = 0;  // of the warp before
            for (int w = 0; w < nwarp; ++w) {
                const BatchSlice s = batch_slice(kBatchWarp, w, cap, nwarp);
                bad += s.offset % 16 || s.bytes % 16 || s.bytes < 0 || s.offset < end || s.offset + s.bytes > cap;
                end = s.offset + s.bytes;
                if (nwarp % 4 != 0) continue;
                // a warp lies inside its own four-warp group and so outside every other one
                const BatchSlice g = batch_slice(kBatchQuad, w / 4 * 4, cap, nwarp);
                bad += g.offset % 16 || s.offset < g.offset || end > g.offset + g.bytes;
                if (w % 4 == 3) bad += end != g.offset + g.bytes;
            }
        }
    std::printf("%lld\n", bad);
    return bad != 0;
}
"""


def test_slices_of_neighbouring_groups_are_disjoint(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no host compiler")
    (tmp_path / "check.cpp").write_text(CHECK)
    exe = tmp_path / "check"
    subprocess.run([cxx, "-std=c++17", "-O2", "-I", CSRC, str(tmp_path / "check.cpp"), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0 and r.stdout.strip() == "0", r.stdout
