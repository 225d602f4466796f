"""The barrier phases of a kernel with two accumulators in turn (csrc/mma_phase.h),
against a model of the two mbarriers: a parity wait passes when the phase of that
parity is the one before the current. After a wait that gave up, tiles may be in
flight; the wait for the last of them must pass exactly when all of them are done
(tensor memory is freed after it). A wait with a fixed parity does not do that.
"""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_1312_4746_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include "mma_phase.h"
struct Bars {
    uint32_t phase[2] = {0, 0};  // completed phases
    explicit Bars(uint32_t done) { for (uint32_t t = 0; t < done; ++t) ++phase[t & 1]; }
    bool passes(uint32_t bar, uint32_t parity) const { return (phase[bar] & 1u) != parity; }
};
int main() {
    int bad = 0, fixed_passes_early = 0;
    MmaPhase p{};
    if (mma_last(0, p)) ++bad;
    for (uint32_t issued = 1; issued <= 64; ++issued)
        // a tile is issued once the second one before it has been waited for
        for (uint32_t done = issued < 2 ? 0 : issued - 2; done <= issued; ++done) {
            const Bars b(done);
            if (!mma_last(issued, p) || b.passes(p.bar, p.parity) != (done == issued)) ++bad;
            if (done < issued && b.passes(0, 0) && b.passes(1, 0)) ++fixed_passes_early;
            for (uint32_t t = done; t < issued; ++t)  // waits in order: tile t - 1 is done
                if (t == done && b.passes(mma_phase(t).bar, mma_phase(t).parity)) ++bad;
            if (done && !b.passes(mma_phase(done - 1).bar, mma_phase(done - 1).parity)) ++bad;
        }
    std::printf("%d %d\n", bad, fixed_passes_early);
    return 0;
}
"""


def test_drain_waits_for_every_tile(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no host compiler")
    src, exe = tmp_path / "phase.cpp", tmp_path / "phase"
    src.write_text(PROGRAM)
    subprocess.run([cxx, "-std=c++17", "-Wall", "-Werror", "-I", CSRC, str(src), "-o", str(exe)],
                   check=True)
    bad, fixed = map(int, subprocess.run([str(exe)], check=True, capture_output=True,
                                         text=True).stdout.split())
    assert bad == 0
    assert fixed > 0  # what a parity of 0, whatever was issued, would let through
