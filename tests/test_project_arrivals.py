"""The projection's pairs of CTAs: every arrival that a CTA sends to its peer's mbarrier is waited for before the peer can end, and every
wait has its arrivals.  The rule is the kernel's own, compiled for the host; no GPU is needed."""
import os
import subprocess

from paper_2407_13885_b200 import build

PROGRAM = r"""
#include "project_qk.cuh"
#include <cstdio>

using namespace attnw::proj;

int main() {
    long long sent = 0;
    for (int pairs : {1, 2, 3, 66, 74}) {
        for (int items = 1; items <= 6 * pairs + 3; ++items) {
            for (int first = 0; first < pairs && first < items; ++first) {
                int released[kSlots] = {}, waited_for[kSlots] = {};  // phases of the accumulators' barriers
                int use = 0;
                for (int t = first; t < items; t += pairs, ++use) {
                    // the issuer, in front of use `use` of a slot: as many phases as the slot has had uses
                    waited_for[use % kSlots] = use / kSlots;
                    if (accumulator_comes_again(t, pairs, items)) ++released[use % kSlots], ++sent;
                }
                for (int s = 0; s < kSlots; ++s)
                    if (released[s] != waited_for[s]) {
                        std::printf("%d items, %d pairs, first %d: slot %d is released %d times and waited for %d times\n", items, pairs, first, s,
                                    released[s], waited_for[s]);
                        return 1;
                    }
            }
        }
    }
    return sent > 0 ? 0 : 2;
}
"""


def test_every_release_of_an_accumulator_is_waited_for(tmp_path):
    source, program = tmp_path / "arrivals.cu", tmp_path / "arrivals"
    source.write_text(PROGRAM)
    csrc = os.path.dirname(build.SOURCES[0])
    subprocess.run([build.nvcc_path(), "-gencode", "arch=compute_100a,code=sm_100a", "-std=c++17", "-I" + csrc, "-o", str(program), str(source)], check=True)
    done = subprocess.run([str(program)], capture_output=True, text=True)
    assert done.returncode == 0, done.stdout
