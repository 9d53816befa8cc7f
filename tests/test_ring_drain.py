"""The bookkeeping of a convolution CTA whose waits ran out (csrc/ring.h), on the host: whatever
the two producers of a ring had issued when they stopped, every copy in flight is waited for,
and no barrier takes more than its two arrivals."""
import os
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2506_15183_gb300", "csrc")

PROGRAM = r"""
#include "ring.h"
#include <cstdio>
int main()
{
    int bad = 0, cases = 0;
    for (int stages = 1; stages <= 12; ++stages)
        for (int used = 0; used <= 30; ++used)
            for (int a = used; a <= used + stages; ++a)  // a producer is at most a ring ahead
                for (int b = used; b <= used + stages; ++b, ++cases) {
                    int arrivals[64] = {}, waited[64] = {};
                    for (int k = 0; k < a; ++k) ++arrivals[k];
                    for (int k = 0; k < b; ++k) ++arrivals[k];
                    int next = used;
                    yoro::ring_drain(used, a, b, [&](int k) { ++arrivals[k]; },
                                     [&](int k) {
                                         if (k != next++ || arrivals[k] != 2) ++bad;  // would run out, or out of turn
                                         waited[k] = 1;
                                     });
                    for (int k = 0; k < 64; ++k) {
                        if (arrivals[k] > 2) ++bad;
                        if (k >= used && (k < a || k < b) && !waited[k]) ++bad;  // a copy left in flight
                        if (k >= a && k >= b && arrivals[k]) ++bad;
                    }
                }
    printf("%d %d\n", cases, bad);
}
"""


def test_every_copy_in_flight_is_waited_for(tmp_path):
    (tmp_path / "ring.cpp").write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", f"-I{CSRC}", str(tmp_path / "ring.cpp"), "-o", str(tmp_path / "ring")], check=True)
    cases, bad = map(int, subprocess.run([str(tmp_path / "ring")], check=True, capture_output=True, text=True).stdout.split())
    assert cases > 1000 and bad == 0


def test_both_forms_drain_through_it():
    src = open(os.path.join(CSRC, "unet.cu")).read()
    for kernel in ("conv3x3_tc(", "conv3x3_halo("):
        body = src[src.index("    " + kernel):]
        body = body[:body.index("\n}\n")]
        assert body.count("ring_drain(") == 1, kernel
