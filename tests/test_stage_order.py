"""The feeding order of the exact dots' ring of stages (csrc/kg_stages.h),
compiled for the host: every wait made to run out in turn, no GPU."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

HARNESS = r"""
#include <cstdio>
#include <vector>
#include "kg_stages.h"

int main() {
    for (int S = 3; S <= 8; ++S)
        for (int nt = 0; nt <= 3 * S + 1; ++nt)
            for (int bad = -1; bad < 5 * S + 10; ++bad)  // the wait that runs out (-1: none)
                for (int stuck = 0; stuck < 2; ++stuck) {  // ... once, or all that follow too
                    int waits = 0, issued = nt < S ? nt : S;
                    std::vector<int> landed(nt, 0), freed(nt, 0), waited(nt, 0);
                    bool failed = false, fault = false;
                    auto wait = [&]() {
                        const bool good = !(waits == bad || (stuck && bad >= 0 && waits > bad));
                        ++waits;
                        failed |= !good;
                        return good;
                    };
                    auto l = [&](int t) {
                        fault |= t < 0 || t >= issued;
                        const bool g = wait();
                        if (t >= 0 && t < nt) waited[t] = 1, landed[t] |= g;
                        return g;
                    };
                    auto f = [&](int t) {
                        fault |= t < 0 || t >= issued;
                        const bool g = wait();
                        if (t >= 0 && t < nt) freed[t] |= g;
                        return g;
                    };
                    auto i = [&](int t) {
                        // in order, after no failure, into a stage that is empty and done with
                        fault |= t != issued || t >= nt || failed || (t >= S && !(landed[t - S] && freed[t - S]));
                        issued = t + 1;
                    };
                    const bool ok = kg::feed_stages(nt, S, l, f, i);
                    fault |= ok == failed || (!failed && issued != nt);
                    for (int t = 0; t < issued; ++t) fault |= !waited[t];  // nothing left in flight unwaited
                    if (fault) {
                        std::printf("S %d nt %d bad %d stuck %d\n", S, nt, bad, stuck);
                        return 1;
                    }
                }
    return 0;
}
"""


def test_every_issued_copy_is_waited_for(tmp_path):
    src, exe = tmp_path / "stages.cpp", tmp_path / "stages"
    src.write_text(HARNESS)
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-I", os.path.join(ROOT, "paper_1109_1205_gb300", "csrc"),
                           str(src), "-o", str(exe)])
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
