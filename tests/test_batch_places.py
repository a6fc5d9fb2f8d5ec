"""Which launches of the batch engine fit beside each other (batch_places.h),
checked on the CPU: the header the engine uses, compiled with the host compiler."""
import os
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1901_05118_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include "batch_places.h"
using namespace excmg;
#define CHECK(c) do { if (!(c)) { std::printf("%s: sms %d per_sm %d resident %d coop %d\n", #c, s, k, r, c0); std::exit(1); } } while (0)
int main() {
    for (int s : {152, 20})
    for (int k : {1, 2})
    for (int r = 0; r <= s; ++r)
    for (int c0 = 0; c0 <= k * (s - r); ++c0) {
        const SmPlaces p{s, k, r, c0};
        CHECK(free_places(p) >= 0);
        for (int ctas : {1, 16, 72, 152})
            CHECK(!on_chip_fits(p, ctas) || c0 <= k * (s - r - ctas));   // they never add up to more than the SMs
        CHECK(r + c0 > 0 || on_chip_fits(p, s));
        for (int want : {1, 2, 45, 90, 152, 304, 1000}) {
            const int g = coop_share(p, want), ask = want < k * s ? want : k * s;
            CHECK(g >= 0 && g <= ask);
            CHECK(g == 0 || 2 * g >= ask);                  // never on a small rest of the SMs
            CHECK(c0 + g <= k * (s - r));                   // all fit on the SMs without on-chip CTAs
            CHECK(r + c0 > 0 || g == ask);                  // an idle GPU keeps no group waiting
        }
    }
    const int s = 152, k = 2, r = 0, c0 = 0;
    CHECK(coop_share(SmPlaces{152, 2, 144, 0}, 180) == 0);   // beside nine 32^3 members
    CHECK(coop_share(SmPlaces{152, 2, 150, 0}, 180) == 0);   // beside a 66^3 one
    CHECK(coop_share(SmPlaces{152, 2, 72, 0}, 180) == 160);
    return 0;
}
"""


def test_places(tmp_path):
    src = tmp_path / "places.cpp"
    src.write_text(PROGRAM.replace("#include <cstdlib>", "#include <cstdlib>\n#include <initializer_list>"))
    exe = tmp_path / "places"
    subprocess.run(["g++", "-O2", "-std=c++17", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], capture_output=True, text=True)
    assert out.returncode == 0, out.stdout
