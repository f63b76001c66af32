"""The choice of 16-CTA clusters (csrc/lu_cluster.h, built for the host) with a fake occupancy query: an answer
for one matrix size or device is not taken for another, and a query that failed is asked again."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SOURCE = r"""
#include <assert.h>
#include <atomic>
#include <thread>
#include <vector>
#include "lu_cluster.h"
int main() {
    afq::BigClusterCache c;
    int asked = 0;
    auto says = [&](int n) { return [&asked, n] { ++asked; return n; }; };
    assert(c.fits(0, 20000, says(9)));    // a small matrix first
    assert(!c.fits(0, 120000, says(1)));  // a large one of which a single cluster fits
    assert(!c.fits(1, 20000, says(0)));   // the small one on another device
    assert(asked == 3);
    assert(c.fits(0, 20000, says(0)) && !c.fits(0, 120000, says(9)) && !c.fits(1, 20000, says(9)));
    assert(asked == 3);  // kept
    assert(!c.fits(0, 60000, says(-1)) && asked == 4);
    assert(c.fits(0, 60000, says(2)) && asked == 5);  // asked again after a failure
    std::atomic<int> calls{0}, yes{0};
    std::vector<std::thread> t;
    for (int j = 0; j < 8; ++j)
        t.emplace_back([&] {
            for (int q = 0; q < 500; ++q) yes += c.fits(q % 5, 1000 + q, [&] { ++calls; return 2; }) ? 1 : 0;
        });
    for (auto& x : t) x.join();
    assert(yes == 4000 && calls == 500);
    return 0;
}
"""


def test_answers_are_kept_per_device_and_footprint(tmp_path):
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(SOURCE)
    subprocess.check_call(["g++", "-O1", "-std=c++17", "-pthread", "-I",
                           os.path.join(ROOT, "paper_2506_09611_gb300", "csrc"), "-o", str(exe), str(src)])
    subprocess.check_call([str(exe)])
