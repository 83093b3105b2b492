"""The process-wide cache of tuned choices: the first choice for a key stays,
the number of keys is bounded, and what leaves is what was used longest ago."""
import os
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1911_10814_gb300", "csrc")

MAIN = r"""
#include "tune_cache.cuh"
#include <thread>
#include <vector>
#define CHECK(x) do { if (!(x)) return __LINE__; } while (0)
int main() {
    nbp::TuneCache<int, int> c(4);
    int v = -1;
    CHECK(!c.find(1, v) && v == -1);
    CHECK(c.keep(1, 10) == 10 && c.keep(1, 11) == 10);   // the first choice stays
    for (int k = 2; k <= 4; ++k) c.keep(k, 10 * k);
    CHECK(c.find(1, v) && v == 10);                      // 1 used after 2
    c.keep(5, 50);
    CHECK(c.size() == 4 && !c.find(2, v) && c.find(1, v) && c.find(3, v) && c.find(4, v) && c.find(5, v));
    for (int k = 0; k < 100000; ++k) c.keep(100 + k, k);
    CHECK(c.size() == 4 && c.find(100 + 99999, v) && v == 99999);
    nbp::TuneCache<int, int> s(64);
    std::vector<std::thread> t;
    std::vector<int> bad(4, 0);
    for (int w = 0; w < 4; ++w)
        t.emplace_back([&, w] {
            for (int r = 0; r < 20000; ++r) {
                const int k = r % 64, got = s.keep(k, 1000 * k + w);
                int f = -1;
                if (!s.find(k, f) || f != got || got / 1000 != k) bad[w] = 1;
            }
        });
    for (auto &x : t) x.join();
    for (int b : bad) CHECK(b == 0);
    CHECK(s.size() == 64);
    return 0;
}
"""


def test_first_choice_stays_and_the_size_is_bounded(tmp_path):
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(MAIN)
    subprocess.run(["g++", "-std=c++17", "-O1", "-pthread", "-I", CSRC, "-o", str(exe), str(src)], check=True)
    assert subprocess.run([str(exe)], timeout=60).returncode == 0
