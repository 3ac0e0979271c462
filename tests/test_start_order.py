"""The order in which the CTAs of one SM started: ages must differ however far apart the starts lie, and over a wrap of the counter."""
import subprocess

from paper_2104_01981_b200 import build

SOURCE = r"""
#include <cstdio>
#include "gc_common.cuh"
int main() {
    const unsigned long long full = 1ull << 54, gaps[][2] = {{0, 0}, {1, 2}, {1500000000ull, 3000000000ull}, {1ull << 31, 1ull << 32},
                                                          {1ull << 40, (1ull << 41) + 5}, {3, 1ull << 50}};
    for (auto& g : gaps)
        for (unsigned long long t0 : {0ull, 1ull << 31, full - 2, full - 2000000000ull, ~0ull - 1})
            for (uint32_t sm : {0u, 147u, 1023u}) {
                const unsigned long long s[3] = {gc::start_word(sm, t0), gc::start_word(sm, t0 + g[0]), gc::start_word(sm, t0 + g[1])};
                const uint32_t cta[3] = {7, 155, 303};                     // (in the order of their starts)
                for (uint32_t i = 0; i < 3; ++i) {
                    uint32_t age = 0;
                    for (uint32_t j = 0; j < 3; ++j) age += j != i && gc::started_before(s[j], cta[j], s[i], cta[i]);
                    if (age != i || gc::start_sm(s[i]) != sm) { std::printf("gap %llu from %llu: age %u of CTA %u\n", g[1], t0, age, i); return 1; }
                }
            }
    return 0;
}
"""


def test_ages_differ(tmp_path):
    src = tmp_path / "order.cu"
    src.write_text(SOURCE)
    exe = str(tmp_path / "order")
    subprocess.run([build._nvcc(), "-std=c++17", "-gencode", "arch=compute_100a,code=sm_100a", "-I", build.CSRC, "-o", exe, str(src)], check=True)
    run = subprocess.run([exe], capture_output=True, text=True)
    assert run.returncode == 0, run.stdout
