"""How the TMA-fed GEMM deals its tiles, on the CPU: the header that the kernel and its launch share is compiled by itself, and for many sizes
and numbers of workers every 64-channel unit of every row tile must be dealt to exactly one worker, inside the boxes and stages it was
planned with, and no worker may be left without work."""
import os
import subprocess

import paper_2509_21302_b200 as q

CSRC = os.path.join(os.path.dirname(q.__file__), "csrc")
PROGRAM = r"""
#include <cstdio>
#include <vector>
#include "gemm_c8_plan.cuh"
using namespace gemm_c8;
#define CHECK(c) do { if (!(c)) { std::printf("%s: M %d N %d K %d workers %d\n", #c, M, N, K, W); return 1; } } while (0)
static int check(int M, int N, int K, int W)
{
    int workers = 0;
    const Plan p = make_plan(M, N, K, W, &workers);
    const int rows = (M + 255) / 256, units = N / 64, resident = K == 1024;
    std::vector<int> dealt((size_t)rows * units);
    CHECK(workers >= 1 && workers <= W);
    CHECK(p.stages >= 2 && p.stages <= (resident ? RES_KB : MAX_STAGES));
    CHECK((resident ? RES_KB * A_BYTES : 0) + p.stages * p.stage_bytes <= OPS_BYTES);
    for (int w = 0; w < workers; ++w) {
        Tiles t(p, w);
        CHECK(t.count >= 1);
        for (int i = 0; i < t.count; ++i, t.next()) {
            const int box = i < p.runs * p.run + p.rounds ? p.wide : p.cut;
            CHECK(t.units >= 1 && t.units <= box && box <= MAX_UNITS && (resident ? 0 : A_BYTES) + box * UNIT_BYTES <= p.stage_bytes);
            CHECK(t.row >= 0 && t.row < rows && t.unit >= 0 && t.unit + t.units <= units);
            for (int u = 0; u < t.units; ++u) ++dealt[(size_t)t.row * units + t.unit + u];
        }
    }
    for (int d : dealt) CHECK(d == 1);
    return 0;
}
int main()
{
    unsigned long long r = 12345;
    auto below = [&](int n) { r = r * 6364136223846793005ull + 1442695040888963407ull; return (int)((r >> 33) % n); };
    for (int i = 0; i < 30000; ++i)
        if (check(1 + below(i % 2 ? 20000 : 2000), 128 * (1 + below(i % 3 ? 40 : 10)), below(2) ? 1024 : 4096, below(3) ? 74 : 1 + below(100))) return 1;
    return check(2200003, 4096, 1024, 74) || check(1, 128, 4096, 74);
}
"""


def test_every_unit_is_dealt_once(tmp_path):
    (tmp_path / "plan.cpp").write_text(PROGRAM)
    subprocess.check_call([os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-I", CSRC, "-o", str(tmp_path / "plan"), str(tmp_path / "plan.cpp")])
    r = subprocess.run([str(tmp_path / "plan")], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
