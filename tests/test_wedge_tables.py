"""Sizes of the wedge anchors' tables: whatever an anchor's wedges and lower
neighbours are, the table of its class has a slot per wedge, holds the
counters' largest value, and fits the bytes of the class."""
from host_check import run_host_program

PROGRAM = r"""
#include <cstdio>
#include <vector>
#include "tg_wedge_table.hpp"
using namespace tg;

static int check(int L, int64_t light, int64_t hub, int64_t W, int64_t most) {
    WedgeLimits lim{light, hub, {kFormBytes[1], kFormBytes[2], kFormBytes[3], kFormBytes[4]}};
    const int c = wedge_class(lim, L, W, most);
    if (c == kHubClass) return 0;
    const int64_t bytes = c == 0 ? light_bytes(L, light) : kFormBytes[c];
    const Pack k = anchor_pack(L, W, most);
    const int64_t slots = slots_for(W, bytes, k.rw), top = most < W ? most : W;   // a counter is at most either
    const bool ok = c >= 0 && slots >= W && slots <= 65536 && table_need(W, slots, k.rw) <= bytes && bytes % 16 == 0 &&
                    top >> k.bits == 0 && k.F * k.rw >= L && k.F * k.bits <= 32;
    if (!ok)
        std::printf("L %d light %ld hub %ld: %ld wedges, %ld neighbours of a type: class %d, %ld slots, rw %d\n", L, (long)light,
                    (long)hub, (long)W, (long)most, c, (long)slots, k.rw);
    return ok ? 0 : 1;
}

int main() {
    std::vector<int64_t> mosts, lights;
    for (int64_t m = 1; m <= 40; ++m) mosts.push_back(m);
    for (int b = 6; b <= 20; ++b)
        for (int64_t d = -1; d <= 1; ++d) mosts.push_back(((int64_t)1 << b) + d);
    for (int64_t l = 1; l <= 300; ++l) lights.push_back(l);
    for (int64_t l : {383, 384, 511, 512, 513, 768, 1023, 1024, 1025, 1536, 2047, 2048}) lights.push_back(l);
    int bad = 0;
    for (int L = 1; L <= 8; ++L) {
        for (int64_t light : lights)                        // the warp form, every limit
            for (int64_t W = 1; W <= light; ++W)
                for (int64_t m : mosts) bad += check(L, light, (int64_t)1 << 30, W, m);
        for (int64_t W = 1; W <= 40000; ++W)                // the forms of a CTA
            for (int64_t m : mosts) bad += check(L, 1, (int64_t)1 << 30, W, m);
        if (bad > 20) break;
    }
    std::printf("%d\n", bad);
    return bad != 0;
}
"""


def test_every_table_has_a_slot_per_wedge(tmp_path):
    assert run_host_program(PROGRAM, tmp_path).split() == ["0"]
