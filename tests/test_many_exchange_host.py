"""The buffers through which two warps of the GEMM for calls of many rows exchange values: the rule itself (csrc/many_exchange.cuh), compiled
for the host, with both warps run in every order that their barriers allow."""
import os
import re
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2407_12021_b200", "csrc")

PROGRAM = r"""
#include <cstdio>
#include <set>
#include <tuple>
#include <vector>
#include "many_exchange.cuh"
// Each warp: for every exchange write (step 0), arrive and wait (1), read (2).  An exchange that reads something else than what the partner
// wrote in it is an error.
static std::vector<int> buffers(const std::vector<int>& items) {
    aded::ManyExchange exchange;
    std::vector<int> used;
    for (int groups : items)
        for (int g = 0; g < groups; ++g) used.push_back(exchange.next());
    return used;
}
static int wrong;
static std::set<std::tuple<int, int, int, int, int, int>> seen;
static void go(const std::vector<int>& buf, int a, int b, std::vector<int> held) {      // held[warp * 2 + buffer]: the exchange whose values lie there
    if (!seen.insert({a, b, held[0], held[1], held[2], held[3]}).second) return;
    const int at[2] = {a, b}, end = 3 * (int)buf.size();
    for (int w = 0; w < 2; ++w) {
        if (at[w] == end) continue;
        const int e = at[w] / 3, step = at[w] % 3;
        std::vector<int> next = held;
        if (step == 0) next[w * 2 + buf[e]] = e;
        if (step == 1 && at[1 - w] < 3 * e + 1) continue;                               // the partner has not arrived
        if (step == 2 && held[(1 - w) * 2 + buf[e]] != e) ++wrong;
        go(buf, a + (w == 0), b + (w == 1), next);
    }
}
int main() {
    for (int groups = 1; groups <= 8; ++groups)
        for (int items = 1; items <= 3; ++items) {
            seen.clear();
            go(buffers(std::vector<int>(items, groups)), 0, 0, {-1, -1, -1, -1});
        }
    printf("%d\n", wrong);
    return 0;
}
"""


def test_no_exchange_overwrites_what_the_partner_still_reads(tmp_path):
    (tmp_path / "exchange.cpp").write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", CSRC, str(tmp_path / "exchange.cpp"), "-o", str(tmp_path / "exchange")], check=True)
    assert subprocess.run([str(tmp_path / "exchange")], capture_output=True, text=True, check=True).stdout == "0\n"
    kernel = open(os.path.join(CSRC, "gemm_many.cu")).read()
    assert kernel.index("ManyExchange exchange;") < kernel.index("for (int q = 0; q < list.count; ++q) {\n                const ManyPiece pc = many_piece(p, list, q);\n                const bool carried")
    assert len(re.findall(r"\* buf = ", kernel)) == 1 and "* buf = xb + exchange.next() * 512;" in kernel
