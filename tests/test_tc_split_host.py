"""The split of a tensor-core translation launch over the SMs (csrc/tc_split.h), compiled for the host: over
random slot counts, tiles without a slot among them, every CTA has a slot, every slot one CTA, and the
pieces of a cut tile that the addition reads are exactly those that the CTAs write, each once."""
import subprocess

from paper_2006_03515_gb300 import build

SRC = r"""
#include <cstdio>
#include <cstdlib>
#include <map>
#include <vector>
#include "tc_split.h"
using namespace kifmm;
static int check(const std::vector<int>& cnt, int max_ctas) {
    const int nt = (int)cnt.size();
    std::vector<int> pre(nt + 1, 0);
    for (int k = 0; k < nt; ++k) pre[k + 1] = pre[k] + cnt[k];
    const int T = pre[nt], n = tc_num_ctas(T, nt, max_ctas);
    if (n < 1 || n > max_ctas) return 1;
    if (T == 0) return 0;
    std::map<int, int> wrote;   // piece -> tile
    for (int c = 0; c < n; ++c) {
        const int g0 = tc_range(c, T, n), g1 = tc_range(c + 1, T, n);
        if (g0 >= g1 || (c == 0 && g0 != 0) || (c == n - 1 && g1 != T)) return 2;
        for (int g = g0; g < g1; ++g)
            if (tc_cta_of(g, T, n) != c) return 3;
        for (int k = 0; k < nt; ++k) {
            if (pre[k + 1] <= g0 || pre[k] >= g1 || (pre[k] >= g0 && pre[k + 1] <= g1)) continue;
            if (!wrote.insert({tc_piece(c, pre[k], T, n), k}).second) return 4;
        }
    }
    size_t read = 0;
    for (int k = 0; k < nt; ++k) {
        if (pre[k] == pre[k + 1]) continue;
        const int c0 = tc_cta_of(pre[k], T, n), c1 = tc_cta_of(pre[k + 1] - 1, T, n);
        for (int c = c0; c0 != c1 && c <= c1; ++c, ++read) {
            auto it = wrote.find(tc_piece(c, pre[k], T, n));
            if (it == wrote.end() || it->second != k) return 5;
        }
    }
    return read == wrote.size() ? 0 : 6;
}
int main() {
    srand(1);
    std::vector<std::vector<int>> cases = {{2, 0, 0, 0, 0, 0, 0}, {2, 0, 0, 0, 0, 0, 0, 0, 0}, {0, 0, 3, 0}, {0}, {1}, {189}};
    for (int t = 0; t < 20000; ++t) {
        std::vector<int> cnt(1 + rand() % 40);
        const int zeros = rand() % 4, most = 1 + rand() % (t % 3 ? 8 : 250);
        for (int& c : cnt) c = rand() % 4 < zeros ? 0 : rand() % (most + 1);
        cases.push_back(cnt);
    }
    for (auto& c : cases)
        for (int m : {1, 2, 76, 152})
            if (int e = check(c, m)) {
                printf("fault %d, %d CTAs at most:", e, m);
                for (int x : c) printf(" %d", x);
                printf("\n");
                return 1;
            }
    return 0;
}
"""


def test_every_piece_read_is_written(tmp_path):
    src, exe = tmp_path / "split.cc", tmp_path / "split"
    src.write_text(SRC)
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-I", build.CSRC, str(src), "-o", str(exe)])
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
