"""The batched engine's global-update items (`sort_global_items`,
`csrc/batch_tables.h`), compiled with g++: on random tables the order is the
plain greedy's (by kind and first row; each next item the first of 256 with the
fewest banks taken among its transaction's neighbours)."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2310_09410_gb300", "csrc")

DRIVER = r"""
#include "batch_tables.h"
#include <cstdio>
#include <random>
#include <set>
using namespace opf;
static std::vector<int> plain(const std::vector<int> &tab, int K, int group) {
    std::vector<std::vector<int>> left, out;
    for (size_t j = 0; j < tab.size(); j += 4) left.push_back({tab[j], tab[j + 1], tab[j + 2], tab[j + 3]});
    auto kind = [](const std::vector<int> &e) { return std::make_pair(-(e[2] & 255), e[3] < 0); };
    std::stable_sort(left.begin(), left.end(), [&](const auto &a, const auto &b) {
        return std::make_tuple(kind(a), a[0]) < std::make_tuple(kind(b), b[0]);
    });
    std::set<int> b0, b1;
    while (!left.empty()) {
        if (out.size() % group == 0) { b0.clear(); b1.clear(); }
        size_t best = 0;
        int fewest = 3;
        for (size_t i = 0; i < left.size() && i < 256 && kind(left[i]) == kind(left[0]); ++i) {
            const int c = (int)b0.count(left[i][0] / K % group) + ((left[i][2] & 255) > 1 ? (int)b1.count(left[i][1] / K % group) : 0);
            if (c < fewest) { fewest = c; best = i; }
        }
        out.push_back(left[best]);
        b0.insert(left[best][0] / K % group);
        if ((left[best][2] & 255) > 1) b1.insert(left[best][1] / K % group);
        left.erase(left.begin() + best);
    }
    std::vector<int> r;
    for (const auto &e : out) r.insert(r.end(), e.begin(), e.end());
    return r;
}
int main() {
    std::mt19937 rng(3);
    for (int K : {1, 2, 4, 8})
        for (int word : {4, 8})
            for (int Gs : {0, 1, 5, 60, 700}) {
                std::vector<int> rows(2 * Gs + 8);
                std::iota(rows.begin(), rows.end(), 0);
                std::shuffle(rows.begin(), rows.end(), rng);
                GlobalTables t;
                t.Gs = Gs;
                for (int j = 0; j < Gs; ++j) {
                    const int cnt = rng() % 8 ? 1 + rng() % 3 : 1 + rng() % 255;
                    const int e[4] = {rows[2 * j] * K, cnt > 1 ? rows[2 * j + 1] * K : 0, cnt | (int)(rng() % 99) << 8, rng() % 2 ? -1 : j};
                    t.gtab.insert(t.gtab.end(), e, e + 4);
                }
                const int group = std::max(1, 128 / (K * word));
                const std::vector<int> want = plain(t.gtab, K, group);
                sort_global_items(&t, K, group);
                if (t.gtab != want) return std::printf("K %d, %d-byte words, %d items\n", K, word, Gs), 1;
            }
    std::puts("ok");
    return 0;
}
"""


@pytest.mark.skipif(shutil.which("g++") is None, reason="no host compiler")
def test_order_is_the_greedy(tmp_path):
    (tmp_path / "t.cpp").write_text(DRIVER)
    exe = tmp_path / "t"
    subprocess.run(["g++", "-O1", "-std=c++17", "-I", CSRC, str(tmp_path / "t.cpp"), "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], capture_output=True, text=True)
    assert out.returncode == 0 and out.stdout.strip() == "ok", out.stdout
