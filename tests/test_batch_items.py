"""Order of the batched engine's global-update items and the swizzle of its slot
array (`csrc/batch_tables.h`, `csrc/opf_internal.h`), compiled with g++ and
checked on the CPU: the items are the same entries, more copies first and the
bounded ones of equal copies first; the rows of a chunk are its own four, and
the lanes of a shared-memory transaction (128 bytes of consecutive chunks, one
slot each) fall on distinct banks at every row width."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2310_09410_gb300", "csrc")

DRIVER = r"""
#include "batch_tables.h"
#include "opf_internal.h"
#include <cstdio>
#include <random>
#include <set>

using namespace opf;

int main() {
    std::mt19937 rng(7);
    for (int Gs : {0, 1, 2, 31, 700}) {
        GlobalTables t;
        t.Gs = Gs;
        std::multiset<std::vector<int>> was, now;
        for (int j = 0; j < Gs; ++j) {
            const std::vector<int> e = {(int)(rng() % 5000), (int)(rng() % 5000), (int)(1 + rng() % 9) | (int)(rng() % 99) << 8,
                                        rng() % 2 ? -1 : j};
            was.insert(e);
            t.gtab.insert(t.gtab.end(), e.begin(), e.end());
        }
        sort_global_items(&t, 4, 8);
        for (int j = 0; j < Gs; ++j) {
            const int *e = &t.gtab[4 * j], *p = e - 4;
            now.insert({e[0], e[1], e[2], e[3]});
            if (!j) continue;
            const int ce = e[2] & 255, cp = p[2] & 255;
            if (cp < ce || (cp == ce && p[3] < 0 && e[3] >= 0)) return std::printf("order at %d of %d\n", j, Gs), 1;
        }
        if (was != now) return std::printf("entries of %d\n", Gs), 1;
    }
    for (int word : {4, 8})
        for (int K : {1, 2, 4, 8}) {
            const int bytes = K * word;
            if (bytes > 32) continue;
            for (int ch = 0; ch < 64; ++ch) {
                std::set<int> rows;
                for (int e = 0; e < 4; ++e) rows.insert(slot_row(ch, e, bytes));
                if (*rows.begin() != 4 * ch || *rows.rbegin() != 4 * ch + 3 || rows.size() != 4)
                    return std::printf("chunk %d, %d bytes\n", ch, bytes), 1;
            }
            const int lanes = 128 / bytes;     // chunks of one transaction
            for (int e = 0; e < 4; ++e)
                for (int ch = 0; ch + lanes <= 64; ch += lanes) {
                    std::set<int> at;
                    for (int i = 0; i < lanes; ++i) at.insert(slot_row(ch + i, e, bytes) * bytes % 128);
                    if ((int)at.size() != lanes) return std::printf("banks: %d bytes, slot %d\n", bytes, e), 1;
                }
        }
    std::puts("ok");
    return 0;
}
"""


@pytest.mark.skipif(shutil.which("g++") is None, reason="no host compiler")
def test_item_order_and_slot_rows(tmp_path):
    src = tmp_path / "t.cpp"
    src.write_text(DRIVER)
    exe = tmp_path / "t"
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    subprocess.run(["g++", "-O1", "-std=c++17", "-I", CSRC, "-I", os.path.join(ROOT, "include"), "-I",
                    os.path.join(cuda, "include"), str(src), "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], capture_output=True, text=True)
    assert out.returncode == 0 and out.stdout.strip() == "ok", out.stdout
