// Host-side partition of an instance over the CTAs of the persistent grid
// engine (no CUDA).
//
// Subsystems are taken in a depth-first order of the graph whose edges are
// shared globals (those with few copies followed first, so that on a feeder
// every subtree is one run) and cut into P runs of balanced work.  A part's
// globals then have most of their copies inside the part: on the 8500-bus
// feeder with 304 parts a part reads 48 entries of other parts per iteration
// on average (134 at most), where runs of the size-sorted order read 474
// (823).  Inside a part the subsystems are in decreasing size, so that the lanes of a warp have
// rows and columns of similar length.
#pragma once

#include <algorithm>
#include <numeric>
#include <vector>

namespace opf {

// Part p owns the subsystems sub[s0[p] .. s0[p+1]) and, in that order, their
// slots slot[k0[p] .. k0[p+1]).  A part sees u through an array of its own
// slots (index = position in the part) followed by the entries it reads from
// other parts, rem[r0[p] .. r0[p+1]) (positions in the global-major copy
// order).  For every global of the part with two or more copies, list[l0[p]
// ..] holds the array index of each copy in copy order; seg[k] = (offset of the
// list in the part's << 8) | copies of the slot's global (offset 0 for a
// single copy), out[k] = the slot's position in the copy order when another
// part reads it, else -1.
struct PersistParts {
    std::vector<int> s0, k0, r0, l0;
    std::vector<int> sub, slot, rem, list, seg, out;
};

// Depth-first order of the S subsystems.  Slots of subsystem d are
// [soff[d], soff[d + 1]) with global gk[k]; the copies of global i are
// uslot[gstart[i] .. gstart[i + 1]).  start: the order in which unvisited
// subsystems begin a new tree.
inline std::vector<int> persist_order(int S, const std::vector<int> &soff, const std::vector<int> &gk,
                                      const std::vector<int> &gstart, const std::vector<int> &uslot,
                                      const std::vector<int> &start) {
    std::vector<int> sub_of(gk.size()), order, stack;
    for (int d = 0; d < S; ++d)
        for (int k = soff[d]; k < soff[d + 1]; ++k) sub_of[k] = d;
    std::vector<char> seen(S, 0), walked(gstart.size(), 0);
    order.reserve(S);
    std::vector<int> by_count;
    for (int first : start) {
        if (seen[first]) continue;
        stack.push_back(first);
        while (!stack.empty()) {
            const int d = stack.back();
            stack.pop_back();
            if (seen[d]) continue;
            seen[d] = 1;
            order.push_back(d);
            // the globals with the fewest copies pushed last, so followed first
            by_count.clear();
            for (int k = soff[d]; k < soff[d + 1]; ++k) {
                const int g = gk[k], cnt = gstart[g + 1] - gstart[g];
                if (cnt < 2 || walked[g]) continue;      // no other copy, or all on the stack or seen
                walked[g] = cnt > 2;
                size_t at = by_count.size();             // insertion sort: few and short
                by_count.push_back(g);
                while (at > 0 && gstart[by_count[at - 1] + 1] - gstart[by_count[at - 1]] < cnt) {
                    by_count[at] = by_count[at - 1];
                    --at;
                }
                by_count[at] = g;
            }
            for (int g : by_count) {
                for (int q = gstart[g + 1] - 1; q >= gstart[g]; --q)
                    if (!seen[sub_of[uslot[q]]]) stack.push_back(sub_of[uslot[q]]);
            }
        }
    }
    return order;
}

// P parts of the given order, balanced by cost[d].
inline PersistParts persist_parts(int P, int S, const std::vector<int> &order, const std::vector<double> &cost,
                                  const std::vector<int> &soff, const std::vector<int> &gk,
                                  const std::vector<int> &pk, const std::vector<int> &gstart,
                                  const std::vector<int> &uslot) {
    PersistParts t;
    const int L = (int)gk.size(), G = (int)gstart.size() - 1;
    t.slot.reserve(L);
    t.list.reserve(2 * (size_t)L);
    t.s0.assign(P + 1, S);
    t.s0[0] = 0;
    double total = 0, acc = 0;
    for (int d = 0; d < S; ++d) total += cost[d];
    int p = 1;
    for (int i = 0; i < S && p < P; ++i) {
        acc += cost[order[i]];
        while (p < P && acc >= total * p / P) t.s0[p++] = i + 1;
    }
    t.sub = order;
    for (int q = 0; q < P; ++q)
        std::stable_sort(t.sub.begin() + t.s0[q], t.sub.begin() + t.s0[q + 1], [&](int a, int b) {
            return soff[a + 1] - soff[a] > soff[b + 1] - soff[b];
        });
    std::vector<int> part_of(L), at(L);          // per slot: part, position in it
    t.k0.assign(P + 1, 0);
    for (int q = 0; q < P; ++q) {
        for (int i = t.s0[q]; i < t.s0[q + 1]; ++i)
            for (int k = soff[t.sub[i]]; k < soff[t.sub[i] + 1]; ++k) {
                part_of[k] = q;
                at[k] = (int)t.slot.size() - t.k0[q];
                t.slot.push_back(k);
            }
        t.k0[q + 1] = (int)t.slot.size();
    }
    t.seg.assign(L, 0);
    t.out.assign(L, -1);
    t.r0.assign(P + 1, 0);
    t.l0.assign(P + 1, 0);
    std::vector<int> done(G, -1), where(G, 0);
    std::vector<char> read(L, 0);                // per slot: another part reads it
    for (int q = 0; q < P; ++q) {
        const int nk = t.k0[q + 1] - t.k0[q];
        for (int j = t.k0[q]; j < t.k0[q + 1]; ++j) {
            const int k = t.slot[j], g = gk[k], c0 = gstart[g], cnt = gstart[g + 1] - c0;
            if (cnt > 1 && done[g] != q) {
                done[g] = q;
                where[g] = (int)t.list.size() - t.l0[q];
                for (int c = c0; c < c0 + cnt; ++c) {
                    const int o = uslot[c];
                    if (part_of[o] == q) {
                        t.list.push_back(at[o]);
                    } else {
                        t.list.push_back(nk + (int)t.rem.size() - t.r0[q]);
                        t.rem.push_back(c);
                        read[o] = 1;
                    }
                }
            }
            t.seg[j] = ((cnt > 1 ? where[g] : 0) << 8) | cnt;
        }
        t.r0[q + 1] = (int)t.rem.size();
        t.l0[q + 1] = (int)t.list.size();
    }
    for (int j = 0; j < L; ++j)
        if (read[t.slot[j]]) t.out[j] = pk[t.slot[j]];
    return t;
}

}  // namespace opf
