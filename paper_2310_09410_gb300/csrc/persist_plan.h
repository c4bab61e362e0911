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
#include <functional>
#include <numeric>
#include <system_error>
#include <thread>
#include <utility>
#include <vector>

namespace opf {

// Part p owns the subsystems sub[s0[p] .. s0[p+1]) and, in that order, their
// slots slot[k0[p] .. k0[p+1]).  A part sees u through an array of its own
// slots (index = position in the part), then the entries it reads from other
// parts, rem[r0[p] .. r0[p+1]) (positions in the global-major copy order), then
// one zero.  For every global of the part with two or more copies, list (16-bit
// entries, part p's from 8 l0[p]) holds the array index of each copy in copy
// order, padded with the zero's index to a multiple of 8; seg[k] = (number of
// the list's first 8 entries in the part << 8) | copies of the slot's global
// (list 0 for a single copy), out[k] = the slot's position in the copy order
// when another part reads it, else -1.  ok: the indices fit 16 bits.
struct PersistParts {
    std::vector<int> s0, k0, r0, l0;
    std::vector<int> sub, slot, rem, seg, out;
    std::vector<unsigned short> list;
    bool ok = true;
};

// Destinations of the exported u when the parts' readers are written to
// directly: per position j of slot[] a list dst[..] of part << 16 | index in
// the reader's remote entries, dseg[j] = (offset in the part's lists << 8) |
// count, part p's lists from d0[p].
struct PersistDests {
    std::vector<int> d0, dst, dseg;
    int most = 0;                     // longest part's lists
    bool ok = true;                   // counts and indices fit their fields
};

inline PersistDests persist_dests(int P, const PersistParts &t, const std::vector<int> &uslot) {
    const int L = (int)t.slot.size();
    PersistDests d;
    std::vector<int> pos(L), n(L, 0);            // position of a slot
    for (int j = 0; j < L; ++j) pos[t.slot[j]] = j;
    for (int c : t.rem) ++n[pos[uslot[c]]];
    d.dseg.assign(L, 0);
    d.d0.assign(P + 1, 0);
    std::vector<int> fill(L);
    int at = 0;
    for (int p = 0; p < P; ++p) {
        for (int j = t.k0[p]; j < t.k0[p + 1]; ++j) {
            if (n[j] > 255 || at - d.d0[p] >= (1 << 22)) d.ok = false;
            d.dseg[j] = ((at - d.d0[p]) << 8) | (n[j] & 255);
            fill[j] = at;
            at += n[j];
        }
        d.d0[p + 1] = at;
        d.most = std::max(d.most, at - d.d0[p]);
    }
    d.dst.assign(at, 0);
    for (int p = 0; p < P; ++p) {
        if (t.r0[p + 1] - t.r0[p] > 0xffff) d.ok = false;
        for (int i = t.r0[p]; i < t.r0[p + 1]; ++i) d.dst[fill[pos[uslot[t.rem[i]]]]++] = (p << 16) | ((i - t.r0[p]) & 0xffff);
    }
    return d;
}

// Depth-first order of the S subsystems.  Slots of subsystem d are
// [soff[d], soff[d + 1]); segp[k] = (first copy of the slot's global in the
// global-major copy order << 8) | copies, pk[k] the slot's own position there.
// start: the order in which unvisited subsystems begin a new tree.
inline std::vector<int> persist_order(int S, const std::vector<int> &soff, const std::vector<int> &segp,
                                      const std::vector<int> &pk, const std::vector<int> &start) {
    std::vector<int> sub_of(pk.size()), order, stack;        // subsystem of a copy
    for (int d = 0; d < S; ++d)
        for (int k = soff[d]; k < soff[d + 1]; ++k) sub_of[pk[k]] = d;
    std::vector<char> seen(S, 0), walked(pk.size(), 0);      // walked: by first copy
    order.reserve(S);
    std::vector<int> by_count;                                // globals of a subsystem (segp words)
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
                const int sp = segp[k], cnt = sp & 255;
                if (cnt < 2 || walked[sp >> 8]) continue;    // no other copy, or all on the stack or seen
                walked[sp >> 8] = cnt > 2;
                size_t at = by_count.size();                 // insertion sort: few and short
                by_count.push_back(sp);
                while (at > 0 && (by_count[at - 1] & 255) < cnt) {
                    by_count[at] = by_count[at - 1];
                    --at;
                }
                by_count[at] = sp;
            }
            for (int sp : by_count)
                for (int c = (sp >> 8) + (sp & 255) - 1; c >= sp >> 8; --c)
                    if (!seen[sub_of[c]]) stack.push_back(sub_of[c]);
        }
    }
    return order;
}

// P parts of the given order, balanced by cost[d].  Subsystems are numbered in
// decreasing size (so a part's are sorted by number).  In two steps: the split
// (s0, sub, k0) tells whether the parts fit a form at all, in an eighth of the
// lists' time.
inline PersistParts persist_split(int P, int S, const std::vector<int> &order, const std::vector<double> &cost,
                                  const std::vector<int> &soff) {
    PersistParts t;
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
    t.k0.assign(P + 1, 0);
    for (int q = 0; q < P; ++q) {
        std::sort(t.sub.begin() + t.s0[q], t.sub.begin() + t.s0[q + 1]);
        t.k0[q + 1] = t.k0[q];
        for (int i = t.s0[q]; i < t.s0[q + 1]; ++i) t.k0[q + 1] += soff[t.sub[i] + 1] - soff[t.sub[i]];
    }
    t.r0.assign(P + 1, 0);
    t.l0.assign(P + 1, 0);
    return t;
}

// Entries of other parts that the parts read, over all parts (rem.size() of
// persist_lists, without the lists): per part and global of several copies, the
// copies that are not the part's own.
inline long long persist_remote(int P, const PersistParts &t, const std::vector<int> &soff,
                                const std::vector<int> &segp) {
    std::vector<int> last(segp.size(), -1);      // by first copy: the last part that counted the global
    long long n = 0;
    for (int q = 0; q < P; ++q)
        for (int i = t.s0[q]; i < t.s0[q + 1]; ++i)
            for (int k = soff[t.sub[i]]; k < soff[t.sub[i] + 1]; ++k) {
                const int cnt = segp[k] & 255;
                if (cnt < 2) continue;
                --n;
                if (last[segp[k] >> 8] == q) continue;
                last[segp[k] >> 8] = q;
                n += cnt;
            }
    return n;
}

// The slots, copy lists and exchanges of split parts.
inline void persist_lists(int P, const std::vector<int> &soff, const std::vector<int> &segp, const std::vector<int> &pk,
                          PersistParts *parts) {
    PersistParts &t = *parts;
    const int L = (int)pk.size();
    // per copy (in copy order) its part and position there, so that a list
    // reads one run of memory
    struct Place { int part, at; };
    std::vector<Place> place(L);
    t.slot.resize(L);
    for (int q = 0, j = 0; q < P; ++q)
        for (int i = t.s0[q]; i < t.s0[q + 1]; ++i)
            for (int k = soff[t.sub[i]]; k < soff[t.sub[i] + 1]; ++k, ++j) {
                place[pk[k]] = {q, j - t.k0[q]};
                t.slot[j] = k;
            }
    t.seg.resize(L);
    t.out.assign(L, -1);
    // Ranges of parts with about as many slots each, on threads of their own when
    // there are many (8500 buses, 119,000 slots: 1.25 ms on one, 0.45 on four).
    // Parts do not depend on each other: a range has its own lists and remote
    // entries, appended in order below, and an export that several ranges mark
    // gets the same value from each.
    struct Range {
        int p0 = 0, p1 = 0;
        bool ok = true;
        std::vector<int> rem;
        std::vector<unsigned short> list;
    };
    auto fill = [&](Range &r) {
        const int slots = t.k0[r.p1] - t.k0[r.p0];
        r.list.resize(4 * (size_t)slots + 8);
        r.rem.reserve(slots / 4);
        size_t used = 0;                             // entries of the lists so far
        std::vector<int> where(L, -1);               // by first copy: number of the part's list, or below the part's first
        for (int q = r.p0; q < r.p1; ++q) {
            const int nk = t.k0[q + 1] - t.k0[q], l0 = (int)(used / 8), r0 = (int)r.rem.size();
            for (int j = t.k0[q]; j < t.k0[q + 1]; ++j) {
                const int sp = segp[t.slot[j]], c0 = sp >> 8, cnt = sp & 255;
                if (cnt == 1) {
                    t.seg[j] = 1;
                    continue;
                }
                if (where[c0] < l0) {
                    where[c0] = (int)(used / 8);
                    const size_t end = used + ((cnt + 7) & ~7);
                    if (end > r.list.size()) r.list.resize(2 * end);
                    unsigned short *e = r.list.data() + used, *last = r.list.data() + end;
                    for (int c = c0; c < c0 + cnt; ++c) {
                        const Place at = place[c];
                        if (at.part == q) {
                            *e++ = (unsigned short)at.at;
                        } else {
                            *e++ = (unsigned short)(nk + (int)r.rem.size() - r0);
                            r.rem.push_back(c);
                            __atomic_store_n(&t.out[t.k0[at.part] + at.at], c, __ATOMIC_RELAXED);
                        }
                    }
                    while (e < last) *e++ = 0xffff;  // past the last copy: the zero, below
                    used = end;
                }
                t.seg[j] = ((where[c0] - l0) << 8) | cnt;
            }
            t.r0[q + 1] = (int)r.rem.size() - r0;    // counts here, places below
            t.l0[q + 1] = (int)(used / 8) - l0;
            const int zero = nk + t.r0[q + 1];
            if (zero >= 0xffff) r.ok = false;
            unsigned short *e = r.list.data() + 8 * (size_t)l0, *last = r.list.data() + used;
            for (; e < last; ++e) *e = *e == 0xffff ? (unsigned short)zero : *e;
        }
        r.list.resize(used);
    };
    const int n_ranges = std::max(1, std::min(4, L / 15000));
    std::vector<Range> ranges(n_ranges);
    for (int i = 0, p = 0; i < n_ranges; ++i) {
        ranges[i].p0 = p;
        while (p < P && (i + 1 == n_ranges || (long long)t.k0[p] * n_ranges < (long long)L * (i + 1))) ++p;
        ranges[i].p1 = p;
    }
    std::vector<std::thread> threads;
    int started = 1;                                 // the first range is this thread's
    try {
        for (; started < n_ranges; ++started) threads.emplace_back(fill, std::ref(ranges[started]));
    } catch (const std::system_error &) {            // no thread to be had: the rest here
    }
    fill(ranges[0]);
    for (int i = started; i < n_ranges; ++i) fill(ranges[i]);
    for (std::thread &th : threads) th.join();
    size_t rems = 0, lists = 0;
    for (const Range &r : ranges) {
        rems += r.rem.size();
        lists += r.list.size();
        t.ok = t.ok && r.ok;
    }
    t.rem.reserve(rems);
    t.list.reserve(lists);
    for (const Range &r : ranges) {
        t.rem.insert(t.rem.end(), r.rem.begin(), r.rem.end());
        t.list.insert(t.list.end(), r.list.begin(), r.list.end());
    }
    for (int q = 0; q < P; ++q) {
        t.r0[q + 1] += t.r0[q];
        t.l0[q + 1] += t.l0[q];
    }
}

inline PersistParts persist_parts(int P, int S, const std::vector<int> &order, const std::vector<double> &cost,
                                  const std::vector<int> &soff, const std::vector<int> &segp,
                                  const std::vector<int> &pk) {
    PersistParts t = persist_split(P, S, order, cost, soff);
    persist_lists(P, soff, segp, pk, &t);
    return t;
}

// Owner form (instances whose globals have many copies): P parts of balanced
// cost, the dearest subsystems placed first, and an owner for every global, its
// copies' entries of u one run of the copy order.  Part p owns the globals
// [g0[p], g0[p+1]) (most copies: most); parts.rem[r0[p] .. r0[p+1]) are the
// distinct globals of part p's slots, parts.seg[j] = (index there << 8) |
// copies, parts.out[j] = the slot's position in the copy order.
struct PersistOwners {
    PersistParts parts;
    std::vector<int> g0;
    int most_globals = 0, most_copies = 0;
};

inline PersistOwners persist_owners(int P, int S, int G, const std::vector<double> &cost, const std::vector<int> &soff,
                                    const std::vector<int> &segp, const std::vector<int> &pk,
                                    const std::vector<int> &gk, const std::vector<int> &gstart) {
    PersistOwners o;
    PersistParts &t = o.parts;
    const int L = (int)pk.size();
    std::vector<int> order(S);
    std::iota(order.begin(), order.end(), 0);
    std::stable_sort(order.begin(), order.end(), [&](int a, int b) { return cost[a] > cost[b]; });
    std::vector<std::vector<int>> of(P);
    std::vector<std::pair<double, int>> load(P);             // min-heap
    for (int p = 0; p < P; ++p) load[p] = {0.0, p};
    const auto more = std::greater<std::pair<double, int>>();
    for (int d : order) {
        std::pop_heap(load.begin(), load.end(), more);
        of[load.back().second].push_back(d);
        load.back().first += cost[d];
        std::push_heap(load.begin(), load.end(), more);
    }
    t.s0.assign(P + 1, 0);
    t.k0.assign(P + 1, 0);
    t.r0.assign(P + 1, 0);
    t.l0.assign(P + 1, 0);
    std::vector<int> at(G, -1), seen(G, -1);
    for (int p = 0; p < P; ++p) {
        std::sort(of[p].begin(), of[p].end());               // decreasing size
        t.sub.insert(t.sub.end(), of[p].begin(), of[p].end());
        for (int d : of[p])
            for (int k = soff[d]; k < soff[d + 1]; ++k) {
                const int g = gk[k];
                if (seen[g] != p) {
                    seen[g] = p;
                    at[g] = (int)t.rem.size() - t.r0[p];
                    t.rem.push_back(g);
                }
                t.slot.push_back(k);
                t.seg.push_back((at[g] << 8) | (segp[k] & 255));
                t.out.push_back(pk[k]);
            }
        t.s0[p + 1] = (int)t.sub.size();
        t.k0[p + 1] = (int)t.slot.size();
        t.r0[p + 1] = (int)t.rem.size();
    }
    // a global weighs one besides its copies
    o.g0.assign(P + 1, G);
    o.g0[0] = 0;
    const long long total = (long long)L + G;
    for (int p = 1, g = 0; p < P; ++p) {
        while (g < G && (long long)gstart[g + 1] + g + 1 <= total * p / P) ++g;
        o.g0[p] = g;
    }
    for (int p = 0; p < P; ++p) {
        o.most_globals = std::max(o.most_globals, o.g0[p + 1] - o.g0[p]);
        o.most_copies = std::max(o.most_copies, gstart[o.g0[p + 1]] - gstart[o.g0[p]]);
    }
    return o;
}

}  // namespace opf
