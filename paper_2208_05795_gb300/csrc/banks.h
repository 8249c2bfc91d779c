// banks.h -- an order of a general code's checks, and of the edges within
// each check, in which a warp's shared-memory gathers hit different banks
// (host code, run once per code by load_code()).
//
// The two-codeword kernel gives lane l of a warp the check in slot 32 w + l,
// and for every position p the warp reads (and later adds to) the 32 words
// P[v(slot, p)], word v in bank v mod 32.  In the order of the matrix those
// are 32 random banks, about 3.4 wavefronts an access.  Min-sum does not
// depend on either order, so both are free:
//   1. the checks are divided into groups of 32 so that no bank is met by
//      more than dc edges of a group (greedily, then by exchanges);
//   2. within a group the edges form a bipartite graph, checks against
//      banks; a proper edge colouring with dc colours (Koenig; alternating
//      paths) gives the positions, each a set of different banks.
// (1008, 504) PEG-like code: 3.36 -> 1.55 wavefronts an access; the decode
// kernel, 97 % of whose cycles moved shared-memory wavefronts, 126 -> 105 ms on
// 150,000 candidates.  Host time 0.5 ms at m = 504, 1.5 at m = 2000, 5 at m = 10,900
// (load_code() makes it on a thread beside its other work).
// The edges by which a bank exceeds dc go to the last positions, as far as
// exchanges within their checks allow.
#pragma once
#include <algorithm>
#include <cstdint>
#include <utility>
#include <vector>

namespace tsx {

// col: [m * dc] variable nodes by check.  Returns them in slot and position order.
inline std::vector<uint16_t> bank_order(int m, int dc, const std::vector<uint16_t> &col) {
    constexpr int W = 32;
    const int ng = (m + W - 1) / W;
    std::vector<int> slot_of(m), chk(m);  // slot of a check, check of a slot
    std::vector<int> cnt((size_t)ng * W, 0), size(ng, 0);
    auto over = [&](int x) { return (x - dc) * (x - dc); };
    std::vector<uint8_t> bk_of((size_t)m * dc);  // bank of a check's p-th edge
    for (size_t e = 0; e < bk_of.size(); e++) bk_of[e] = col[e] & (W - 1);
    auto bank = [&](int c, int p) { return (int)bk_of[(size_t)c * dc + p]; };
    // greedy: each check into the group with room where its banks are met least
    // (a group's count of a bank weighs as its square)
    uint32_t rng = 12345u;
    auto rnd = [&](uint32_t n) {
        rng = rng * 1664525u + 1013904223u;
        return (uint32_t)(((uint64_t)(rng >> 8) * n) >> 24);
    };
    for (int c = 0; c < m; c++) {
        int best = -1, best_cost = 0;
        const int tries = ng < 24 ? ng : 24;  // (large codes: a sample of the groups)
        const int g0 = ng <= 24 ? 0 : (int)rnd((uint32_t)ng);
        for (int t = 0, seen = 0, g = g0; t < ng && seen < tries; t++, g = g + 1 < ng ? g + 1 : 0) {
            const int room = g == ng - 1 ? m - W * (ng - 1) : W;
            if (size[g] >= room) continue;
            seen++;
            int cost = 2 * size[g] * dc / W;  // (fill evenly)
            const int *cn = &cnt[(size_t)g * W];
            for (int p = 0; p < dc; p++) cost += 2 * cn[bank(c, p)] + 1;
            if (best < 0 || cost < best_cost) {
                best = g;
                best_cost = cost;
            }
        }
        slot_of[c] = best * W + size[best]++;
        chk[slot_of[c]] = c;
        for (int p = 0; p < dc; p++) cnt[(size_t)best * W + bank(c, p)]++;
    }
    // exchanges of two checks of different groups that do not raise the squared
    // distance of the counts from dc: a check of an overfull bank against any other
    const int tries = ng > 1 ? (80 * m < 80000 ? 80 * m : 80000) : 0;
    for (int t = 0; t < tries; t++) {
        const int a = (int)rnd((uint32_t)m), b = (int)rnd((uint32_t)m);
        const int ga = slot_of[a] / W, gb = slot_of[b] / W;
        if (ga == gb) continue;
        int *ca = &cnt[(size_t)ga * W], *cb = &cnt[(size_t)gb * W];
        // moving a check out of a group lowers the cost by 2 (count - dc) - 1 per edge, into it raises it
        int gain = 0;
        const uint8_t *xa = &bk_of[(size_t)a * dc], *xb = &bk_of[(size_t)b * dc];
        for (int p = 0; p < dc; p++) gain += ca[xa[p]] - cb[xa[p]] + cb[xb[p]] - ca[xb[p]];
        if (gain <= dc) continue;  // (at most 2 dc more than the exact change: edges of the two in one bank)
        auto add = [&](int *cn, int c, int s, int &d) {
            for (int p = 0; p < dc; p++) {
                int &x = cn[bank(c, p)];
                d -= over(x);
                x += s;
                d += over(x);
            }
        };
        int d = 0, back = 0;
        add(ca, a, -1, d);
        add(cb, b, -1, d);
        add(ca, b, 1, d);
        add(cb, a, 1, d);
        if (d <= 0) {
            std::swap(slot_of[a], slot_of[b]);
            chk[slot_of[a]] = a;
            chk[slot_of[b]] = b;
        } else {
            add(ca, b, -1, back);
            add(cb, a, -1, back);
            add(ca, a, 1, back);
            add(cb, b, 1, back);
        }
    }
    // positions: colour the edges of each group
    std::vector<uint16_t> out((size_t)m * dc);
    std::vector<int> atC((size_t)W * dc), atB((size_t)W * dc), color(W * dc), hist(W * dc), path;
    for (int g = 0; g < ng; g++) {
        const int rows = g == ng - 1 ? m - W * (ng - 1) : W;
        std::fill(atC.begin(), atC.end(), -1);
        std::fill(atB.begin(), atB.end(), -1);
        std::fill(color.begin(), color.end(), -1);
        auto bk = [&](int ed) { return bank(chk[g * W + ed / dc], ed % dc); };
        auto set = [&](int ed, int k) {
            color[ed] = k;
            atC[(ed / dc) * dc + k] = ed;
            atB[bk(ed) * dc + k] = ed;
        };
        for (int ed = 0; ed < rows * dc; ed++) {
            const int r = ed / dc, b = bk(ed);
            int fc = -1, fb = -1, both = -1;
            for (int k = 0; k < dc; k++) {
                const bool c0 = atC[r * dc + k] < 0, b0 = atB[b * dc + k] < 0;
                if (c0 && fc < 0) fc = k;
                if (b0 && fb < 0) fb = k;
                if (c0 && b0 && both < 0) both = k;
            }
            if (both < 0 && fb >= 0) {
                // exchange the colours fc and fb along the path from bank b: then fc is free at both ends
                path.clear();
                int node = b, k = fc;
                for (bool at_bank = true;; at_bank = !at_bank, k = k == fc ? fb : fc) {
                    const int x = at_bank ? atB[node * dc + k] : atC[node * dc + k];
                    if (x < 0) break;
                    path.push_back(x);
                    node = at_bank ? x / dc : bk(x);
                }
                for (int x : path) atC[(x / dc) * dc + color[x]] = atB[bk(x) * dc + color[x]] = -1;
                for (int x : path) set(x, color[x] == fc ? fb : fc);
                both = fc;
            }
            if (both >= 0) set(ed, both);
        }
        // What a bank has more than dc of takes the position left; then exchanges of two
        // positions within a check move the conflicts towards the last position, where they cost
        // a wavefront together instead of one each.
        std::fill(hist.begin(), hist.end(), 0);
        for (int ed = 0; ed < rows * dc; ed++) {
            if (color[ed] < 0)
                for (int k = 0; k < dc && color[ed] < 0; k++)
                    if (atC[(ed / dc) * dc + k] < 0) {
                        color[ed] = k;
                        atC[(ed / dc) * dc + k] = ed;
                    }
            hist[color[ed] * W + bk(ed)]++;
        }
        auto weight = [&](int k) { return 2 * (dc - k) + 1; };
        for (int sweep = 0; sweep < 8; sweep++) {
            bool moved = false;
            for (int e1 = 0; e1 < rows * dc; e1++) {
                const int k1 = color[e1], b1 = bk(e1);
                if (hist[k1 * W + b1] < 2) continue;
                for (int e2 = e1 / dc * dc; e2 < e1 / dc * dc + dc; e2++) {
                    const int k2 = color[e2], b2 = bk(e2);
                    if (k2 == k1 || b2 == b1) continue;
                    // excess taken away and added by the exchange
                    const int d = weight(k2) * ((hist[k2 * W + b1] > 0) - (hist[k2 * W + b2] > 1)) +
                                  weight(k1) * ((hist[k1 * W + b2] > 0) - 1);
                    if (d >= 0) continue;
                    hist[k1 * W + b1]--;
                    hist[k2 * W + b2]--;
                    hist[k1 * W + b2]++;
                    hist[k2 * W + b1]++;
                    std::swap(color[e1], color[e2]);
                    moved = true;
                    break;
                }
            }
            if (!moved) break;
        }
        for (int ed = 0; ed < rows * dc; ed++)
            out[(size_t)(g * W + ed / dc) * dc + color[ed]] = col[(size_t)chk[g * W + ed / dc] * dc + ed % dc];
    }
    return out;
}

}  // namespace tsx
