// How one long sequence is cut into segments that are scanned side by side: plain host arithmetic on sizes, used by the calls and
// by the workspace sizes they state.
#pragma once

#include <algorithm>

namespace lkv {

constexpr int kMaxSegments = 16;   // of a cut that the library chooses

// Segment i covers blocks at[i] .. at[i + 1]; n = 1: the plain scan.
struct Cut {
    int n;
    int at[kMaxSegments + 1];
};

// GDN.  The first pass computes the states that segments 0 .. n-2 reach and the transitions of segments 1 .. n-2, (2 n - 3) CTAs
// a head; the last pass scans all segments, n CTAs a head.  Two ways to stay within one round of CTAs, one per SM: n equal
// segments, or segment n-2 half as long as the others, so that its state and its transition follow one another on one SM
// (at 32 heads on 148 SMs n = 4 of 3 1/2 full segments, against 3 equal ones).
// Both passes take as long as a full segment; between them stands the composition, a chain of n - 2 steps of about a block's
// time each (1.8 us against 1.9), and the launches and the fill of two more pipelines cost about twelve blocks: what was
// measured with n = 4 (one sequence of 16384 tokens, 32 heads: 480 -> 298 us).  The cheapest n is taken if it beats the plain
// scan's chain of blocks.
inline Cut gdn_cut_blocks(int blocks, int heads, int sms) {
    Cut c{1, {0, blocks}};
    if (heads < 1 || blocks < 1) return c;
    const int slots = sms / heads;
    int best = blocks;
    for (int n = 3; n <= std::min(kMaxSegments, slots); ++n) {
        const bool equal = 2 * n - 3 <= slots;
        if (!equal && 2 * n - 3 > slots + 1) break;
        const int full = equal ? (blocks + n - 1) / n : (2 * blocks + 2 * n - 2) / (2 * n - 1);
        if ((n - 1) * full >= blocks) break;   // nothing left for the last of n segments
        const int cost = 2 * full + (n - 2) + 12;
        if (cost >= best) continue;
        best = cost;
        c.n = n;
        for (int i = 0; i < n - 1; ++i) c.at[i] = i * full;
        c.at[n - 1] = blocks - full;           // the last segment is full, the one before it takes what is left
        c.at[n] = blocks;
    }
    return c;
}

// SSD.  Two heads a CTA; no transitions (the composition needs the segments' log-decays only), so n - 1 and n CTAs a pair.  A block
// of the first pass takes 2.0 K cycles against 3.2 K with outputs and the two more launches cost about 16 blocks: worth it from
// three segments of at least eight blocks up -- two would save 0.6 K cycles a block.
inline Cut ssd_cut_blocks(int blocks, int pairs, int sms) {
    Cut c{1, {0, blocks}};
    if (pairs < 1 || blocks < 1) return c;
    const int n = std::min({sms / pairs, blocks / 8, kMaxSegments});
    if (n < 3) return c;
    const int full = (blocks + n - 1) / n;
    c.n = (blocks + full - 1) / full;          // rounding up may leave nothing for the last ones
    for (int i = 0; i <= c.n; ++i) c.at[i] = std::min(i * full, blocks);
    return c;
}

}  // namespace lkv
