// resident_plan.h -- host side of a resident launch (fdtd_resident.cu): which
// nodes each block works, and which block works each source and probe.  Plain
// C++ over the board descriptor, so that it can be checked without a GPU.
#pragma once

#include <algorithm>
#include <cmath>
#include <vector>

#include "fdtd_internal.h"

namespace fdtd {

// Boxes of a board: its slab boxes, then the z-UPML planes of the fused region
// below and above, then the planes between them.
inline int res_boxes(const Board &h) { return h.n_slab + 3; }
inline void res_box_range(const Board &h, int box, int lo[3], int hi[3])
{
    if (box < h.n_slab) {
        const Slab &s = h.slab[box];
        lo[0] = s.i0; hi[0] = s.i1; lo[1] = s.j0; hi[1] = s.j1; lo[2] = s.k0; hi[2] = s.k1;
        return;
    }
    const int z = box - h.n_slab;
    lo[0] = h.ix0; hi[0] = h.ix1; lo[1] = h.iy0; hi[1] = h.iy1;
    lo[2] = z == 0 ? h.zlo : (z == 1 ? std::max(h.iz1, h.iz0) : h.iz0);
    hi[2] = z == 0 ? h.iz0 : (z == 1 ? h.nz : h.iz1);
}
// Column quads of a box: rows start at i0 rounded down to a multiple of four.
struct ResRange {
    int lo[3], hi[3];
    int np, nj, nq;               // quads per row, rows per plane, quads (0: empty box)
    ResRange(const Board &h, int box)
    {
        res_box_range(h, box, lo, hi);
        np = (hi[0] - (lo[0] & ~3) + 3) / 4;
        nj = hi[1] - lo[1];
        nq = hi[0] > lo[0] && nj > 0 && hi[2] > lo[2] ? np * nj * (hi[2] - lo[2]) : 0;
    }
    bool holds(int i, int j, int k) const
    {
        return nq > 0 && i >= lo[0] && i < hi[0] && j >= lo[1] && j < hi[1] && k >= lo[2] && k < hi[2];
    }
    int quad(int i, int j, int k) const { return ((k - lo[2]) * nj + (j - lo[1])) * np + (i - (lo[0] & ~3)) / 4; }
    int units() const { return (nq + 31) / 32; }
};
inline int res_box_of(const Board &h, int i, int j, int k)
{
    for (int x = 0; x < res_boxes(h); ++x)
        if (ResRange(h, x).holds(i, j, k)) return x;
    return -1;
}

// Relative cost of a unit of a box: an interior unit 10; a graded box more with
// every auxiliary, and more again where its rows are short, so that a warp
// touches many row segments.  The constants are those of the best step time
// over boards of 0.25 to 14 M cells and 24 boards at once, in us: 97x61x43
// 7.9, 232x192x39 21.7, 280x230x100 92.0, 420x335x100 215, 24 boards 608.  With
// 13 + ... + 9: 8.4, 22.1, 95.4, 219, 620; 10 + ... + 12: 8.3, 21.8, 89.5, -,
// 608; graded boxes a tenth lighter or short rows + 7: 24 boards 639 and more.
inline int res_weight(const Board &h, int box)
{
    if (box == h.n_slab + 2) return 10;
    int naux = 2, width = h.ix1 - h.ix0;
    if (box < h.n_slab) {
        naux = 0;
        for (int a = 0; a < 6; ++a) naux += h.slab[box].aux[a] != nullptr;
        width = h.slab[box].ni;
    }
    return 11 + (8 * naux + 4) / 5 + (width < 64 ? 11 : 0);
}

// Work of a step of a board, in those weights.
inline double res_work(const Board &h)
{
    double total = 0.0;
    for (int x = 0; x < res_boxes(h); ++x) total += (double)ResRange(h, x).units() * res_weight(h, x);
    return total;
}

struct ResAt {                    // a source or probe edge
    int i, j, k, comp, probe, index;
};

struct ResHost {
    std::vector<ResTeam> teams;
    std::vector<ResBlock> blocks;
    std::vector<ResPiece> pieces;
    std::vector<ResPort> ports;
    int max_pieces = 1, max_ports = 1, max_factors = 1, max_units = 0;
};

// Whether a board's units fit nblk blocks at one a warp.
inline bool res_pinned(const Board &h, int nblk)
{
    int units = 0;
    for (int x = 0; x < res_boxes(h); ++x) units += ResRange(h, x).units();
    return units <= nblk * kPinWarps;
}

// Add the team that advances board number b on nblk blocks: the boxes' units
// go to the blocks in turn, each up to its share of the weight, or of the
// units' number where each warp keeps one unit.
inline void res_team(const Board &h, const std::vector<ResAt> &at, int b, int nblk, ResHost &R)
{
    const int nbox = res_boxes(h);
    std::vector<ResRange> box;
    for (int x = 0; x < nbox; ++x) box.emplace_back(h, x);
    const bool pinned = res_pinned(h, nblk);
    double total = 0.0;
    for (int x = 0; x < nbox; ++x) total += (double)box[x].units() * (pinned ? 1 : res_weight(h, x));
    std::vector<std::vector<ResPiece>> mine(nblk);
    std::vector<int> count(nblk, 0);
    double done = 0.0;
    int blk = 0;
    for (int x = 0; x < nbox; ++x) {
        const int units = box[x].units(), w = pinned ? 1 : res_weight(h, x);
        for (int u = 0; u < units;) {
            const double want = total * (blk + 1) / nblk;
            const int take = blk == nblk - 1 ? units - u
                                             : std::min(units - u, std::max(0, (int)std::floor((want - done) / w + 0.5)));
            if (take > 0) {
                mine[blk].push_back({x, 32 * u, std::min(box[x].nq - 32 * u, 32 * take), count[blk]});
                count[blk] += take;
                u += take;
                done += (double)take * w;
            }
            if (blk < nblk - 1 && (take == 0 || done + 0.5 * w >= want)) ++blk;
        }
    }
    std::vector<std::vector<ResPort>> port(nblk);
    for (const ResAt &a : at) {
        const int x = res_box_of(h, a.i, a.j, a.k);
        if (x < 0) continue;
        const int t = box[x].quad(a.i, a.j, a.k);
        for (int q = 0; q < nblk; ++q)
            for (const ResPiece &p : mine[q])
                if (p.box == x && t >= p.t0 && t < p.t0 + p.nq)
                    port[q].push_back({p.unit0 + (t - p.t0) / 32, (short)((t - p.t0) % 32), (short)(a.i & 3), (short)a.comp,
                                       (short)a.probe, a.index});
    }
    const int team = (int)R.teams.size();
    R.teams.push_back({b, nblk});
    for (int q = 0; q < nblk; ++q) {
        R.blocks.push_back({team, q == 0, (int)R.pieces.size(), (int)mine[q].size(), (int)R.ports.size(), (int)port[q].size()});
        R.pieces.insert(R.pieces.end(), mine[q].begin(), mine[q].end());
        R.ports.insert(R.ports.end(), port[q].begin(), port[q].end());
        R.max_units = std::max(R.max_units, count[q]);
        R.max_pieces = std::max(R.max_pieces, (int)mine[q].size());
        R.max_ports = std::max(R.max_ports, (int)port[q].size());
    }
    R.max_factors = std::max(R.max_factors, 8 * (res_fac_len(h.nx) + res_fac_len(h.ny) + res_fac_len(h.nz)));
}

// Boards of a batch grouped so that the states of a group (bytes each) together
// stay within cap, at most `most` boards a group: largest first, each into the
// first group with room; a board larger than cap is a group of its own.
inline std::vector<std::vector<int>> res_groups(const std::vector<double> &bytes, double cap, int most)
{
    std::vector<int> order(bytes.size());
    for (size_t b = 0; b < order.size(); ++b) order[b] = (int)b;
    std::stable_sort(order.begin(), order.end(), [&](int x, int y) { return bytes[x] > bytes[y]; });
    std::vector<std::vector<int>> group;
    std::vector<double> used;
    for (int b : order) {
        size_t g = 0;
        while (g < group.size() && (used[g] + bytes[b] > cap || (int)group[g].size() >= most)) ++g;
        if (g == group.size()) {
            group.emplace_back();
            used.push_back(0.0);
        }
        group[g].push_back(b);
        used[g] += bytes[b];
    }
    return group;
}

// Blocks for the boards of a group: one each, then one by one to the board with
// the most work per block.
inline std::vector<int> res_share(const std::vector<double> &work, int blocks)
{
    std::vector<int> n(work.size(), 1);
    for (int left = blocks - (int)n.size(); left > 0; --left) {
        size_t most = 0;
        for (size_t t = 1; t < n.size(); ++t)
            if (work[t] * n[most] > work[most] * n[t]) most = t;
        ++n[most];
    }
    return n;
}

}  // namespace fdtd
