"""Host plan of the resident launches, checked on the CPU.

csrc/resident_plan.h is compiled into a host program that builds plans for
boards of many shapes (odd extents, narrow and missing boxes, one box over the
whole grid) and block counts, and checks what the kernel relies on:
* every quad of every box belongs to exactly one piece, pieces hold whole
  units (but for a box's last) and number the block's units consecutively;
* a port names the block, unit, lane and node that update its edge;
* every address a quad's update reads lies inside the six components of a
  field set, also past the first and last row, column and plane;
* no block has much more than its share of the weight;
* groups hold every board once and stay within the cap; shares add up;
* res_quot divides exactly.
"""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1008_2602_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include <map>
#include "resident_plan.h"
using namespace fdtd;

static float some;   // an auxiliary that exists

static void add_box(Board &h, int i0, int i1, int j0, int j1, int k0, int k1, int naux)
{
    if (i1 <= i0 || j1 <= j0 || k1 <= k0) return;
    Slab &s = h.slab[h.n_slab++];
    s = Slab{};
    s.i0 = i0; s.i1 = i1; s.j0 = j0; s.j1 = j1; s.k0 = k0; s.k1 = k1;
    s.ni = i1 - i0; s.nj = j1 - j0;
    for (int a = 0; a < naux; ++a) s.aux[a] = &some;
}

// A board with its fused region [ix0,ix1) x [iy0,iy1) x [zlo,nz) and the boxes
// around it (hx, hy, hz: whether the high wall planes hold unknowns).
static Board board(int nx, int ny, int nz, int d, bool fused, bool high)
{
    Board h{};
    h.nx = nx; h.ny = ny; h.nz = nz;
    h.pitch = row_pitch(nx);
    h.plane = (long long)h.pitch * (ny + 1);
    h.nodes = h.plane * (nz + 1);
    const int xe = nx + high, ye = ny + high, ze = nz + high;
    if (!fused) {
        h.ix0 = h.ix1 = h.iy0 = h.iy1 = 0;
        h.iz0 = 1; h.iz1 = nz; h.zlo = 1;
        add_box(h, 0, nx + 1, 0, ny + 1, 0, nz + 1, 6);
        return h;
    }
    h.ix0 = d > 1 ? d : 1; h.ix1 = nx - d;
    h.iy0 = d > 1 ? d : 1; h.iy1 = ny - d;
    h.iz0 = d > 1 ? d : 1; h.iz1 = nz - d;
    h.zlo = d > 0 ? 0 : 1;
    const int a0 = (h.ix0 + 7) / 8 * 8, a1 = h.ix1 / 8 * 8;
    if (a1 - a0 >= 8) { h.ix0 = a0; h.ix1 = a1; }
    const int xs[4] = {0, h.ix0, h.ix1, xe}, ys[4] = {0, h.iy0, h.iy1, ye}, zs[4] = {0, h.iz0, h.iz1, ze};
    for (int z = 0; z < 3; ++z)
        for (int y = 0; y < 3; ++y)
            for (int x = 0; x < 3; ++x) {
                if (x == 1 && y == 1) continue;
                add_box(h, xs[x], xs[x + 1], ys[y], ys[y + 1], zs[z], zs[z + 1], x == 1 && z == 1 ? 2 : 6);
            }
    if (h.zlo == 1) add_box(h, h.ix0, h.ix1, h.iy0, h.iy1, 0, 1, 0);
    if (ze > nz) add_box(h, h.ix0, h.ix1, h.iy0, h.iy1, nz, ze, 0);
    return h;
}

int main()
{
    int bad = 0;
    const int shapes[][4] = {{5, 4, 3, 0}, {9, 8, 7, 2}, {37, 29, 23, 3}, {64, 40, 21, 4}, {150, 21, 31, 6},
                             {41, 31, 22, 0}, {232, 192, 39, 10}, {33, 90, 18, 5}, {3, 200, 2, 0}};
    for (const auto &s : shapes)
        for (int fused = 0; fused < 2; ++fused)
            for (int high = 0; high < 2; ++high)
                for (int nblk : {1, 2, 7, 19, 152}) {
                    const Board h = board(s[0], s[1], s[2], s[3], fused && s[0] > 2 * s[3] + 2, high);
                    std::vector<ResAt> at;
                    for (int t = 0; t < 40; ++t) {
                        ResAt a{rand() % (h.nx + high), rand() % (h.ny + high), rand() % (h.nz + high), t % 3, t & 1, t};
                        if (res_box_of(h, a.i, a.j, a.k) >= 0) at.push_back(a);
                    }
                    ResHost R;
                    res_team(h, at, 3, nblk, R);
                    bad += (int)R.blocks.size() != nblk || R.teams.size() != 1 || R.teams[0].board != 3 ||
                           R.teams[0].n_blocks != nblk;
                    std::vector<std::vector<int>> hit;
                    for (int x = 0; x < res_boxes(h); ++x) hit.emplace_back(ResRange(h, x).nq, 0);
                    double most = 0.0, heaviest = 0.0;
                    size_t pieces = 0, ports = 0;
                    for (const ResBlock &b : R.blocks) {
                        bad += b.piece0 != (int)pieces || b.port0 != (int)ports;
                        pieces += b.n_piece;
                        ports += b.n_port;
                        int unit = 0;
                        double w = 0.0;
                        for (int p = 0; p < b.n_piece; ++p) {
                            const ResPiece &pc = R.pieces[b.piece0 + p];
                            const ResRange r(h, pc.box);
                            bad += pc.unit0 != unit || pc.nq <= 0 || pc.t0 % 32 || (pc.nq % 32 && pc.t0 + pc.nq != r.nq);
                            for (int q = 0; q < pc.nq; ++q) ++hit[pc.box][pc.t0 + q];
                            unit += (pc.nq + 31) / 32;
                            w += (pc.nq + 31) / 32 * res_weight(h, pc.box);
                            heaviest = std::max(heaviest, (double)res_weight(h, pc.box));
                        }
                        most = std::max(most, w);
                        bad += b.n_piece > R.max_pieces || b.n_port > R.max_ports;
                    }
                    bad += pieces != R.pieces.size() || ports != R.ports.size() || ports != at.size();
                    for (const auto &v : hit)
                        for (int n : v) bad += n != 1;
                    bad += !res_pinned(h, nblk) && most > res_work(h) / nblk + 2 * heaviest;
                    bad += res_pinned(h, nblk) != (R.max_units <= kPinWarps);   // one unit a warp, or balanced
                    // ports: the node they name is theirs
                    std::map<int, int> seen;
                    for (const ResBlock &b : R.blocks)
                        for (int p = 0; p < b.n_port; ++p) {
                            const ResPort &q = R.ports[b.port0 + p];
                            ++seen[q.index];
                            const ResAt *a = nullptr;
                            for (const ResAt &v : at)
                                if (v.index == q.index) a = &v;
                            bool ok = a && a->comp == q.comp && a->probe == q.probe;
                            for (int c = 0; ok && c < b.n_piece; ++c) {
                                const ResPiece &pc = R.pieces[b.piece0 + c];
                                if (q.unit < pc.unit0 || q.unit >= pc.unit0 + (pc.nq + 31) / 32) continue;
                                const ResRange r(h, pc.box);
                                const int t = pc.t0 + 32 * (q.unit - pc.unit0) + q.lane, row = t / r.np;
                                ok = (r.lo[0] & ~3) + 4 * (t % r.np) + q.col == a->i && r.lo[1] + row % r.nj == a->j &&
                                     r.lo[2] + row / r.nj == a->k;
                            }
                            bad += !ok;
                        }
                    for (const auto &v : seen) bad += v.second != 1;
                    // addresses of a quad's update, in elements of a field set
                    for (int x = 0; x < res_boxes(h); ++x) {
                        const ResRange r(h, x);
                        if (!r.nq) continue;
                        const long long N = h.nodes, X = h.pitch, P = h.plane;
                        const long long lo = (long long)r.lo[2] * P + (long long)r.lo[1] * X + (r.lo[0] & ~3);
                        const long long hi = (long long)(r.hi[2] - 1) * P + (long long)(r.hi[1] - 1) * X + (r.lo[0] & ~3) +
                                             4 * (r.np - 1);
                        bad += lo + 3 * N - P < 0 || lo + 4 * N - P < 0 || lo + 3 * N - X < 0 || lo + 4 * N - 1 < 0;
                        for (long long v : {hi + 3, hi + N + 4, hi + 2 * N + 4, hi + X + 3, hi + 2 * N + X + 3, hi + P + 3,
                                            hi + N + P + 3, hi + 5 * N + 3})
                            bad += v >= 6 * N;
                        bad += hi + 3 >= N && hi + 3 >= h.nodes;          // ids: inside one volume
                        bad += (lo & 3) || (X & 3) || (P & 3) || (N & 3); // 16-byte accesses
                    }
                }
    // groups and shares
    for (int n = 1; n < 40; ++n) {
        std::vector<double> bytes, work;
        for (int b = 0; b < n; ++b) bytes.push_back(1.0 + rand() % 60), work.push_back(1.0 + rand() % 1000);
        std::vector<int> seen(n, 0);
        for (const auto &g : res_groups(bytes, 90.0, 5)) {
            double sum = 0.0;
            for (int b : g) { ++seen[b]; sum += bytes[b]; }
            bad += sum > 90.0 || g.empty() || g.size() > 5;
        }
        for (int v : seen) bad += v != 1;
        int sum = 0;
        for (int v : res_share(work, 152)) { sum += v; bad += v < 1; }
        bad += sum != 152;
    }
    bad += res_groups({200.0, 10.0}, 90.0, 5).size() != 2;   // one larger than the cap stands alone
    for (int t = 0; t < 400000; ++t) {
        const int d = 1 + (t % 3 == 0 ? t % 70 : rand() % (t % 3 == 1 ? 5000 : 1 << 20));
        const int v = t & 1 ? rand() & 0x7fffffff : (int)std::min(0x7fffffffll, (long long)d * (1 + rand() % 4000) - (t & 2 ? 1 : 0));
        unsigned m;
        int s;
        res_recip(d, m, s);
        bad += res_quot(v, m, s) != v / d;
    }
    std::printf("%d\n", bad);
    return bad != 0;
}
"""


def test_resident_plans_cover_the_board(tmp_path):
    gxx = shutil.which("g++")
    cuda_inc = "/usr/local/cuda/include"
    if gxx is None or not os.path.exists(os.path.join(cuda_inc, "cuda.h")):
        pytest.skip("g++ and the CUDA headers are needed to compile the host program")
    src = tmp_path / "plan.cpp"
    src.write_text(PROGRAM)
    exe = tmp_path / "plan"
    subprocess.run([gxx, "-std=c++17", "-O1", "-I", CSRC, "-I", cuda_inc, "-o", str(exe), str(src)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0 and r.stdout.strip() == "0", r.stdout
