// fdtd_resident.cu -- many leapfrog steps in one launch (Model section:
// H^{n+1/2} from E^n, then E^{n+1} from H and J; Eqs. 1-5 in the UPML; Eq. 8
// sources; probe samples).
//
// What bounds a small board in the launch-per-phase path is its chain of
// dependent launches: five per step, each a chain of plane or node marches,
// 56-62 us a step on boards of 25 k to 250 k cells whatever their size.
// k_resident is one cooperative launch for many steps: every block keeps the
// same nodes for all of them, a step is an H phase and an E phase, and a
// barrier ends each (1.2 us measured over 152 blocks).  Nothing is recomputed
// and nothing is staged: all reads of a phase are of values the phases before
// it finished, so every warp issues its loads at once and L2 serves them
// (12-13.7 TB/s measured up to 90 MB).  A phase is bound by L2 latency and the
// barrier on small boards, by the load pipe's wavefronts in the middle (with
// H held in shared memory 232x192x39 gained only 1 %), past L2 by HBM at 73 B a
// node and step.
//
// Measured (us a step, launch-per-phase path as it was before this file ->
// here): 38x33x20 57 -> 4.5 and 56x48x30 62 -> 4.5 (k_pinned), 181x131x6 34 ->
// 5.9, 232x192x39 90 -> 21.7, 280x230x100 160 -> 92; a batch of 24 boards (41 M
// cells) 852 -> 607.  Larger boards: see kResPoints.
//
// The work is cut into units of 32 column quads (128 nodes), taken in x, y, z
// order from one box at a time.  The boxes are the board's own (slab boxes,
// the two z-UPML boxes of the fused region, the interior), because a box
// decides which auxiliaries its nodes carry and where they lie; the update of
// a node is the arithmetic of the launch-per-phase kernels, so the fields,
// auxiliaries and traces come out bit for bit the same and a board may change
// between the two at any step.
#include "fdtd_device.h"

namespace fdtd {

namespace {

// Graded: UPML factors along some axis.  GradedX: along x.  Low: the box holds
// nodes on a low wall plane behind a PEC wall (their image is 0).  Walls: it
// holds nodes on a high wall plane, or on a low one behind a PMC wall.  Whole: its quads lie whole inside it, and so do
// those of its auxiliary arrays (16-byte accesses).  Parity: B~z alternates
// between two arrays.
enum : int { kGraded = 1, kGradedX = 2, kWalls = 4, kWhole = 8, kParity = 16, kLow = 32 };

struct BoxS {     // one box of the board
    float *aux[6];          // auxiliary read and written (nullptr: none)
    float *zb[2];           // z-UPML boxes: B~z by step parity (replaces aux[5])
    int flags;
    int i0, i1, ie;         // ie: i0 rounded down to a whole quad
    int j0, k0;
    int np, nj;             // quads per row, rows per plane
    unsigned mp, mj;        // reciprocals of np and nj
    int sp, sj;
    int apitch;             // row pitch of the auxiliaries (nj rows per plane)
    int pad;
};

struct BoardS {   // the block's board, in shared memory
    float *f[3];                // field sets: six components, NN nodes apart
    const void *cid;
    const float4 *ctab;         // rows of 1 / eps_r for 16-bit ids (the block keeps a copy of those of 8-bit ids)
    float *trace;
    int *status;
    double dt;
    long long step0;
    float scale;
    int n_total;
    int X, P, NN, id16;         // strides of a row, a plane and a component
    int nact;                   // steps this launch advances the board
    int first, work, last;      // field sets: read by the first step, kept in place between, written by the last
    int n[3];
    int wall[6];
    float S[3];
    int fac[3][2];              // UPML factors in shared memory: float offset per axis and position
    int row;                    // coefficient rows in shared memory: byte offset
    int port, n_port, drive;    // sources and probes: offsets of their places and drives, and count
    BoxS box[kMaxSlab + 3];
};

struct Drive {    // a source of the block, its Eq. 8 value at the current step, and what a current source takes off E
    Source s;
    double w;
    float take;
};

extern __shared__ __align__(16) unsigned char smem[];
__device__ __forceinline__ BoardS &board_s() { return *reinterpret_cast<BoardS *>(smem); }

constexpr int kWarps = 16, kResThreads = 32 * kWarps, kPinThreads = 32 * kPinWarps;

// UPML factors of a quad or a row.  The block's copies are four arrays (b1, g, ap, am)
// per axis and position, so a quad's factors along x are four 16-byte reads
// and a row's along y or z four scalars.
__device__ __forceinline__ C4 fac_quad(int at, int n, int i)
{
    const float *f = reinterpret_cast<const float *>(smem) + at + i;
    const int m = res_fac_len(n);
    return C4{ld4(f), ld4(f + m), ld4(f + 2 * m), ld4(f + 3 * m)};
}
__device__ __forceinline__ C4 fac_row(int at, int n, int j)
{
    const float *f = reinterpret_cast<const float *>(smem) + at + j;
    const int m = res_fac_len(n);
    return C4{four(f[0]), four(f[m]), four(f[2 * m]), four(f[3 * m])};
}
// Walk of a warp through its units of a piece: quads t0 + 32 u + lane below end.
struct Walk {
    int np, nj, ie, i0, i1, apitch;
    unsigned mp, mj;
    int sp, sj, at0, row, plane;   // node index of a quad: at0 + 4 p + r row + kk plane (r: row of the box, kk: plane)
    __device__ __forceinline__ explicit Walk(const BoxS &x)
    {
        const BoardS &B = board_s();
        np = x.np; nj = x.nj; ie = x.ie; i0 = x.i0; i1 = x.i1; apitch = x.apitch;
        mp = x.mp; mj = x.mj; sp = x.sp; sj = x.sj;
        at0 = x.k0 * B.P + x.j0 * B.X + x.ie;
        row = B.X;
        plane = B.P - x.nj * B.X;
    }
};
struct Pos {
    int p, r, kk;           // quad of the row, row of the box, plane of the box
    int at, ax;             // node and auxiliary index
    unsigned own;           // bit q: node q of the quad belongs to the box
};
__device__ __forceinline__ Pos locate(const Walk &w, int t, int end, bool whole)
{
    Pos q;
    const bool live = t < end;
    t = min(t, end - 1);
    q.r = res_quot(t, w.mp, w.sp);
    q.p = t - q.r * w.np;
    q.kk = res_quot(q.r, w.mj, w.sj);
    q.at = w.at0 + 4 * q.p + q.r * w.row + q.kk * w.plane;
    q.own = 15u;
    if (!whole) {
        const int i = w.ie + 4 * q.p;
        q.own = (15u << max(w.i0 - i, 0)) & (15u >> max(i + 4 - w.i1, 0));
    }
    if (!live) q.own = 0;
    q.ax = q.r * w.apitch + 4 * q.p + (w.ie - w.i0);
    return q;
}

// Auxiliaries of a quad (only the box's own nodes lie in the array).
__device__ __forceinline__ F4 ldaux(const float *p, const Pos &q, bool whole)
{
    if (!p) return four(0.f);
    p += q.ax;
    if (whole) return ld4(p);
    F4 v = four(0.f);
    if (q.own & 1u) v.a.x = p[0];
    if (q.own & 2u) v.a.y = p[1];
    if (q.own & 4u) v.b.x = p[2];
    if (q.own & 8u) v.b.y = p[3];
    return v;
}
__device__ __forceinline__ void staux(float *p, const Pos &q, const F4 &v, unsigned own, bool whole)
{
    if (!p) return;
    p += q.ax;
    if (whole) {
        if (own) *reinterpret_cast<float4 *>(p) = make_float4(v.a.x, v.a.y, v.b.x, v.b.y);
        return;
    }
    if (own & 1u) p[0] = v.a.x;
    if (own & 2u) p[1] = v.a.y;
    if (own & 4u) p[2] = v.b.x;
    if (own & 8u) p[3] = v.b.y;
}

// Auxiliary array of component c of a box, read from shared memory at each use
// (held in registers, the six pointers of a graded box would spill); B~z of the
// z-UPML boxes by parity.
__device__ __forceinline__ float *aux_of(const BoxS &x, int c, int par = -1)
{
    unsigned long long v;
    float *const *p = par >= 0 && (x.flags & kParity) ? &x.zb[par] : &x.aux[c];
    asm volatile("ld.shared.u64 %0, [%1];" : "=l"(v) : "r"((unsigned)__cvta_generic_to_shared(p)));
    return (float *)v;
}

// H~^{n+1/2} of the units turn, turn + kWarps, ... < nu of a piece, from field
// set I into set O.  G: the box is graded or touches an outer wall.
template <bool G>
__device__ __forceinline__ void run_h(const BoxS &x, int t0, int end, int turn, int nu, const float *I, float *O, int par)
{
    const BoardS &B = board_s();
    const int lane = threadIdx.x & 31;
    const Walk w(x);
    const bool whole = (x.flags & kWhole) != 0, GX = (x.flags & kGradedX) != 0;
    const int X = B.X, P = B.P, N = B.NN;
    for (int u = turn; u < nu; u += kWarps) {
        const Pos q = locate(w, t0 + 32 * u + lane, end, whole);
        const int at = q.at;
        // neighbours past the grid's last column, row or plane read the next
        // component's memory: in bounds, and used only by nodes that are not stored
        const F4 ex = ld4(I + at), ey = ld4(I + (at + N)), ez = ld4(I + (at + 2 * N));
        const float eyi = I[at + N + 4], ezi = I[at + 2 * N + 4];
        const F4 exj = ld4(I + (at + X)), ezj = ld4(I + (at + 2 * N + X));
        const F4 exk = ld4(I + (at + P)), eyk = ld4(I + (at + N + P));
        const F4 ox = ld4(I + (at + 3 * N)), oy = ld4(I + (at + 4 * N)), oz = ld4(I + (at + 5 * N));
        F4 b0, b1, b2;
        if (G) {
            b0 = ldaux(aux_of(x, 3), q, whole);
            b1 = ldaux(aux_of(x, 4), q, whole);
            b2 = ldaux(aux_of(x, 5, par), q, whole);
        }
        const float Sx = B.S[0], Sy = B.S[1], Sz = B.S[2];
        const F4 eyr{make_float2(ey.a.y, ey.b.x), make_float2(ey.b.y, eyi)};   // E_y, E_z at i + 1
        const F4 ezr{make_float2(ez.a.y, ez.b.x), make_float2(ez.b.y, ezi)};
        const F4 cx = curl4(ezj, ez, eyk, ey, Sy, Sz);
        const F4 cy = curl4(exk, ex, ezr, ez, Sz, Sx);
        const F4 cz = curl4(eyr, ey, exj, ex, Sx, Sy);
        if (!G) {
            st4(O + (at + 3 * N), sub4(ox, cx), q.own);
            st4(O + (at + 4 * N), sub4(oy, cy), q.own);
            st4(O + (at + 5 * N), sub4(oz, cz), q.own);
            continue;
        }
        const int i = w.ie + 4 * q.p, j = x.j0 + q.r - q.kk * w.nj, k = x.k0 + q.kk;
        unsigned mx = q.own, my = q.own, mz = q.own;
        if (x.flags & kWalls) {   // samples that exist: not past the last row, column or plane
            const bool yin = j < B.n[1], zin = k < B.n[2];
            const unsigned xin = below(i, B.n[0]);
            if (!(yin && zin)) mx = 0;
            my = zin ? my & xin : 0u;
            mz = yin ? mz & xin : 0u;
        }
        F4 n;
        {
            float *const a = aux_of(x, 3);
            const F4 h = upml_h4(ox, cx, fac_row(B.fac[1][1], B.n[1], j), fac_row(B.fac[2][1], B.n[2], k),
                                 GX ? fac_quad(B.fac[0][0], B.n[0], i) : fac_one(), a != nullptr, b0, n);
            st4(O + (at + 3 * N), h, mx);
            staux(a, q, n, mx, whole);
        }
        {
            float *const a = aux_of(x, 4);
            const F4 h = upml_h4(oy, cy, fac_row(B.fac[2][1], B.n[2], k), GX ? fac_quad(B.fac[0][1], B.n[0], i) : fac_one(),
                                 fac_row(B.fac[1][0], B.n[1], j), a != nullptr, b1, n);
            st4(O + (at + 4 * N), h, my);
            staux(a, q, n, my, whole);
        }
        {
            float *const a = aux_of(x, 5, par ^ 1);
            const F4 h = upml_h4(oz, cz, GX ? fac_quad(B.fac[0][1], B.n[0], i) : fac_one(), fac_row(B.fac[1][1], B.n[1], j),
                                 fac_row(B.fac[2][0], B.n[2], k), a != nullptr, b2, n);
            st4(O + (at + 5 * N), h, mz);
            staux(a, q, n, mz, whole);
        }
    }
}

__device__ __forceinline__ void images(const BoardS &B, int i, int j, int k, F4 &hyx, F4 &hzx, F4 &hxy, F4 &hzy, F4 &hxz, F4 &hyz,
                                       F4 &hyl, F4 &hzl, F4 &hxj, F4 &hzj, F4 &hxk, F4 &hyk)
{
    image_x(i, B.n[0], B.wall[0], B.wall[1], hyx, hyl);
    image_x(i, B.n[0], B.wall[0], B.wall[1], hzx, hzl);
    image4(j == 0, j == B.n[1], B.wall[2], B.wall[3], hxy, hxj);
    image4(j == 0, j == B.n[1], B.wall[2], B.wall[3], hzy, hzj);
    image4(k == 0, k == B.n[2], B.wall[4], B.wall[5], hxz, hxk);
    image4(k == 0, k == B.n[2], B.wall[4], B.wall[5], hyz, hyk);
}

// 1 / eps_r of a quad's edges from its ids.
__device__ __forceinline__ void rows_of(const BoardS &B, bool id16, const uint2 &id, F4 &kx, F4 &ky, F4 &kz)
{
    float4 r0, r1, r2, r3;
    if (id16) {
        const float4 *const r = B.ctab;
        r0 = __ldg(r + (id.x & 0xffffu)); r1 = __ldg(r + (id.x >> 16));
        r2 = __ldg(r + (id.y & 0xffffu)); r3 = __ldg(r + (id.y >> 16));
    } else {
        const float4 *const r = reinterpret_cast<const float4 *>(smem + B.row);
        r0 = r[id.x & 0xffu]; r1 = r[(id.x >> 8) & 0xffu]; r2 = r[(id.x >> 16) & 0xffu]; r3 = r[id.x >> 24];
    }
    kx = F4{make_float2(r0.x, r1.x), make_float2(r2.x, r3.x)};
    ky = F4{make_float2(r0.y, r1.y), make_float2(r2.y, r3.y)};
    kz = F4{make_float2(r0.z, r1.z), make_float2(r2.z, r3.z)};
}

// The block's sources on edges of unit `unit`, in order (several may share an
// edge), then its probe samples: nx, ny, nz is the new E of the lane's quad, ex,
// ey, ez its E before.
__device__ __forceinline__ void work_ports(int unit, int s, F4 &nx, F4 &ny, F4 &nz, const F4 &ex, const F4 &ey, const F4 &ez)
{
    const BoardS &B = board_s();
    const int lane = threadIdx.x & 31;
    const ResPort *const list = reinterpret_cast<const ResPort *>(smem + B.port);
    for (int v0 = 0; v0 < B.n_port; v0 += 32) {
        const int mine = v0 + lane;
        unsigned hit = __ballot_sync(0xffffffffu, mine < B.n_port && list[mine].unit == unit);
        for (; hit; hit &= hit - 1) {
            const int v = v0 + __ffs(hit) - 1;
            const ResPort &p = list[v];
            if (p.lane != lane) continue;
            const int e = p.col;
            const float now = get(p.comp == 0 ? nx : p.comp == 1 ? ny : nz, e);
            if (p.probe) {
                const float f = now * B.scale;
                const long long n = B.step0 + s;
                if (n < (long long)B.n_total) B.trace[(long long)p.index * B.n_total + n] = f;
                if (!isfinite(f)) atomicOr(B.status, kStatusNonFinite);
            } else {
                const Drive &d = reinterpret_cast<const Drive *>(smem + B.drive)[v];
                const float f = d.s.kind == kSrcCurrent
                                    ? __fsub_rn(now, d.take)
                                    : src_apply(d.s, d.w, now, get(p.comp == 0 ? ex : p.comp == 1 ? ey : ez, e));
                if (p.comp == 0) set(nx, e, f);
                else if (p.comp == 1) set(ny, e, f);
                else set(nz, e, f);
            }
        }
    }
}

// E^{n+1} of the units turn, turn - kWarps, ... > stop of a piece: E^n from set
// I, H~^{n+1/2} from set O, into set O.  PORTS: the units hold sources or probes
// (unit `base + u` of the block, local step s).
template <bool G, bool PORTS>
__device__ __forceinline__ void run_e(const BoxS &x, int t0, int end, int turn, int stop, const float *I, float *O, int s, int base)
{
    const BoardS &B = board_s();
    const int lane = threadIdx.x & 31;
    const Walk w(x);
    const bool whole = (x.flags & kWhole) != 0, GX = (x.flags & kGradedX) != 0;
    const int X = B.X, P = B.P, N = B.NN;
    const void *const cid = B.cid;
    const bool id16 = B.id16 != 0;
    for (int u = turn; u > stop; u -= kWarps) {
        const Pos q = locate(w, t0 + 32 * u + lane, end, whole);
        const int at = q.at;
        uint2 id;
        if (id16) id = *reinterpret_cast<const uint2 *>((const uint16_t *)cid + at);
        else id.x = *reinterpret_cast<const unsigned *>((const uint8_t *)cid + at);
        // neighbours before the grid's first column, row or plane read the
        // previous component's memory: in bounds, and replaced by the wall's image below
        const F4 hx = ld4(O + (at + 3 * N)), hy = ld4(O + (at + 4 * N)), hz = ld4(O + (at + 5 * N));
        const float hyi = O[at + 4 * N - 1], hzi = O[at + 5 * N - 1];
        F4 hxj = ld4(O + (at + 3 * N - X)), hzj = ld4(O + (at + 5 * N - X));
        F4 hxk = ld4(O + (at + 3 * N - P)), hyk = ld4(O + (at + 4 * N - P));
        const F4 ex = ld4(I + at), ey = ld4(I + (at + N)), ez = ld4(I + (at + 2 * N));
        F4 d0, d1, d2;
        if (G) {
            d0 = ldaux(aux_of(x, 0), q, whole);
            d1 = ldaux(aux_of(x, 1), q, whole);
            d2 = ldaux(aux_of(x, 2), q, whole);
        }
        const float Sx = B.S[0], Sy = B.S[1], Sz = B.S[2];
        F4 hyl{make_float2(hyi, hy.a.x), make_float2(hy.a.y, hy.b.x)};   // H~y, H~z at i - 1
        F4 hzl{make_float2(hzi, hz.a.x), make_float2(hz.a.y, hz.b.x)};
        unsigned mx = q.own, my = q.own, mz = q.own;
        const int i = w.ie + 4 * q.p, j = x.j0 + q.r - q.kk * w.nj, k = x.k0 + q.kk;
        F4 cx, cy, cz;
        if (G && (x.flags & kWalls)) {
            // H~ on the + side of the node, per axis of difference
            F4 hyx = hy, hzx = hz, hxy = hx, hzy = hz, hxz = hx, hyz = hy;
            images(B, i, j, k, hyx, hzx, hxy, hzy, hxz, hyz, hyl, hzl, hxj, hzj, hxk, hyk);
            mx &= below(i, B.n[0]);
            if (j >= B.n[1]) my = 0;
            if (k >= B.n[2]) mz = 0;
            cx = curl4(hzy, hzj, hyz, hyk, Sy, Sz);
            cy = curl4(hxz, hxk, hzx, hzl, Sz, Sx);
            cz = curl4(hyx, hyl, hxy, hxj, Sx, Sy);
        } else {
            if (G && (x.flags & kLow)) {   // what lies across a low PEC wall counts as 0
                if (i == 0) hyl.a.x = hzl.a.x = 0.f;
                if (j == 0) hxj = hzj = four(0.f);
                if (k == 0) hxk = hyk = four(0.f);
            }
            cx = curl4(hz, hzj, hy, hyk, Sy, Sz);
            cy = curl4(hx, hxk, hz, hzl, Sz, Sx);
            cz = curl4(hy, hyl, hx, hxj, Sx, Sy);
        }
        F4 kx, ky, kz;
        rows_of(B, id16, id, kx, ky, kz);
        F4 nx, ny, nz;
        if (!G) {
            nx = fma4(kx, cx, ex);
            ny = fma4(ky, cy, ey);
            nz = fma4(kz, cz, ez);
        } else {
            F4 n;
            {
                float *const a = aux_of(x, 0);
                nx = upml_e4(ex, cx, kx, fac_row(B.fac[1][0], B.n[1], j), fac_row(B.fac[2][0], B.n[2], k),
                             GX ? fac_quad(B.fac[0][1], B.n[0], i) : fac_one(), a != nullptr, d0, n);
                staux(a, q, n, mx, whole);
            }
            {
                float *const a = aux_of(x, 1);
                ny = upml_e4(ey, cy, ky, fac_row(B.fac[2][0], B.n[2], k), GX ? fac_quad(B.fac[0][0], B.n[0], i) : fac_one(),
                             fac_row(B.fac[1][1], B.n[1], j), a != nullptr, d1, n);
                staux(a, q, n, my, whole);
            }
            {
                float *const a = aux_of(x, 2);
                nz = upml_e4(ez, cz, kz, GX ? fac_quad(B.fac[0][0], B.n[0], i) : fac_one(), fac_row(B.fac[1][0], B.n[1], j),
                             fac_row(B.fac[2][1], B.n[2], k), a != nullptr, d2, n);
                staux(a, q, n, mz, whole);
            }
        }
        if (PORTS) work_ports(base + u, s, nx, ny, nz, ex, ey, ez);
        st4(O + at, nx, mx);
        st4(O + (at + N), ny, my);
        st4(O + (at + 2 * N), nz, mz);
    }
}

// A unit that holds sources or probes: out of line, so that the others carry none of its state.
__device__ __noinline__ void port_unit(int bx, int t0, int end, int u, int si, int so, int s, int base)
{
    const BoardS &B = board_s();
    const BoxS &x = B.box[bx];
    if (x.flags & (kGraded | kWalls | kLow)) run_e<true, true>(x, t0, end, u, u - 1, B.f[si], B.f[so], s, base);
    else run_e<false, true>(x, t0, end, u, u - 1, B.f[si], B.f[so], s, base);
}

// Shared tables of a block, built from the board's descriptor at the start of
// a launch (a descriptor may change between launches).
__device__ void fill_board(const Board *B, BoardS &o, int nsteps)
{
    for (int s = 0; s < 3; ++s) o.f[s] = (float *)B->f[s][0];
    o.n[0] = B->nx; o.n[1] = B->ny; o.n[2] = B->nz;
    for (int a = 0; a < 3; ++a) o.S[a] = B->S[a];
    o.cid = B->cid;
    o.ctab = B->ctab;
    o.trace = B->trace;
    o.status = B->status;
    o.dt = B->dt;
    o.scale = B->scale;
    o.n_total = B->n_total;
    o.P = (int)B->plane;
    o.X = B->pitch;
    o.NN = (int)B->nodes;
    o.id16 = B->id16;
    for (int w = 0; w < 6; ++w) o.wall[w] = B->wall[w];
    o.step0 = *((volatile long long *)B->step);
    const long long left = *((volatile long long *)B->stop) - o.step0;
    o.nact = (int)(left < 0 ? 0 : (left < nsteps ? left : nsteps));
    // H of a node is written over by its own update alone, and so is E: all
    // steps but the last work in place in the set that has to hold the state
    // before the last (for the energy and checkpoints), so one field set and
    // not two has to stay in L2
    o.first = set_of(B->tdepth, o.step0);
    o.work = set_of(B->tdepth, o.step0 + o.nact - 1);
    o.last = set_of(B->tdepth, o.step0 + o.nact);
}
__device__ void fill_box(const Board *B, int kind, BoxS &o)
{
    int lo[3], hi[3];
    for (int c = 0; c < 6; ++c) o.aux[c] = nullptr;
    o.zb[0] = o.zb[1] = nullptr;
    o.flags = 0;
    if (kind < B->n_slab) {
        const Slab &s = B->slab[kind];
        lo[0] = s.i0; hi[0] = s.i1; lo[1] = s.j0; hi[1] = s.j1; lo[2] = s.k0; hi[2] = s.k1;
        for (int c = 0; c < 6; ++c) o.aux[c] = s.aux[c];
        o.apitch = s.ni;
        o.flags = kGraded;
        if (lo[0] < B->depth[0] || hi[0] > B->nx - B->depth[1]) o.flags |= kGradedX;
    } else {
        lo[0] = B->ix0; hi[0] = B->ix1; lo[1] = B->iy0; hi[1] = B->iy1;
        const int z = kind - B->n_slab;   // 0: below, 1: above, 2: between the z-UPML layers
        lo[2] = z == 0 ? B->zlo : (z == 1 ? max(B->iz1, B->iz0) : B->iz0);
        hi[2] = z == 0 ? B->iz0 : (z == 1 ? B->nz : B->iz1);
        if (z < 2) {
            o.aux[2] = B->zD[z];
            o.aux[5] = B->zB[z][0];
            o.zb[0] = B->zB[z][0];
            o.zb[1] = B->zB[z][1];
            o.flags = kGraded | kParity;
        }
        o.apitch = B->zpitch;
    }
    const int n[3] = {B->nx, B->ny, B->nz};
    for (int a = 0; a < 3; ++a)
        if (hi[a] > n[a] || (lo[a] == 0 && B->wall[2 * a] != 0)) o.flags |= kWalls;
        else if (lo[a] == 0) o.flags |= kLow;
    if ((lo[0] & 3) == 0 && (hi[0] & 3) == 0 && (o.apitch & 3) == 0) o.flags |= kWhole;
    o.i0 = lo[0]; o.i1 = hi[0]; o.ie = lo[0] & ~3; o.j0 = lo[1]; o.k0 = lo[2];
    o.np = max((hi[0] - o.ie + 3) / 4, 1);
    o.nj = max(hi[1] - lo[1], 1);
    res_recip(o.np, o.mp, o.sp);
    res_recip(o.nj, o.mj, o.sj);
}

// Shared memory, in this order: the board with its boxes, pieces, ports,
// drives, coefficient rows, UPML factors.
struct Layout {
    int piece, port, drive, row, fac, bytes;
};
__host__ __device__ inline Layout layout_of(const ResPlan &p)
{
    Layout l;
    auto up = [](size_t x) { return (int)((x + 15) & ~(size_t)15); };
    l.piece = up(sizeof(BoardS));
    l.port = up(l.piece + sizeof(ResPiece) * p.max_pieces);
    l.drive = up(l.port + sizeof(ResPort) * p.max_ports);
    l.row = up(l.drive + sizeof(Drive) * p.max_ports);
    l.fac = l.row + (int)sizeof(float4) * kMaxCombo;
    l.bytes = l.fac + (int)sizeof(float) * p.max_factors;
    return l;
}

// Barrier of a team of blocks: `target` arrivals on a counter zeroed before
// the launch (release on arrival, acquire on the way out).  The wait is
// bounded; a block that gives up reports it and returns false, and the other
// blocks' waits run out alike.
__device__ __forceinline__ void team_arrive(unsigned *bar)
{
    __syncthreads();
    if (threadIdx.x == 0) asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(bar) : "memory");
}
__device__ __forceinline__ bool team_wait(unsigned *bar, unsigned target, int *status, int *gave_up,
                                          unsigned max_polls = kBarrierPolls)
{
    if (threadIdx.x == 0) {
        unsigned v = 0, it = 0;
        do asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(bar) : "memory");
        while (v < target && ++it < max_polls);
        if (v < target) {
            atomicOr(status, kStatusBarrier);
            *gave_up = 1;
        }
    }
    __syncthreads();
    return *(volatile int *)gave_up == 0;
}

// Fills a block's shared memory; ends with a barrier.  marks: units with a
// source or probe, by unit number modulo 1024.
__device__ __forceinline__ void set_up(const ResPlan &plan, const Layout &l, const ResBlock &blk, const Board *board, int nsteps,
                                       int *gave_up, unsigned *marks)
{
    BoardS &B = board_s();
    ResPiece *const piece = reinterpret_cast<ResPiece *>(smem + l.piece);
    ResPort *const port = reinterpret_cast<ResPort *>(smem + l.port);
    Drive *const drive = reinterpret_cast<Drive *>(smem + l.drive);
    const int tid = threadIdx.x, nt = blockDim.x;
    if (tid == 0) {
        fill_board(board, B, nsteps);
        int at = l.fac / 4;
        for (int a = 0; a < 3; ++a)
            for (int h = 0; h < 2; ++h) {
                B.fac[a][h] = at;
                at += 4 * res_fac_len(B.n[a]);
            }
        B.row = l.row;
        B.port = l.port;
        B.n_port = blk.n_port;
        B.drive = l.drive;
        *gave_up = 0;
    }
    for (int x = tid; x < board->n_slab + 3; x += nt) fill_box(board, x, B.box[x]);
    for (int x = tid; x < blk.n_piece; x += nt) piece[x] = plan.pieces[blk.piece0 + x];
    for (int x = tid; x < blk.n_port; x += nt) port[x] = plan.ports[blk.port0 + x];
    if (tid < 32) marks[tid] = 0;
    __syncthreads();
    for (int p = tid; p < blk.n_port; p += nt)
        if (!port[p].probe) drive[p].s = board->src[port[p].index];
    for (int p = tid; p < blk.n_port; p += nt) atomicOr(&marks[(port[p].unit >> 5) & 31], 1u << (port[p].unit & 31));
    if (!B.id16)
        for (int r = tid; r < kMaxCombo; r += nt) reinterpret_cast<float4 *>(smem + l.row)[r] = board->ctab[r];
    for (int a = 0; a < 3; ++a)
        for (int h = 0; h < 2; ++h) {
            const int m = res_fac_len(B.n[a]);
            float *const f = reinterpret_cast<float *>(smem) + B.fac[a][h];
            for (int r = tid; r < m; r += nt) {
                const Coef c = ldcoef(board->cw[a][h] + min(r, B.n[a]));
                f[r] = c.b1;
                f[m + r] = c.g;
                f[2 * m + r] = c.ap;
                f[3 * m + r] = c.am;
            }
        }
    __syncthreads();
}

// Eq. 8 of the block's sources at local step s (by one warp).
__device__ __forceinline__ void pulses(const Layout &l, const ResBlock &blk, int s)
{
    const BoardS &B = board_s();
    const ResPort *const port = reinterpret_cast<const ResPort *>(smem + l.port);
    Drive *const drive = reinterpret_cast<Drive *>(smem + l.drive);
    for (int q = threadIdx.x & 31; q < blk.n_port; q += 32)
        if (!port[q].probe) {
            drive[q].w = src_pulse(drive[q].s, B.step0 + s, B.dt);
            drive[q].take = (float)(drive[q].s.coef * drive[q].w);
        }
}

// A team of blocks advances one board; a launch holds one team per board.
// Every block updates H on its own pieces, waits for the team, updates E on
// them, waits, and so on.  The E phase takes the pieces and their units
// backwards, so that it starts with what the H phase left in L2 last, and the
// next H phase with what the E phase left last.
__global__ void __launch_bounds__(kResThreads, 1) k_resident(ResPlan plan, int nsteps)
{
    const Layout l = layout_of(plan);
    BoardS &B = board_s();
    const ResPiece *const piece = reinterpret_cast<const ResPiece *>(smem + l.piece);
    __shared__ int gave_up;
    __shared__ unsigned marks[32];
    const int tid = threadIdx.x, warp = tid >> 5;
    const ResBlock blk = plan.blocks[blockIdx.x];
    const ResTeam team = plan.teams[blk.team];
    const Board *const board = plan.boards[team.board];
    unsigned *const bar = plan.arrive + (size_t)blk.team * 32;   // a 128-byte line of its own
    set_up(plan, l, blk, board, nsteps, &gave_up, marks);
    const int nact = B.nact;
    unsigned target = 0;
    for (int s = 0; s < nact; ++s) {
        const float *const I = B.f[s == 0 ? B.first : B.work];
        float *const O = B.f[s == nact - 1 ? B.last : B.work];
        int turn = warp;   // units go round the warps, on from piece to piece
        for (int p = 0; p < blk.n_piece; ++p) {
            const ResPiece pc = piece[p];
            const int nu = (pc.nq + 31) >> 5;
            if (turn < nu) {
                const BoxS &x = B.box[pc.box];
                if (x.flags & (kGraded | kWalls | kLow)) run_h<true>(x, pc.t0, pc.t0 + pc.nq, turn, nu, I, O, (int)((B.step0 + s) & 1));
                else run_h<false>(x, pc.t0, pc.t0 + pc.nq, turn, nu, I, O, 0);
                turn += (nu - turn + kWarps - 1) / kWarps * kWarps;
            }
            turn -= nu;
        }
        team_arrive(bar);
        if (warp == 1) pulses(l, blk, s);   // while the block waits
        target += team.n_blocks;
        if (!team_wait(bar, target, B.status, &gave_up)) return;
        turn = warp;
        for (int p = blk.n_piece - 1; p >= 0; --p) {
            const ResPiece pc = piece[p];
            const int nu = (pc.nq + 31) >> 5;
            if (turn < nu) {
                const BoxS &x = B.box[pc.box];
                for (int v = nu - 1 - turn; v >= 0;) {
                    // units with a source or probe one by one, the others in runs between them
                    int f = v;
                    if (blk.n_port)
                        while (f >= 0 && !((marks[((pc.unit0 + f) >> 5) & 31] >> ((pc.unit0 + f) & 31)) & 1u)) f -= kWarps;
                    else f = -1;
                    if (f < v) {
                        const int stop = max(f, -1);
                        if (x.flags & (kGraded | kWalls | kLow)) run_e<true, false>(x, pc.t0, pc.t0 + pc.nq, v, stop, I, O, s, 0);
                        else run_e<false, false>(x, pc.t0, pc.t0 + pc.nq, v, stop, I, O, s, 0);
                    }
                    if (f >= 0)
                        port_unit(pc.box, pc.t0, pc.t0 + pc.nq, f, s == 0 ? B.first : B.work, s == nact - 1 ? B.last : B.work, s,
                                  pc.unit0);
                    v = f - kWarps;
                }
                turn += (nu - turn + kWarps - 1) / kWarps * kWarps;
            }
            turn -= nu;
        }
        team_arrive(bar);
        target += team.n_blocks;
        if (!team_wait(bar, target, B.status, &gave_up)) return;
    }
    // every block of the team has read the counters (before its first barrier)
    if (tid == 0 && nact > 0 && blk.first) *((volatile long long *)board->step) = B.step0 + nact;
}

// The same for boards of at most kPinWarps units a block.  There a step of
// k_resident is latency: two barriers, and in each phase the way from the
// barrier to the loads, L2, and back to the barrier.  Here a warp has one unit
// and a lane keeps its quad for the whole launch, its E, H~, auxiliaries and
// ids in registers, so that a phase is the six loads of its neighbours, the
// update and three stores.  (A quad cut by the box's edge reads itself again:
// its other nodes are some other lane's.)  38x33x20 5.65 -> 4.5, 56x48x30 5.95
// -> 4.5 us a step, of which the two barriers take 2.4.  Auxiliaries go back to memory at the
// end; B~z of the z-UPML boxes alternates between two arrays, so its last two
// values do.
__global__ void __launch_bounds__(kPinThreads, 1) k_pinned(ResPlan plan, int nsteps)
{
    const Layout l = layout_of(plan);
    BoardS &B = board_s();
    __shared__ int gave_up;
    __shared__ unsigned marks[32];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const ResBlock blk = plan.blocks[blockIdx.x];
    const ResTeam team = plan.teams[blk.team];
    const Board *const board = plan.boards[team.board];
    unsigned *const bar = plan.arrive + (size_t)blk.team * 32;
    set_up(plan, l, blk, board, nsteps, &gave_up, marks);
    const int nact = B.nact, X = B.X, P = B.P, N = B.NN;
    // the warp's unit and the lane's quad
    ResPiece pc{0, 0, 0, 0};
    bool live = false;
    for (int p = 0; p < blk.n_piece && !live; ++p) {
        pc = reinterpret_cast<const ResPiece *>(smem + l.piece)[p];
        live = warp >= pc.unit0 && warp < pc.unit0 + ((pc.nq + 31) >> 5);
    }
    live = live && nact > 0;
    const BoxS &x = B.box[live ? pc.box : 0];
    const bool whole = (x.flags & kWhole) != 0, gx = (x.flags & kGradedX) != 0;
    const bool graded = (x.flags & (kGraded | kWalls | kLow)) != 0;
    const bool ports = live && ((marks[warp >> 5] >> (warp & 31)) & 1u);
    Pos q{};
    int i = 0, j = 0, k = 0;
    unsigned mh[3] = {0, 0, 0}, me[3] = {0, 0, 0};   // nodes of the quad whose H~, E exist
    F4 ex{}, ey{}, ez{}, hx{}, hy{}, hz{}, b0{}, b1{}, b2{}, d0{}, d1{}, d2{};
    unsigned kept = 0;                               // auxiliaries the box keeps (bit c)
    uint2 id = make_uint2(0, 0);
    const bool id16 = B.id16 != 0;
    if (live) {
        const Walk w(x);
        q = locate(w, pc.t0 + 32 * (warp - pc.unit0) + lane, pc.t0 + pc.nq, whole);
        i = w.ie + 4 * q.p; j = x.j0 + q.r - q.kk * w.nj; k = x.k0 + q.kk;
        const bool yin = j < B.n[1], zin = k < B.n[2];
        const unsigned bx = below(i, B.n[0]);
        mh[0] = yin && zin ? q.own : 0u; mh[1] = zin ? q.own & bx : 0u; mh[2] = yin ? q.own & bx : 0u;
        me[0] = q.own & bx; me[1] = yin ? q.own : 0u; me[2] = zin ? q.own : 0u;
        const float *const I = B.f[B.first];
        ex = ld4(I + q.at); ey = ld4(I + (q.at + N)); ez = ld4(I + (q.at + 2 * N));
        hx = ld4(I + (q.at + 3 * N)); hy = ld4(I + (q.at + 4 * N)); hz = ld4(I + (q.at + 5 * N));
        for (int c = 0; c < 6; ++c) kept |= (x.aux[c] != nullptr ? 1u : 0u) << c;
        const int par = (int)(B.step0 & 1);
        d0 = ldaux(x.aux[0], q, whole); d1 = ldaux(x.aux[1], q, whole); d2 = ldaux(x.aux[2], q, whole);
        b0 = ldaux(x.aux[3], q, whole); b1 = ldaux(x.aux[4], q, whole);
        b2 = ldaux(x.flags & kParity ? x.zb[par] : x.aux[5], q, whole);
        if (id16) id = *reinterpret_cast<const uint2 *>((const uint16_t *)B.cid + q.at);
        else id.x = *reinterpret_cast<const unsigned *>((const uint8_t *)B.cid + q.at);
    }
    const bool cut = q.own != 15u && q.own != 0u;
    const int at = q.at;
    unsigned target = 0;
    for (int s = 0; s < nact; ++s) {
        const float *const I = B.f[s == 0 ? B.first : B.work];
        float *const O = B.f[s == nact - 1 ? B.last : B.work];
        if (live) {
            const F4 exj = ld4(I + (at + X)), ezj = ld4(I + (at + 2 * N + X));
            const F4 exk = ld4(I + (at + P)), eyk = ld4(I + (at + N + P));
            const float eyi = I[at + N + 4], ezi = I[at + 2 * N + 4];
            F4 vy = ey, vz = ez;
            if (cut) { vy = ld4(I + (at + N)); vz = ld4(I + (at + 2 * N)); }
            const F4 cx = curl4(ezj, ez, eyk, ey, B.S[1], B.S[2]);
            const F4 cy = curl4(exk, ex, F4{make_float2(vz.a.y, vz.b.x), make_float2(vz.b.y, ezi)}, ez, B.S[2], B.S[0]);
            const F4 cz = curl4(F4{make_float2(vy.a.y, vy.b.x), make_float2(vy.b.y, eyi)}, ey, exj, ex, B.S[0], B.S[1]);
            if (!graded) {
                hx = sub4(hx, cx);
                hy = sub4(hy, cy);
                hz = sub4(hz, cz);
            } else {
                const C4 y1 = fac_row(B.fac[1][1], B.n[1], j), z1 = fac_row(B.fac[2][1], B.n[2], k);
                const C4 x1 = gx ? fac_quad(B.fac[0][1], B.n[0], i) : fac_one();
                F4 n;
                hx = upml_h4(hx, cx, y1, z1, gx ? fac_quad(B.fac[0][0], B.n[0], i) : fac_one(), kept & 8u, b0, n);
                if (kept & 8u) b0 = n;
                hy = upml_h4(hy, cy, z1, x1, fac_row(B.fac[1][0], B.n[1], j), kept & 16u, b1, n);
                if (kept & 16u) b1 = n;
                hz = upml_h4(hz, cz, x1, y1, fac_row(B.fac[2][0], B.n[2], k), kept & 32u, b2, n);
                if (kept & 32u) b2 = n;
            }
            st4(O + (at + 3 * N), hx, mh[0]);
            st4(O + (at + 4 * N), hy, mh[1]);
            st4(O + (at + 5 * N), hz, mh[2]);
        }
        team_arrive(bar);
        if (warp == 1) pulses(l, blk, s);   // while the block waits
        target += team.n_blocks;
        if (!team_wait(bar, target, B.status, &gave_up)) return;
        if (live) {
            F4 hxj = ld4(O + (at + 3 * N - X)), hzj = ld4(O + (at + 5 * N - X));
            F4 hxk = ld4(O + (at + 3 * N - P)), hyk = ld4(O + (at + 4 * N - P));
            const float hyi = O[at + 4 * N - 1], hzi = O[at + 5 * N - 1];
            F4 vy = hy, vz = hz;
            if (cut) { vy = ld4(O + (at + 4 * N)); vz = ld4(O + (at + 5 * N)); }
            F4 hyl{make_float2(hyi, vy.a.x), make_float2(vy.a.y, vy.b.x)};   // H~y, H~z at i - 1
            F4 hzl{make_float2(hzi, vz.a.x), make_float2(vz.a.y, vz.b.x)};
            // H~ on the + side of the node, per axis of difference
            F4 hyx = hy, hzx = hz, hxy = hx, hzy = hz, hxz = hx, hyz = hy;
            if (x.flags & kWalls) images(B, i, j, k, hyx, hzx, hxy, hzy, hxz, hyz, hyl, hzl, hxj, hzj, hxk, hyk);
            else if (x.flags & kLow) {
                if (i == 0) hyl.a.x = hzl.a.x = 0.f;
                if (j == 0) hxj = hzj = four(0.f);
                if (k == 0) hxk = hyk = four(0.f);
            }
            F4 kx, ky, kz;
            rows_of(B, id16, id, kx, ky, kz);
            const F4 cx = curl4(hzy, hzj, hyz, hyk, B.S[1], B.S[2]);
            const F4 cy = curl4(hxz, hxk, hzx, hzl, B.S[2], B.S[0]);
            const F4 cz = curl4(hyx, hyl, hxy, hxj, B.S[0], B.S[1]);
            F4 nx, ny, nz;
            if (!graded) {
                nx = fma4(kx, cx, ex);
                ny = fma4(ky, cy, ey);
                nz = fma4(kz, cz, ez);
            } else {
                const C4 y0 = fac_row(B.fac[1][0], B.n[1], j), z0 = fac_row(B.fac[2][0], B.n[2], k);
                const C4 x0 = gx ? fac_quad(B.fac[0][0], B.n[0], i) : fac_one();
                F4 n;
                nx = upml_e4(ex, cx, kx, y0, z0, gx ? fac_quad(B.fac[0][1], B.n[0], i) : fac_one(), kept & 1u, d0, n);
                if (kept & 1u) d0 = n;
                ny = upml_e4(ey, cy, ky, z0, x0, fac_row(B.fac[1][1], B.n[1], j), kept & 2u, d1, n);
                if (kept & 2u) d1 = n;
                nz = upml_e4(ez, cz, kz, x0, y0, fac_row(B.fac[2][1], B.n[2], k), kept & 4u, d2, n);
                if (kept & 4u) d2 = n;
            }
            if (ports) work_ports(warp, s, nx, ny, nz, ex, ey, ez);
            ex = nx; ey = ny; ez = nz;
            st4(O + at, ex, me[0]);
            st4(O + (at + N), ey, me[1]);
            st4(O + (at + 2 * N), ez, me[2]);
            if (s >= nact - 2 && (x.flags & kParity)) staux(x.zb[(B.step0 + s + 1) & 1], q, b2, mh[2], whole);
            if (s == nact - 1) {
                staux(x.aux[0], q, d0, me[0], whole);
                staux(x.aux[1], q, d1, me[1], whole);
                staux(x.aux[2], q, d2, me[2], whole);
                staux(x.aux[3], q, b0, mh[0], whole);
                staux(x.aux[4], q, b1, mh[1], whole);
                if (!(x.flags & kParity)) staux(x.aux[5], q, b2, mh[2], whole);
            }
        }
        team_arrive(bar);
        target += team.n_blocks;
        if (!team_wait(bar, target, B.status, &gave_up)) return;
    }
    if (tid == 0 && nact > 0 && blk.first) *((volatile long long *)board->step) = B.step0 + nact;
}

// Self-test of that bounded wait: a team of two of which one block arrives.
__global__ void k_barrier_selftest(int *status, unsigned *count, unsigned max_polls)
{
    __shared__ int gave_up;
    if (threadIdx.x == 0) gave_up = 0;
    team_arrive(count);
    team_wait(count, 2, status, &gave_up, max_polls);
}

}  // namespace

cudaError_t launch_barrier_selftest(int *status, unsigned *count, unsigned max_polls, cudaStream_t st)
{
    k_barrier_selftest<<<1, 32, 0, st>>>(status, count, max_polls);
    return cudaGetLastError();
}

size_t resident_smem(const ResPlan &p) { return (size_t)layout_of(p).bytes; }

cudaError_t resident_set_smem_limit()
{
    const cudaError_t e = cudaFuncSetAttribute(k_resident, cudaFuncAttributeMaxDynamicSharedMemorySize, kResSmem);
    return e != cudaSuccess ? e : cudaFuncSetAttribute(k_pinned, cudaFuncAttributeMaxDynamicSharedMemorySize, kResSmem);
}

size_t resident_arrive_bytes(int n_teams) { return (size_t)n_teams * 128; }

static bool pins(const ResPlan &plan) { return plan.max_units <= kPinWarps; }
static const void *kernel_of(const ResPlan &plan) { return pins(plan) ? (const void *)k_pinned : (const void *)k_resident; }
static int threads_of(const ResPlan &plan) { return pins(plan) ? kPinThreads : kResThreads; }

// The driver refuses a cooperative launch whose blocks cannot all be resident
// at once (too few SMs for this process, or too little of each).
bool resident_fits(const ResPlan &plan)
{
    int dev = 0, coop = 0, sms = 0, per = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kernel_of(plan), threads_of(plan), resident_smem(plan)) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return coop != 0 && plan.n_blocks <= sms * per;
}

cudaError_t launch_resident(const ResPlan &plan, int nsteps, cudaStream_t st)
{
    cudaError_t e = cudaMemsetAsync(plan.arrive, 0, resident_arrive_bytes(plan.all_teams), st);
    if (e != cudaSuccess) return e;
    ResPlan p = plan;
    void *args[] = {&p, &nsteps};
    return cudaLaunchCooperativeKernel(kernel_of(plan), dim3(plan.n_blocks), dim3(threads_of(plan)), args, resident_smem(plan), st);
}

}  // namespace fdtd
