// step_strip_block.cuh -- the marching form's step (step_strip.cuh) by blocks of 16 x 8 cells, for
// batches that hold too little work for marching warps.
//
// Every value is formed by the operations of step_strip.cuh, one for one, so that the two
// forms give the same bits: a batch may change from one to the other as instances come and
// go, and an instance's results still depend on its own grid only.  A marching warp does its
// rows one after the other, at least three rows' time in all; here a step is three short
// phases with barriers, as in cart_tile, whose division of a block among the threads this
// takes over: fbar+ of the block and its two-cell ring, every face once, every cell once, one
// each per thread.  Paired FP32 instructions do two velocities of a cell or face (the marching form:
// one velocity of two cells), which halves each thread's chain.
//
// Measured (GB300, us per step of a batch, marching / this form / cart_tile's blocks): 1 cavity of 32^2
// 4.5 / 2.7 / 3.0, 4 of 128^2 9.3 / 5.1 / 5.0, 1 of 256^2 8.5 / 5.0 / 5.0, 64 of 64^2 12.7 / 14.8 / 16.0, 256 of
// 32^2 36.4 / 15.4 / 16.0.  Two columns per thread, as in the marching form, took 3.5 and 5.8 us in the place
// of 2.7 and 5.0 (1 of 32^2, of 256^2).  Bound by the latency of the phases, and on full lists by issue.
#pragma once
#include "step_strip.cuh"

namespace sdugks {

using SB = CartShape<16, BATCH_TY>;
// The faces on the block's right edge: by a warp of their own (WIDE), or after its own faces by the
// warp of the top row's, whose upper half is free.  WIDE is the shorter chain, but only three such CTAs
// fit an SM: for lists that they hold at once.
template <bool WIDE> __host__ __device__ constexpr int sb_threads() { return 32 * (SB::WX + SB::WY + (WIDE ? 1 : 0)); }
template <bool WIDE> constexpr int sb_ctas() { return WIDE ? 3 : 4; }
static_assert(SB::NT == 32 * SB::WX && SB::LX * SB::LY <= sb_threads<false>(), "cells, then the ring, in one round of staging");

struct StripBlockSmem {
    float f[NQ * SB::PLANE], x[6 * SB::NSX], y[6 * SB::NSY];
    StripInst m;
};

// feq_pair for one cell, in pairs of velocities: o = out[0], then (1, 2), (3, 4), (5, 6), (7, 8).
__device__ __forceinline__ void feq_cell(float b0, float rho, float ux, float uy, float &o, float2 p[4])
{
    const float ss = __fmaf_rn(ux, ux, __fmul_rn(uy, uy));
    const float base = __fmaf_rn(__fmul_rn(-1.5f, rho), ss, b0);
    o = __fmul_rn(4.0f / 9.0f, base);
    auto four = [&](float2 e, float bw, float h, float l, float n, float2 &u, float2 &v) {
        const float2 t = __ffma2_rn(__fmul2_rn(dup(h), e), e, dup(bw));
        u = __ffma2_rn(dup(l), e, t);
        v = __ffma2_rn(dup(n), e, t);
    };
    four(make_float2(ux, uy), __fmul_rn(1.0f / 9.0f, base), __fmul_rn(0.5f, rho), __fmul_rn(1.0f / 3.0f, rho),
         __fmul_rn(-1.0f / 3.0f, rho), p[0], p[1]);
    four(make_float2(__fadd_rn(ux, uy), __fsub_rn(uy, ux)), __fmul_rn(1.0f / 36.0f, base), __fmul_rn(0.125f, rho),
         __fmul_rn(1.0f / 12.0f, rho), __fmul_rn(-1.0f / 12.0f, rho), p[2], p[3]);
}

// strip_face for one face: the pairs v of its six crossing distributions (slots 0 1, 2 3, 4 5) and
// the tangential sums.
template <int AX>
__device__ __forceinline__ void face_cell(float2 flux[3], const float2 v[3], float t0, float ta, float tb, const StripInst &m)
{
    t0 = __fmul_rn(0.5f, t0); ta = __fmul_rn(0.5f, ta); tb = __fmul_rn(0.5f, tb);
    const float2 d = sub2(v[1], v[2]), s = __fadd2_rn(v[1], v[2]);          // 5 - 7, 6 - 8 and sums
    const float dn = __fsub_rn(v[0].x, v[0].y), dt_ = __fsub_rn(ta, tb), sn = __fadd_rn(v[0].x, v[0].y), st = __fadd_rn(ta, tb);
    const float w0 = __fadd_rn(__fadd_rn(__fadd_rn(t0, sn), st), __fadd_rn(s.x, s.y));
    const float w1 = __fadd_rn(AX == 0 ? dn : dt_, __fsub_rn(d.x, d.y));
    const float w2 = __fadd_rn(AX == 0 ? dt_ : dn, __fadd_rn(d.x, d.y));
    const float rb = __fadd_rn(1.0f, w0), inv = recip<float>(rb), bg = m.bg[AX].x;
    float o;
    float2 fe[4];
    feq_cell(__fmul_rn(bg, w0), __fmul_rn(bg, rb), __fmul_rn(w1, inv), __fmul_rn(w2, inv), o, fe);
    const float2 n = AX == 0 ? make_float2(fe[0].x, fe[1].x) : make_float2(fe[0].y, fe[1].y);
    const float2 g = dup(m.g[AX].x);
    flux[0] = __ffma2_rn(g, v[0], n);
    flux[1] = __ffma2_rn(g, v[1], fe[2]);
    flux[2] = __ffma2_rn(g, v[2], fe[3]);
}

// strip_boundary for one cell.
template <int D>
__device__ __forceinline__ void wall_cell(float F[NQ], const float out[3], const float fn[NQ], float b0, float rho, float ux,
                                          float uy, const StripInst &m, int side)
{
    const int bk = m.side_kind[side];
    float rb = rho, drb = b0, ubx = 0.0f, uby = 0.0f;
    if (bk == BK_MOVING_WALL) { ubx = m.side_par[side][0]; uby = m.side_par[side][1]; }
    else if (bk == BK_FARFIELD) { rb = m.side_par[side][0]; drb = m.side_drho[side]; ubx = m.side_par[side][1]; uby = m.side_par[side][2]; }
    else if (bk == BK_OUTLET) { ubx = ux; uby = uy; }
    float o;
    float2 pb[4], pn[4];
    feq_cell(drb, rb, ubx, uby, o, pb);
    feq_cell(b0, rho, ux, uy, o, pn);
    auto of = [](const float2 p[4], int a) { return (a - 1) % 2 == 0 ? p[(a - 1) / 2].x : p[(a - 1) / 2].y; };
    const float lp = m.len_dtV[D < 2 ? 0 : 1];
    int k = 0;
#pragma unroll
    for (int q = 0; q < 6; q++) {
        const int a = D < 2 ? XSLOT_A(q) : YSLOT_A(q);
        const int sg = D == 0 ? EX(a) : D == 1 ? -EX(a) : D == 2 ? EY(a) : -EY(a);
        float fb;
        if (sg < 0) fb = __fadd_rn(of(pb, a), __fsub_rn(fn[a], of(pn, a)));
        else fb = __fmul_rn(__fmaf_rn(m.sb, of(pb, a), out[k++]), m.sc);
        F[a] = __fmaf_rn(sg > 0 ? lp : -lp, fb, F[a]);
    }
}

// The block at (x0, y0): reads buffer `par`, writes buffer 1 - par.  EDGE: it has a grid side
// (without a wrap) within its ring.
template <bool EDGE, bool WIDE>
__device__ __forceinline__ void strip_block(StripBlockSmem &S, int par, int x0, int y0)
{
    constexpr int SX = SB::SX, PL = SB::PLANE;
    const StripInst &m = S.m;
    const int nx = m.nx, ny = m.ny, pitch = m.pitch, np = m.npad, tid = threadIdx.x;
    const bool perx = m.periodic_x != 0, pery = m.periodic_y != 0;
    const float *__restrict__ fin = m.f[par];
    const double *__restrict__ Wn = m.W[par];

    // ---- fbar+ of the block, by the threads that update its cells, and of its ring, by the others
    // (positions past a side without a wrap are not staged)
    const int ti = tid & 15, tj = slot_row(tid);
    const bool mine = tid < SB::NT, right_edge = WIDE && tid >= sb_threads<false>();
    float fn[NQ];
    double w0 = 0.0, w1 = 0.0, w2 = 0.0;
    {
        int li = ti + 2, lj = tj + 2;
        if (!mine) {
            // two rows below, two above, then two columns left and right
            const int r = tid - SB::NT, h = 2 * SB::LX, t = r - 2 * h;
            li = r < 2 * h ? r % SB::LX : (t & 3) + ((t & 3) < 2 ? 0 : 16);
            lj = r < h ? r / SB::LX : r < 2 * h ? BATCH_TY + r / SB::LX : 2 + t / 4;
        }
        int c = x0 - 2 + li, j = y0 - 2 + lj;
        bool in = tid < SB::LX * SB::LY;
        if (EDGE && (c < 0 || c >= nx)) {
            in = in && perx;
            c %= nx;
            if (c < 0) c += nx;
        }
        if (EDGE && (j < 0 || j >= ny)) {
            in = in && pery;
            j %= ny;
            if (j < 0) j += ny;
        }
        if (in) {
            const int64_t o = (int64_t)pitch * j + c;
            float e0;
            float2 fe[4];
            w0 = Wn[o]; w1 = Wn[o + np]; w2 = Wn[o + 2 * (int64_t)np];
#pragma unroll
            for (int a = 0; a < NQ; a++) fn[a] = fin[o + (int64_t)np * a];
            const float b0 = d2f_short(w0), rho = __fadd_rn(1.0f, b0), inv = recip<float>(rho), b = m.b.x;
            feq_cell(b0, rho, __fmul_rn(d2f_short(w1), inv), __fmul_rn(d2f_short(w2), inv), e0, fe);
            float *const s = S.f + lj * SX + li;
            s[0] = __fmaf_rn(b, __fsub_rn(e0, fn[0]), fn[0]);
#pragma unroll
            for (int k = 0; k < 4; k++) {
                const float2 f = make_float2(fn[2 * k + 1], fn[2 * k + 2]), v = __ffma2_rn(dup(b), sub2(fe[k], f), f);
                s[(2 * k + 1) * PL] = v.x;
                s[(2 * k + 2) * PL] = v.y;
            }
        }
    }
    __syncthreads();

    // the differences of a staged cell as strip_march forms them: a missing neighbour repeats the
    // cell itself, and the difference is doubled
    struct Near {
        int q, E, W, N, S;           // position, and offsets of its neighbours
        float sx, sy;
    };
    auto near = [&](int li, int lj) {
        Near n;
        n.q = lj * SX + li;
        n.E = 1; n.W = -1; n.N = SX; n.S = -SX;
        n.sx = n.sy = 1.0f;
        if (EDGE) {
            const int c = x0 - 2 + li, j = y0 - 2 + lj;
            if (!perx && c >= nx - 1) { n.E = 0; n.sx = 2.0f; }
            if (!perx && c <= 0) { n.W = 0; n.sx = 2.0f; }
            if (!pery && j >= ny - 1) { n.N = 0; n.sy = 2.0f; }
            if (!pery && j <= 0) { n.S = 0; n.sy = 2.0f; }
        }
        return n;
    };
    auto at = [&](int a, int q) { return S.f[a * PL + q]; };
    auto xd = [&](int a, const Near &n) {
        const float d = __fsub_rn(at(a, n.q + n.E), at(a, n.q + n.W));
        return EDGE ? __fmul_rn(d, n.sx) : d;
    };
    auto yd = [&](int a, const Near &n) {
        const float d = __fsub_rn(at(a, n.q + n.N), at(a, n.q + n.S));
        return EDGE ? __fmul_rn(d, n.sy) : d;
    };
    // velocity a of cell p and velocity b of cell q with their differences, as pairs
    auto val = [&](int a, const Near &p, int b, const Near &q) { return make_float2(at(a, p.q), at(b, q.q)); };
    auto dx = [&](int a, const Near &p, int b, const Near &q) { return make_float2(xd(a, p), xd(b, q)); };
    auto dy = [&](int a, const Near &p, int b, const Near &q) { return make_float2(yd(a, p), yd(b, q)); };
    auto sum = [](float2 v) { return __fadd_rn(v.x, v.y); };

    // ---- faces, by slot as in cart_tile: of constant x left of each cell, of constant y below each cell
    // and above the top row
    auto x_face = [&](int i, int r, int slot) {
        const int c = x0 + i;
        if (y0 + r >= ny || (perx ? c > nx : c <= 0 || c >= nx)) return;
        const Near L = near(i + 1, r + 2), R = near(i + 2, r + 2);
        const float k = m.xo[0].x, d = m.ydt[0].x;
        const float2 xo = make_float2(k, -k), xh = make_float2(STRIP_XH, -STRIP_XH), up = dup(-d), dn = dup(d);
        const float2 t0 = __ffma2_rn(xh, dx(0, L, 0, R), val(0, L, 0, R));
        const float2 t2 = __ffma2_rn(up, dy(2, L, 2, R), __ffma2_rn(xh, dx(2, L, 2, R), val(2, L, 2, R)));
        const float2 t4 = __ffma2_rn(dn, dy(4, L, 4, R), __ffma2_rn(xh, dx(4, L, 4, R), val(4, L, 4, R)));
        const float2 v13 = __ffma2_rn(xo, dx(1, L, 3, R), val(1, L, 3, R));
        const float2 v56 = __ffma2_rn(up, dy(5, L, 6, R), __ffma2_rn(xo, dx(5, L, 6, R), val(5, L, 6, R)));
        const float2 v87 = __ffma2_rn(dn, dy(8, L, 7, R), __ffma2_rn(xo, dx(8, L, 7, R), val(8, L, 7, R)));
        const float2 v[3] = {v13, v56, make_float2(v87.y, v87.x)};
        float2 fl[3];
        face_cell<0>(fl, v, sum(t0), sum(t2), sum(t4), m);
#pragma unroll
        for (int k = 0; k < 3; k++) { S.x[2 * k * SB::NSX + slot] = fl[k].x; S.x[(2 * k + 1) * SB::NSX + slot] = fl[k].y; }
    };
    if (mine) {
        x_face(ti, tj, tid);
    } else if (right_edge) {
        const int r = tid - sb_threads<false>();
        if (r < BATCH_TY) x_face(16, r, 32 * SB::WX + r);
    } else {
        const int u = tid - 32 * SB::WX, i = u & 15, r = slot_row(u), j = y0 + r;
        if (r <= BATCH_TY && x0 + i < nx && (pery ? j <= ny : j > 0 && j < ny)) {
            const Near B = near(i + 2, r + 1), A = near(i + 2, r + 2);        // below, above
            const float k = m.yo[0].x, d = m.xdt[0].x;
            const float2 yo = make_float2(k, -k), yh = make_float2(STRIP_XH, -STRIP_XH);
            const float2 xpm = make_float2(-d, d);                           // velocities with xi_x = 1, -1
            const float2 t0 = __ffma2_rn(yh, dy(0, B, 0, A), val(0, B, 0, A));
            const float2 t1 = __ffma2_rn(yh, dy(1, B, 1, A), __ffma2_rn(dup(-d), dx(1, B, 1, A), val(1, B, 1, A)));
            const float2 t3 = __ffma2_rn(yh, dy(3, B, 3, A), __ffma2_rn(dup(d), dx(3, B, 3, A), val(3, B, 3, A)));
            const float2 v24 = __ffma2_rn(yo, dy(2, B, 4, A), val(2, B, 4, A));
            const float2 v56 = __ffma2_rn(dup(k), dy(5, B, 6, B), __ffma2_rn(xpm, dx(5, B, 6, B), val(5, B, 6, B)));
            const float2 v87 = __ffma2_rn(dup(-k), dy(8, A, 7, A), __ffma2_rn(xpm, dx(8, A, 7, A), val(8, A, 7, A)));
            const float2 v[3] = {v24, v56, make_float2(v87.y, v87.x)};
            float2 fl[3];
            face_cell<1>(fl, v, sum(t0), sum(t1), sum(t3), m);
#pragma unroll
            for (int k = 0; k < 3; k++) { S.y[2 * k * SB::NSY + u] = fl[k].x; S.y[(2 * k + 1) * SB::NSY + u] = fl[k].y; }
        } else if (!WIDE && (u >> 5) == SB::WY - 1 && (u & 16) && i < BATCH_TY) {
            x_face(16, i, 32 * SB::WX + i);
        }
    }
    __syncthreads();

    // ---- cells
    const int c = x0 + ti, j = y0 + tj;
    if (!mine || c >= nx || j >= ny) return;
    const int64_t o = (int64_t)pitch * j + c;
    const int fW = tid, fE = ti < 15 ? tid + 1 : 32 * SB::WX + tj, fS = row_slot(tj, ti), fN = row_slot(tj + 1, ti);
    float F[NQ];
    F[0] = F[2] = F[4] = 0.0f;
    const bool hW = !EDGE || perx || c > 0, hE = !EDGE || perx || c < nx - 1;
    const bool hS = !EDGE || pery || j > 0, hN = !EDGE || pery || j < ny - 1;
    auto minus = [](float f, float fl, int sg) { return sg > 0 ? __fsub_rn(f, fl) : __fadd_rn(f, fl); };
    auto plus = [](float f, float fl, int sg) { return sg > 0 ? __fadd_rn(f, fl) : __fsub_rn(f, fl); };
    const float b0 = d2f_short(w0), m1 = d2f_short(w1), m2 = d2f_short(w2);
    if (!EDGE || (hW && hE)) {
#pragma unroll
        for (int k = 0; k < 6; k++) {
            const float l = S.x[k * SB::NSX + fW], r = S.x[k * SB::NSX + fE];
            F[XSLOT_A(k)] = EX(XSLOT_A(k)) > 0 ? __fsub_rn(r, l) : __fsub_rn(l, r);
        }
    }
    if (EDGE) {
        const Near n = near(ti + 2, tj + 2);
        auto wall = [&](auto dir, int side, const float out[3]) {
            const float rho = __fadd_rn(1.0f, b0), inv = recip<float>(rho);
            wall_cell<decltype(dir)::value>(F, out, fn, b0, rho, __fmul_rn(m1, inv), __fmul_rn(m2, inv), m, side);
        };
        // normal velocity a, and b and d whose other component is along the side
        auto out_x = [&](int a, int b, int d, int s, float k1, float k2) {
            const float xo = m.xo[s].x;
            const float out[3] = {__fmaf_rn(xo, xd(a, n), at(a, n.q)),
                                  __fmaf_rn(k1, yd(b, n), __fmaf_rn(xo, xd(b, n), at(b, n.q))),
                                  __fmaf_rn(k2, yd(d, n), __fmaf_rn(xo, xd(d, n), at(d, n.q)))};
            if (s == 0) wall(std::integral_constant<int, 0>{}, 1, out);
            else wall(std::integral_constant<int, 1>{}, 3, out);
        };
        auto out_y = [&](int a, int b, int d, int s, float k1, float k2) {
            const float yo = m.yo[s].x;
            const float out[3] = {__fmaf_rn(yo, yd(a, n), at(a, n.q)),
                                  __fmaf_rn(yo, yd(b, n), __fmaf_rn(k1, xd(b, n), at(b, n.q))),
                                  __fmaf_rn(yo, yd(d, n), __fmaf_rn(k2, xd(d, n), at(d, n.q)))};
            if (s == 0) wall(std::integral_constant<int, 2>{}, 2, out);
            else wall(std::integral_constant<int, 3>{}, 0, out);
        };
        if (!(hW && hE)) {
#pragma unroll
            for (int k = 0; k < 6; k++)
                F[XSLOT_A(k)] = hW ? minus(0.0f, S.x[k * SB::NSX + fW], EX(XSLOT_A(k))) : 0.0f;
            if (!hW) out_x(3, 6, 7, 1, m.ydt[1].x, m.ydt[0].x);
            if (hE) {
#pragma unroll
                for (int k = 0; k < 6; k++) F[XSLOT_A(k)] = plus(F[XSLOT_A(k)], S.x[k * SB::NSX + fE], EX(XSLOT_A(k)));
            } else out_x(1, 5, 8, 0, m.ydt[1].x, m.ydt[0].x);
        }
        if (!hS) out_y(4, 7, 8, 1, m.xdt[0].x, m.xdt[1].x);
    }
    if (hS) {
#pragma unroll
        for (int k = 0; k < 6; k++) F[YSLOT_A(k)] = minus(F[YSLOT_A(k)], S.y[k * SB::NSY + fS], EY(YSLOT_A(k)));
    }
    if (hN) {
#pragma unroll
        for (int k = 0; k < 6; k++) F[YSLOT_A(k)] = plus(F[YSLOT_A(k)], S.y[k * SB::NSY + fN], EY(YSLOT_A(k)));
    } else if (EDGE) {
        const Near n = near(ti + 2, tj + 2);
        const float yo = m.yo[0].x;
        const float out[3] = {__fmaf_rn(yo, yd(2, n), at(2, n.q)),
                              __fmaf_rn(yo, yd(5, n), __fmaf_rn(m.xdt[1].x, xd(5, n), at(5, n.q))),
                              __fmaf_rn(yo, yd(6, n), __fmaf_rn(m.xdt[0].x, xd(6, n), at(6, n.q)))};
        const float rho = __fadd_rn(1.0f, b0), inv = recip<float>(rho);
        wall_cell<2>(F, out, fn, b0, rho, __fmul_rn(m1, inv), __fmul_rn(m2, inv), m, 2);
    }
    // strip_update for one cell
    const float d57 = __fsub_rn(F[5], F[7]), d68 = __fsub_rn(F[6], F[8]);
    const float s1 = __fadd_rn(__fadd_rn(F[1], F[3]), __fadd_rn(F[5], F[7]));
    const float s2 = __fadd_rn(__fadd_rn(F[2], F[4]), __fadd_rn(F[6], F[8]));
    const float d0 = __fadd_rn(s1, s2), d1 = __fadd_rn(__fsub_rn(F[1], F[3]), __fsub_rn(d57, d68));
    const float d2 = __fadd_rn(__fsub_rn(F[2], F[4]), __fadd_rn(d57, d68));
    const float drho = __fsub_rn(b0, d0), rho = __fadd_rn(1.0f, drho), inv = recip<float>(rho), ri = m.ri.x;
    float e0;
    float2 fe[4];
    feq_cell(drho, rho, __fmul_rn(__fsub_rn(m1, d1), inv), __fmul_rn(__fsub_rn(m2, d2), inv), e0, fe);
    float *const fo = m.f[1 - par] + o;
    fo[0] = __fmaf_rn(ri, __fsub_rn(e0, fn[0]), fn[0]);
#pragma unroll
    for (int k = 0; k < 4; k++) {
        const float2 t = sub2(make_float2(fn[2 * k + 1], fn[2 * k + 2]), make_float2(F[2 * k + 1], F[2 * k + 2]));
        const float2 v = __ffma2_rn(dup(ri), sub2(fe[k], t), t);
        fo[(int64_t)np * (2 * k + 1)] = v.x;
        fo[(int64_t)np * (2 * k + 2)] = v.y;
    }
    double *const Wo = m.W[1 - par] + o;
    Wo[0] = w0 - to_f64<float>(d0);
    Wo[np] = w1 - to_f64<float>(d1);
    Wo[2 * (int64_t)np] = w2 - to_f64<float>(d2);
}

}  // namespace sdugks
