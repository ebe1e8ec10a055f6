// step_strip.cuh -- fused S-DUGKS step on uniform Cartesian grids by marching warps
// (FP32 storage and compute).
//
// The update of cart_tile (step_cart.cuh) on another split of the work: a warp owns a
// strip of 64 columns, two neighbouring columns per lane, and marches upwards through a
// range of rows.  Per row j it holds fbar+ of rows j-1, j and j+1 in registers, takes the
// x neighbours from the next lanes by shuffles, evaluates each face once and finishes row
// j-1 as soon as the face between j-1 and j is known.  f^n and W^n travel one row ahead
// from global to shared memory by asynchronous copies; every lane reads back only what
// it copied itself, so there is no barrier anywhere.
//
// Why: the block form computes fbar+ of a two-cell ring (1.9x the cells of a 16x8
// block), evaluates the block-border faces twice, forms the two-point differences anew
// for every face, and waits at two barriers per block: 1,169 thread instructions per cell.
// Here the ring is four columns in 64 and four rows per range, each difference is formed
// once per cell, both cells of a lane go through the same paired FP32 instructions
// (FFMA2/FMUL2/FADD2), and the faces' equilibria come scaled by the factor they are used with:
// about 415 per cell (1024^2, 16 rows per warp).  Measured (GB300, FP32 cavity, us per step,
// blocks -> strips): 512^2 14.0 -> 11.7, 723^2 23.7 -> 19.3, 1024^2 48.1 -> 31.8, 2048^2
// 180 -> 113 (4.5 TB/s of the state's bytes).
//
// What bounds it now: latency.  Eight warps per SM (226 registers) issue in 45 % of the
// cycles; dependent FP32 pairs and the shared-memory/shuffle queue (which also carries the
// six FP64 additions per row, 16 cycles each on this GPU's two FP64 lanes per SM) are the
// stalls.  Measured without gain: twelve warps per SM at 168 registers (the queue then
// saturates), three rows per loop turn without register moves (the code outgrows the
// instruction cache: 34 % slower), a three-row ring (the copies are then only half a row
// ahead), the flux sums in shared memory (3 % slower).
//
// fbar+ = f + b (feq - f) and f^{n+1} = t + r/(1+r) (feq - t), t = f - flux sum, take the equilibrium unscaled
// and by the same operations: the rounding of feq that f took over then cancels in feq - f.  With the
// equilibria scaled by b and by r/(1+r), each rounded its own way, what they differ by was multiplied by b
// = dt/(2 tau), 10 to 100 on small grids at high Re: the FP32 residual's floor was 1.3 to 2.4 times
// that of the blocks (48^2, Re 1000: 6.0e-7; blocks 3.6e-7, now 3.1e-7), and 4 of 100 served solves no
// longer reached 1e-6.
#pragma once
#include "step_cart.cuh"

namespace sdugks {

constexpr int STRIP_W = 64;        // columns a warp stages (two per lane)
constexpr int STRIP_STEP = 60;     // columns from one strip to the next
constexpr int STRIP_RING = 4;      // rows of f^n, W^n in shared memory: j - 1 .. j + 2
constexpr int STRIP_CTAS = 8;      // warps (one-warp CTAs) per SM
constexpr float STRIP_XH = 0.25f;  // (h / 2) / (2 h): StripInst's xh and yh

// Shared memory of a row: W^n (3 planes of 32 x two cells), then f^n (9 planes).
constexpr int STRIP_WB = 3 * 32 * 16, STRIP_ROW = STRIP_WB + NQ * 32 * 8;
constexpr size_t STRIP_SMEM = (size_t)STRIP_RING * STRIP_ROW;

__device__ __forceinline__ float2 dup(float v) { return make_float2(v, v); }
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return __ffma2_rn(b, make_float2(-1.0f, -1.0f), a); }
__device__ __forceinline__ float2 rcp2(float2 v) { return make_float2(recip<float>(v.x), recip<float>(v.y)); }

// The deviation-form equilibrium (feq9fd) of two cells from s (rho - 1), s rho and u:
// scaled by s, with the weights folded into the shared factors.
__device__ __forceinline__ void feq_pair(float2 b0, float2 rho, float2 ux, float2 uy, float2 out[NQ])
{
    const float2 ss = __ffma2_rn(ux, ux, __fmul2_rn(uy, uy));
    const float2 base = __ffma2_rn(__fmul2_rn(dup(-1.5f), rho), ss, b0);
    out[0] = __fmul2_rn(dup(4.0f / 9.0f), base);
    auto two = [&](float2 e, float2 bw, float2 r45, float2 r3, float2 r3m, float2 &p, float2 &q) {
        const float2 t = __ffma2_rn(__fmul2_rn(r45, e), e, bw);
        p = __ffma2_rn(r3, e, t);
        q = __ffma2_rn(r3m, e, t);
    };
    const float2 b1 = __fmul2_rn(dup(1.0f / 9.0f), base), b5 = __fmul2_rn(dup(1.0f / 36.0f), base);
    const float2 h1 = __fmul2_rn(dup(0.5f), rho), h5 = __fmul2_rn(dup(0.125f), rho);
    const float2 l1 = __fmul2_rn(dup(1.0f / 3.0f), rho), l5 = __fmul2_rn(dup(1.0f / 12.0f), rho);
    const float2 n1 = __fmul2_rn(dup(-1.0f / 3.0f), rho), n5 = __fmul2_rn(dup(-1.0f / 12.0f), rho);
    two(ux, b1, h1, l1, n1, out[1], out[3]);
    two(uy, b1, h1, l1, n1, out[2], out[4]);
    two(__fadd2_rn(ux, uy), b5, h5, l5, n5, out[5], out[7]);
    two(sub2(uy, ux), b5, h5, l5, n5, out[6], out[8]);
}

// d2f_fields in four integer instructions: magnitudes below the binary32 normal range
// become some magnitude below it (d2f_fields: zero); zero stays zero.
__device__ __forceinline__ float d2f_short(double d)
{
    const int hi = __double2hiint(d);
    const int t = max((hi & 0x7fffffff) - 0x38000000, 0);
    return __uint_as_float(__funnelshift_l((unsigned)__double2loint(d), (unsigned)t, 3) | ((unsigned)hi & 0x80000000u));
}
__device__ __forceinline__ float2 d2f2(double2 d) { return make_float2(d2f_short(d.x), d2f_short(d.y)); }

// Conversions of the three flux sums of two cells to FP64 (f2d_fields of each, but for
// the sign of zero): the field arithmetic of normal numbers, and the full rules when any
// of the six is zero, subnormal or not finite.
__device__ __forceinline__ double f2d_normal(float f)
{
    const int u = __float_as_int(f);
    return __hiloint2double(((u >> 3) & (int)0x8fffffff) + 0x38000000, u << 29);
}
__device__ __forceinline__ void f2d_six(const float2 d[3], double2 out[3])
{
    constexpr float MIN = 1.17549435e-38f;
    const float2 s = __fadd2_rn(__fadd2_rn(d[0], d[1]), d[2]);      // not finite if one of them is not
    const bool normal = fabsf(d[0].x) >= MIN && fabsf(d[0].y) >= MIN && fabsf(d[1].x) >= MIN && fabsf(d[1].y) >= MIN &&
                        fabsf(d[2].x) >= MIN && fabsf(d[2].y) >= MIN && fabsf(s.x) < INFINITY && fabsf(s.y) < INFINITY;
    if (normal) {
#pragma unroll
        for (int k = 0; k < 3; k++) out[k] = make_double2(f2d_normal(d[k].x), f2d_normal(d[k].y));
    } else {
        auto one = [](float f) {
            if (fabsf(f) < MIN) return 0.0;
            return fabsf(f) < INFINITY ? f2d_normal(f)
                                       : __hiloint2double(f != f ? 0x7ff80000 : (__float_as_int(f) | 0x7ff00000), 0);
        };
#pragma unroll
        for (int k = 0; k < 3; k++) out[k] = make_double2(one(d[k].x), one(d[k].y));
    }
}

template <int B> __device__ __forceinline__ void strip_copy(uint32_t dst, const void *src)
{
    if constexpr (B == 16) asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
    else asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(dst), "l"(src) : "memory");
}

// Two cells' values of every plane (n elements apart), where `on`.
__device__ __forceinline__ void strip_store(double *p, int n, const double2 v[3], bool on)
{
    asm volatile("{\n\t.reg .pred q;\n\t.reg .b64 r;\n\tsetp.ne.s32 q, %2, 0;\n\t"
                 "@q st.global.v2.f64 [%0], {%3, %4};\n\t"
                 "mad.wide.s32 r, %1, 8, %0;\n\t@q st.global.v2.f64 [r], {%5, %6};\n\t"
                 "mad.wide.s32 r, %1, 16, %0;\n\t@q st.global.v2.f64 [r], {%7, %8};\n\t}"
                 ::"l"(p), "r"(n), "r"((int)on), "d"(v[0].x), "d"(v[0].y), "d"(v[1].x), "d"(v[1].y), "d"(v[2].x),
                 "d"(v[2].y) : "memory");
}
__device__ __forceinline__ void strip_store(float *p, int n, const float2 v[NQ], bool on)
{
#define SDUGKS_ST(k, x, y) "mad.wide.s32 r, %1, " #k ", %0;\n\t@q st.global.v2.f32 [r], {%" #x ", %" #y "};\n\t"
    asm volatile("{\n\t.reg .pred q;\n\t.reg .b64 r;\n\tsetp.ne.s32 q, %2, 0;\n\t"
                 "@q st.global.v2.f32 [%0], {%3, %4};\n\t"
                 SDUGKS_ST(4, 5, 6) SDUGKS_ST(8, 7, 8) SDUGKS_ST(12, 9, 10) SDUGKS_ST(16, 11, 12) SDUGKS_ST(20, 13, 14)
                 SDUGKS_ST(24, 15, 16) SDUGKS_ST(28, 17, 18) SDUGKS_ST(32, 19, 20) "}"
                 ::"l"(p), "r"(n), "r"((int)on), "f"(v[0].x), "f"(v[0].y), "f"(v[1].x), "f"(v[1].y), "f"(v[2].x),
                 "f"(v[2].y), "f"(v[3].x), "f"(v[3].y), "f"(v[4].x), "f"(v[4].y), "f"(v[5].x), "f"(v[5].y), "f"(v[6].x),
                 "f"(v[6].y), "f"(v[7].x), "f"(v[7].y), "f"(v[8].x), "f"(v[8].y) : "memory");
#undef SDUGKS_ST
}

// Two cells' values of every plane at p, of the cells that are `on`; ODD: where one of the
// two alone can be.
template <class T, int N, class P>
__device__ __forceinline__ void strip_put_n(P *p, int np, const T v[N], bool on0, bool on1, bool odd)
{
    strip_store(p, np, v, on0 && on1);
    if (odd && on0 != on1) {
#pragma unroll
        for (int k = 0; k < N; k++) p[(int64_t)np * k + (on0 ? 0 : 1)] = on0 ? v[k].x : v[k].y;
    }
}
__device__ __forceinline__ void strip_put(double *p, int np, const double2 v[3], bool on0, bool on1, bool odd)
{
    strip_put_n<double2, 3>(p, np, v, on0, on1, odd);
}
__device__ __forceinline__ void strip_put(float *p, int np, const float2 v[NQ], bool on0, bool on1, bool odd)
{
    strip_put_n<float2, NQ>(p, np, v, on0, on1, odd);
}

// W^{n+1} and f^{n+1} of two cells from their flux sums F; W^n and f^n by W(k), f(a), the
// results to put_W and put_f.
template <class GetW, class GetF, class PutW, class PutF>
__device__ __forceinline__ void strip_update(const float2 F[NQ], const StripInst &m, GetW &&W, GetF &&f, PutW &&put_W,
                                             PutF &&put_f)
{
    const float2 sm1 = __fadd2_rn(__fadd2_rn(F[1], F[3]), __fadd2_rn(F[5], F[7]));
    const float2 sm2 = __fadd2_rn(__fadd2_rn(F[2], F[4]), __fadd2_rn(F[6], F[8]));
    const float2 d57 = sub2(F[5], F[7]), d68 = sub2(F[6], F[8]);
    float2 d[3] = {__fadd2_rn(sm1, sm2), __fadd2_rn(sub2(F[1], F[3]), sub2(d57, d68)),
                   __fadd2_rn(sub2(F[2], F[4]), __fadd2_rn(d57, d68))};
    float2 b0, m1, m2;
    {
        double2 w[3], dd[3];
        f2d_six(d, dd);
#pragma unroll
        for (int k = 0; k < 3; k++) w[k] = W(k);
        b0 = d2f2(w[0]); m1 = d2f2(w[1]); m2 = d2f2(w[2]);
#pragma unroll
        for (int k = 0; k < 3; k++) w[k] = make_double2(w[k].x - dd[k].x, w[k].y - dd[k].y);
        put_W(w);
    }
    const float2 drho1 = sub2(b0, d[0]), rho1 = __fadd2_rn(dup(1.0f), drho1), inv = rcp2(rho1);
    const float2 ux1 = __fmul2_rn(sub2(m1, d[1]), inv), uy1 = __fmul2_rn(sub2(m2, d[2]), inv);
    float2 fe[NQ], v[NQ];
    feq_pair(drho1, rho1, ux1, uy1, fe);
#pragma unroll
    for (int a = 0; a < NQ; a++) {
        const float2 fn = f(a), t = a == 0 ? fn : sub2(fn, F[a]);
        v[a] = __ffma2_rn(m.ri, sub2(fe[a], t), t);
    }
    put_f(v);
}

// Interface moments of the pair of faces, then their six fluxes times dt / V, from the
// six crossing distributions v[6] (slot order XSLOT_A / YSLOT_A) and the sums of the three
// tangential ones over both sides: AX 0: (0, 2, 4), AX 1: (0, 1, 3).  The fluxes carry no
// sign: xi . n_+ is +1 or -1 times them.
template <int AX>
__device__ __forceinline__ void strip_face(float2 flux[6], const float2 v[6], float2 t0, float2 ta, float2 tb,
                                           const StripInst &m)
{
    const float2 half = dup(0.5f);
    t0 = __fmul2_rn(half, t0); ta = __fmul2_rn(half, ta); tb = __fmul2_rn(half, tb);
    // AX 0: slots 1 3 5 6 7 8; AX 1: slots 2 4 5 6 7 8
    const float2 d57 = sub2(v[2], v[4]), d68 = sub2(v[3], v[5]);
    const float2 s57 = __fadd2_rn(v[2], v[4]), s68 = __fadd2_rn(v[3], v[5]);
    const float2 dn = sub2(v[0], v[1]), dt_ = sub2(ta, tb), sn = __fadd2_rn(v[0], v[1]), st = __fadd2_rn(ta, tb);
    const float2 w0 = __fadd2_rn(__fadd2_rn(__fadd2_rn(t0, sn), st), __fadd2_rn(s57, s68));
    const float2 w1 = __fadd2_rn(AX == 0 ? dn : dt_, sub2(d57, d68));
    const float2 w2 = __fadd2_rn(AX == 0 ? dt_ : dn, __fadd2_rn(d57, d68));
    const float2 rb = __fadd2_rn(dup(1.0f), w0), inv = rcp2(rb);
    float2 fe[NQ];
    feq_pair(__fmul2_rn(m.bg[AX], w0), __fmul2_rn(m.bg[AX], rb), __fmul2_rn(w1, inv), __fmul2_rn(w2, inv), fe);
#pragma unroll
    for (int q = 0; q < 6; q++) flux[q] = __ffma2_rn(m.g[AX], v[q], fe[AX == 0 ? XSLOT_A(q) : YSLOT_A(q)]);
}

// Boundary face of two cells (on0, on1: of which) in direction D (0 +x, 1 -x, 2 +y,
// 3 -y) on grid side `side`: adds the outward flux, times dt / V, of every crossing
// velocity to F (Sec. III rules, as cart_boundary_face).  out: the reconstructions of the
// three leaving velocities, in slot order; fn and (rho - 1, rho, u): the state of the cells.
template <int D>
__device__ __forceinline__ void strip_boundary(float2 F[NQ], const float2 out[3], const float2 fn[NQ], float2 b0,
                                               float2 rho, float2 ux, float2 uy, const StripInst &m, int side, bool on0,
                                               bool on1)
{
    const int bk = m.side_kind[side];
    float2 rb = rho, drb = b0, ubx = dup(0.0f), uby = dup(0.0f);
    if (bk == BK_MOVING_WALL) { ubx = dup(m.side_par[side][0]); uby = dup(m.side_par[side][1]); }
    else if (bk == BK_FARFIELD) {
        rb = dup(m.side_par[side][0]); drb = dup(m.side_drho[side]);
        ubx = dup(m.side_par[side][1]); uby = dup(m.side_par[side][2]);
    } else if (bk == BK_OUTLET) { ubx = ux; uby = uy; }
    float2 feqb[NQ], feqn[NQ];
    feq_pair(drb, rb, ubx, uby, feqb);
    feq_pair(b0, rho, ux, uy, feqn);
    const float2 bb = dup(m.sb), cc = dup(m.sc), lp = dup(m.len_dtV[D < 2 ? 0 : 1]), lm = dup(-m.len_dtV[D < 2 ? 0 : 1]);
    int o = 0;
#pragma unroll
    for (int q = 0; q < 6; q++) {
        const int a = D < 2 ? XSLOT_A(q) : YSLOT_A(q);
        const int sg = D == 0 ? EX(a) : D == 1 ? -EX(a) : D == 2 ? EY(a) : -EY(a);
        float2 fb;
        if (sg < 0) fb = __fadd2_rn(feqb[a], sub2(fn[a], feqn[a]));        // non-equilibrium extrapolation
        else fb = __fmul2_rn(__ffma2_rn(bb, feqb[a], out[o++]), cc);
        const float2 s = __ffma2_rn(sg > 0 ? lp : lm, fb, F[a]);
        if (on0) F[a].x = s.x;
        if (on1) F[a].y = s.y;
    }
}

// rho - 1, rho and u of two cells from W^n
__device__ __forceinline__ void strip_state(double2 w0, double2 w1, double2 w2, float2 &b0, float2 &rho, float2 &ux, float2 &uy)
{
    b0 = d2f2(w0);
    rho = __fadd2_rn(dup(1.0f), b0);
    const float2 inv = rcp2(rho);
    ux = __fmul2_rn(d2f2(w1), inv);
    uy = __fmul2_rn(d2f2(w2), inv);
}

// F plus or minus the unsigned flux of a velocity with the sign sg.
__device__ __forceinline__ float2 strip_minus(float2 F, float2 fl, int sg) { return sg > 0 ? sub2(F, fl) : __fadd2_rn(F, fl); }
__device__ __forceinline__ float2 strip_plus(float2 F, float2 fl, int sg) { return sg > 0 ? __fadd2_rn(F, fl) : sub2(F, fl); }

// One warp: rows [y0, y1) of the strip whose first staged column is xb; reads buffer
// `par`, writes buffer 1 - par.  sm: the warp's shared memory.  EDGE: the strip meets
// a grid side in x (a wall or a wrap) or ends past the grid; other strips update lanes
// 1 .. 30 and take every neighbour for granted.
template <bool EDGE>
__device__ __forceinline__ void strip_march(const StripInst &m, int par, int xb, int y0, int y1, unsigned char *sm)
{
    const int lane = threadIdx.x;
    const int nx = m.nx, ny = m.ny, pitch = m.pitch;
    const bool perx = EDGE && m.periodic_x != 0, pery = m.periodic_y != 0;
    const int np = m.npad;
    // columns c0 and c0 + 1; on a periodic grid (even nx) a pair wraps as a whole, past
    // the sides of another the last pair is staged again and never used
    const int c0 = xb + 2 * lane;
    int cm = c0;
    if (EDGE) {
        if (perx) { cm %= nx; if (cm < 0) cm += nx; }
        else if (cm >= nx) cm = (nx - 1) & ~1;
    }
    // neighbours that exist, and cells that this lane updates
    const bool hW0 = !EDGE || perx || c0 > 0, hE0 = !EDGE || perx || c0 < nx - 1, hE1 = !EDGE || perx || c0 + 1 < nx - 1;
    const bool in = EDGE ? ((lane > 0 || (!perx && xb == 0)) && (lane < 31 || (!perx && c0 + 2 >= nx))) : (lane > 0 && lane < 31);
    const bool up0 = in && (!EDGE || (c0 >= 0 && c0 < nx)), up1 = in && (!EDGE || (c0 + 1 >= 0 && c0 + 1 < nx));
    const float *__restrict__ fin = m.f[par] + cm;
    float *__restrict__ fout = m.f[1 - par] + cm;
    const double *__restrict__ Wn = m.W[par] + cm;
    double *__restrict__ Wout = m.W[1 - par] + cm;
    const uint32_t rs = (uint32_t)__cvta_generic_to_shared(sm) + lane * 16;
    const unsigned char *const lw = sm + lane * 16, *const lf = sm + STRIP_WB + lane * 8;

    auto fetch = [&](int row, int slot) {
        const int64_t o = (int64_t)pitch * row;
        const uint32_t d = rs + (uint32_t)(slot * STRIP_ROW), df = d + STRIP_WB - lane * 8;
#pragma unroll
        for (int k = 0; k < 3; k++) strip_copy<16>(d + k * 512, Wn + o + (int64_t)np * k);
#pragma unroll
        for (int a = 0; a < NQ; a++) strip_copy<8>(df + a * 256, fin + o + (int64_t)np * a);
    };
    auto arrived = [] { asm volatile("cp.async.wait_group 1;" ::: "memory"); };      // all but the last row fetched
    auto row_W = [&](int slot, int k) { return *reinterpret_cast<const double2 *>(lw + slot * STRIP_ROW + k * 512); };
    auto row_f = [&](int slot, int a) { return *reinterpret_cast<const float2 *>(lf + slot * STRIP_ROW + a * 256); };
    // rho - 1, rho and u of a row that has arrived
    auto state = [&](int slot, float2 &b0, float2 &rho, float2 &ux, float2 &uy) {
        strip_state(row_W(slot, 0), row_W(slot, 1), row_W(slot, 2), b0, rho, ux, uy);
    };
    // fbar+ of a row that has arrived
    auto stage = [&](int slot, float2 out[NQ]) {
        float2 b0, rho, ux, uy;
        state(slot, b0, rho, ux, uy);
        float2 fe[NQ];
        feq_pair(b0, rho, ux, uy, fe);
#pragma unroll
        for (int a = 0; a < NQ; a++) {
            const float2 f = row_f(slot, a);
            out[a] = __ffma2_rn(m.b, sub2(fe[a], f), f);
        }
    };

    // next to a wall the one-sided difference takes the factor 1/h in the place of 1/(2h):
    // the difference is doubled (exactly), so that every coefficient is the solver's
    const float2 sx = EDGE ? make_float2(hW0 && hE0 ? 1.0f : 2.0f, hE1 ? 1.0f : 2.0f) : dup(1.0f);

    // W^{n+1} and f^{n+1} of the row in `slot` (at row `row` of the grid) from its flux sums
    auto update = [&](int slot, int row, const float2 F[NQ]) {
        const int64_t o = (int64_t)pitch * row;
        strip_update(F, m, [&](int k) { return row_W(slot, k); }, [&](int a) { return row_f(slot, a); },
                     [&](const double2 w[3]) { strip_put(Wout + o, np, w, up0, up1, EDGE); },
                     [&](const float2 v[NQ]) { strip_put(fout + o, np, v, up0, up1, EDGE); });
    };
    // a boundary face of the row in `slot` in direction D
    auto boundary = [&](auto dir, int slot, int side, float2 F[NQ], const float2 out[3], bool on0, bool on1) {
        constexpr int D = decltype(dir)::value;
        float2 b0, rho, ux, uy, fn[NQ];
        state(slot, b0, rho, ux, uy);
#pragma unroll
        for (int a = 1; a < NQ; a++) fn[a] = row_f(slot, a);
        strip_boundary<D>(F, out, fn, b0, rho, ux, uy, m, side, on0, on1);
    };

    const int js = (y0 == 0 && !pery) ? 0 : y0 - 1, je = (y1 == ny && !pery) ? ny - 1 : y1;   // rows processed
    const bool below = pery || js > 0;
    int fr = js - 1;                              // the next row to fetch
    if (pery && fr < 0) { fr += ny; if (fr < 0) fr += ny; }
    auto fetch_next = [&](int slot) {
        if (fr >= 0 && fr < ny) fetch(fr, slot);
        asm volatile("cp.async.commit_group;" ::: "memory");
        fr++;
        if (pery && fr >= ny) fr -= ny;
    };
    fetch_next(0);
    fetch_next(1);
    fetch_next(2);
    // fbar+ of rows j - 1, j, j + 1; through the upper face of row j - 1: velocities 2 5 6
    // and the tangential 0 1 3
    float2 X[NQ], Y[NQ], Z[NQ], Nout[6];
    arrived();
    stage(1, Y);
    if (below) stage(0, X);
    else {
#pragma unroll
        for (int a = 0; a < NQ; a++) X[a] = Y[a];
    }
#pragma unroll
    for (int q = 0; q < 6; q++) Nout[q] = dup(0.0f);

    float2 F[NQ];
#pragma unroll
    for (int a = 0; a < NQ; a++) F[a] = dup(0.0f);
    int j = js;
    // one row; s0 .. s3: the slots of rows j - 1 .. j + 2.  A leaves as scratch.
    auto one_row = [&](float2 (&A)[NQ], float2 (&B)[NQ], float2 (&C)[NQ], int s0, int s1, int s2, int s3) {
        const bool hS = pery || j > 0, hN = pery || j < ny - 1;
        if (j < je) fetch_next(s3);
        else asm volatile("cp.async.commit_group;" ::: "memory");
        arrived();
        if (hN) stage(s2, C);
        else {
#pragma unroll
            for (int a = 0; a < NQ; a++) C[a] = B[a];
        }
        // two-point differences (a missing neighbour repeats the cell itself): A becomes
        // the y difference, xdiff is the x difference
#pragma unroll
        for (int a = 0; a < NQ; a++) A[a] = sub2(C[a], A[a]);
        if (!(hS && hN)) {
#pragma unroll
            for (int a = 0; a < NQ; a++) A[a] = __fadd2_rn(A[a], A[a]);
        }
        auto xdiff = [&](int a) {
            float l = __shfl_up_sync(0xffffffffu, B[a].y, 1), r = __shfl_down_sync(0xffffffffu, B[a].x, 1);
            float e0 = B[a].y;
            if (EDGE) {
                if (!hW0) l = B[a].x;
                if (!hE0) e0 = B[a].x;
                if (!hE1) r = B[a].y;
            }
            const float2 d = make_float2(e0 - l, r - B[a].x);
            return EDGE ? __fmul2_rn(d, sx) : d;
        };
        // tangential velocities of the y faces, up to the y term
        const float2 X1 = xdiff(1), X3 = xdiff(3), X7 = xdiff(7), X8 = xdiff(8);
        const float2 T1 = __ffma2_rn(m.xdt[1], X1, B[1]), T3 = __ffma2_rn(m.xdt[0], X3, B[3]);
        float2 yf[6];
        if (j >= y0) {
            float2 v[6];
            // from row j, through its lower face: velocities 4 7 8 (slots 1 4 5)
            v[1] = __ffma2_rn(m.yo[1], A[4], B[4]);
            v[4] = __ffma2_rn(m.yo[1], A[7], __ffma2_rn(m.xdt[0], X7, B[7]));
            v[5] = __ffma2_rn(m.yo[1], A[8], __ffma2_rn(m.xdt[1], X8, B[8]));
            if (hS) {
                const float2 t0 = __fadd2_rn(Nout[3], __ffma2_rn(m.yh[1], A[0], B[0]));
                const float2 t1 = __fadd2_rn(Nout[4], __ffma2_rn(m.yh[1], A[1], T1));
                const float2 t3 = __fadd2_rn(Nout[5], __ffma2_rn(m.yh[1], A[3], T3));
                v[0] = Nout[0]; v[2] = Nout[1]; v[3] = Nout[2];
                strip_face<1>(yf, v, t0, t1, t3, m);
                if (j > y0) {
#pragma unroll
                    for (int q = 0; q < 6; q++) F[YSLOT_A(q)] = strip_plus(F[YSLOT_A(q)], yf[q], EY(YSLOT_A(q)));
                    update(s0, j > 0 ? j - 1 : ny - 1, F);
                }
            } else {
                yf[0] = v[1]; yf[1] = v[4]; yf[2] = v[5];      // for the wall below row 0
            }
        }
        if (j < y1) {
            const float2 X5 = xdiff(5), X6 = xdiff(6);
            if (j >= y0) {
                // faces of constant x: from the left cell 1 5 8 and tangential 0 2 4 (E), from the right 3 6 7
                // the left faces of the two cells: left values (lane - 1's second cell, own first cell)
                auto left = [](float2 e) { return make_float2(__shfl_up_sync(0xffffffffu, e.y, 1), e.x); };
                auto both = [&](int a) {            // either side of a tangential velocity
                    const float2 D = xdiff(a);
                    float2 e = __ffma2_rn(m.xh[0], D, B[a]), w = __ffma2_rn(m.xh[1], D, B[a]);
                    if (a == 2) { e = __ffma2_rn(m.ydt[1], A[2], e); w = __ffma2_rn(m.ydt[1], A[2], w); }
                    if (a == 4) { e = __ffma2_rn(m.ydt[0], A[4], e); w = __ffma2_rn(m.ydt[0], A[4], w); }
                    return __fadd2_rn(left(e), w);
                };
                const float2 t0 = both(0), t2 = both(2), t4 = both(4);
                const float2 E1 = __ffma2_rn(m.xo[0], X1, B[1]), W3 = __ffma2_rn(m.xo[1], X3, B[3]);
                const float2 E5 = __ffma2_rn(m.ydt[1], A[5], __ffma2_rn(m.xo[0], X5, B[5]));
                const float2 W6 = __ffma2_rn(m.ydt[1], A[6], __ffma2_rn(m.xo[1], X6, B[6]));
                const float2 W7 = __ffma2_rn(m.ydt[0], A[7], __ffma2_rn(m.xo[1], X7, B[7]));
                const float2 E8 = __ffma2_rn(m.ydt[0], A[8], __ffma2_rn(m.xo[0], X8, B[8]));
                const float2 v[6] = {left(E1), W3, left(E5), W6, W7, left(E8)};
                float2 xf[6];
                strip_face<0>(xf, v, t0, t2, t4, m);
                if (EDGE && !perx) {
                    // -x, then +x; boundary faces in the place of interior ones
                    float2 fl[6];
#pragma unroll
                    for (int q = 0; q < 6; q++) {
                        const float2 n = strip_minus(dup(0.0f), xf[q], EX(XSLOT_A(q)));
                        fl[q] = make_float2(xf[q].y, __shfl_down_sync(0xffffffffu, xf[q].x, 1));
                        F[XSLOT_A(q)] = make_float2(hW0 ? n.x : 0.0f, n.y);
                    }
                    F[2] = F[4] = dup(0.0f);
                    if (!hW0 && up0) {
                        const float2 out[3] = {W3, W6, W7};
                        boundary(std::integral_constant<int, 1>{}, s1, 3, F, out, true, false);
                    }
#pragma unroll
                    for (int q = 0; q < 6; q++) {
                        const float2 p = strip_plus(F[XSLOT_A(q)], fl[q], EX(XSLOT_A(q)));
                        if (hE0) F[XSLOT_A(q)].x = p.x;
                        if (hE1) F[XSLOT_A(q)].y = p.y;
                    }
                    if ((!hE0 && up0) || (!hE1 && up1)) {
                        const float2 out[3] = {E1, E5, E8};
                        boundary(std::integral_constant<int, 0>{}, s1, 1, F, out, !hE0, !hE1 && hE0);
                    }
                } else {
#pragma unroll
                    for (int q = 0; q < 6; q++) {
                        const float r = __shfl_down_sync(0xffffffffu, xf[q].x, 1);
                        F[XSLOT_A(q)] = EX(XSLOT_A(q)) > 0 ? make_float2(xf[q].y - xf[q].x, r - xf[q].y)
                                                                    : make_float2(xf[q].x - xf[q].y, xf[q].y - r);
                    }
                    F[2] = F[4] = dup(0.0f);
                }
                if (hS) {
#pragma unroll
                    for (int q = 0; q < 6; q++) F[YSLOT_A(q)] = strip_minus(F[YSLOT_A(q)], yf[q], EY(YSLOT_A(q)));
                } else {
                    boundary(std::integral_constant<int, 3>{}, s1, 0, F, yf, true, true);
                }
            }
            // through the upper face of row j: 2 5 6 and the tangential 0 1 3
            Nout[0] = __ffma2_rn(m.yo[0], A[2], B[2]);
            Nout[1] = __ffma2_rn(m.yo[0], A[5], __ffma2_rn(m.xdt[1], X5, B[5]));
            Nout[2] = __ffma2_rn(m.yo[0], A[6], __ffma2_rn(m.xdt[0], X6, B[6]));
            Nout[3] = __ffma2_rn(m.yh[0], A[0], B[0]);
            Nout[4] = __ffma2_rn(m.yh[0], A[1], T1);
            Nout[5] = __ffma2_rn(m.yh[0], A[3], T3);
        }
    };
    // the wall above the last row, in slot s
    auto top = [&](int s) {
        boundary(std::integral_constant<int, 2>{}, s, 2, F, Nout, true, true);
        update(s, ny - 1, F);
    };
    int s0 = 0, last;
#pragma unroll 1
    for (;;) {
        last = (s0 + 1) & 3;
        one_row(X, Y, Z, s0, last, (s0 + 2) & 3, (s0 + 3) & 3);
        if (j++ == je) break;
        s0 = last;
#pragma unroll
        for (int a = 0; a < NQ; a++) { X[a] = Y[a]; Y[a] = Z[a]; }
    }
    if (y1 == ny && !pery) top(last);
}

// Whether the strip from column xb meets a side in x or ends past the grid.
__device__ __forceinline__ bool strip_is_edge(const StripInst &m, int xb)
{
    return m.periodic_x ? (xb < 0 || xb + STRIP_W > m.nx) : (xb == 0 || xb + STRIP_W >= m.nx);
}

// Strip k, rows [seg rows, (seg + 1) rows) of a grid.
__device__ __forceinline__ void strip_item(const StripInst &m, int par, int k, int seg, int rows, unsigned char *sm)
{
    const int xb = STRIP_STEP * k - (m.periodic_x ? 2 : 0);
    const int y0 = seg * rows, y1 = y0 + rows < m.ny ? y0 + rows : m.ny;
    if (strip_is_edge(m, xb)) strip_march<true>(m, par, xb, y0, y1, sm);
    else strip_march<false>(m, par, xb, y0, y1, sm);
}

}  // namespace sdugks
