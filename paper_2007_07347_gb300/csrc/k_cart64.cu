// k_cart64.cu -- fused S-DUGKS step on uniform Cartesian grids in FP64.
//
// The update of cart_tile (step_cart.cuh) in three phases per block of BX x BY cells:
// fbar+ of the block and its two-cell ring into shared memory, every face once, every
// cell once.
//
// What bounds it: the FP64 pipe.  This GPU has two FP64 lanes per SM, so an FP64 warp
// instruction holds its SM's pipe for 16 cycles, and a step costs the sum over the blocks
// of an SM.  The form therefore spends as few FP64 instructions as it can: products are
// contracted, the three divisions of a state become one Newton reciprocal, the division by
// 1 + r a product, the faces' equilibria come scaled by the factor they are used with
// (weights, dt/V, face length), the two sides of a tangential velocity are averaged before they are
// extrapolated, and beside a wall the missing neighbour is staged as the linear
// extrapolation 2 f_0 - f_1, which makes the one-sided difference a central one and every
// face of a block the same code.  About 400 FP64 warp instructions per 32 cells of a 16x14
// block, where the earlier form took about 800 (256^2: 56 us a step, where it took 129).
//
// fbar+ = f + b (feq - f) and f^{n+1} = t + r/(1+r) (feq - t), t = f less the flux sum, take the equilibrium
// unscaled and by the same operations: the rounding of feq that f took over then cancels.  Scaled by b and by
// r/(1+r) (54 us a step), what the two differ by was multiplied by b = dt/(2 tau): u of 256^2 at Re 5000 was
// off by 2.5e-14 (the earlier form 1.7e-14, now 1.5e-14), of 48^2 at Re 4000 by 1.6e-13 (1.3e-13, 0.96e-13).
//
// Block shapes: 16x14 where that fills the SMs, 8x8 and 4x4 for smaller grids, whose few
// blocks would leave most SMs' pipes idle (a 4 x 64 channel: 16 blocks of 4x4 in the place of
// 4 of 16x16, of whose columns 12 were padding).  The shape with the fewest FP64 instructions
// on the fullest SM is taken.
#include "step_cart.cuh"

namespace sdugks {
namespace {

// Coefficients (host-computed); reconstruction offsets times 1 / (2 h).
struct Cart64K {
    double b, ri, dtV, rdtV;           // ri = r / (1 + r), rdtV = 1 / dtV
    double g[2], bg[2];                // faces of constant x, y: c l dt/V, b c l dt/V
    double lv[2], c;                   // l dt/V; c
    double xdt, xh, xo, ydt, yh, yo;   // dt, h/2, h/2 - dt along x and y, times 1/(2 h)
};

// 1/x by Newton's iteration y <- y + y (1 - x y) from the hardware's approximate
// reciprocal (relative error about 2^-20, so 2^-40 and then rounding after two iterations).
__device__ __forceinline__ double recip64(double x)
{
    double y;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    y = fma(y, fma(-x, y, 1.0), y);
    return fma(y, fma(-x, y, 1.0), y);
}

// s feq(rho, u) from s rho and u; NEED0: with the rest velocity's.
template <bool NEED0> __device__ __forceinline__ void feq64(double rs, double ux, double uy, double out[NQ])
{
    const double uu = fma(ux, ux, uy * uy), base = fma(-1.5 * uu, rs, rs);
    const double b1 = base * (1.0 / 9.0), b5 = base * (1.0 / 36.0), h1 = 0.5 * rs, h5 = 0.125 * rs;
    const double l1 = rs * (1.0 / 3.0), l5 = rs * (1.0 / 12.0);
    if (NEED0) out[0] = base * (4.0 / 9.0);
    auto two = [](double e, double bw, double h, double l, double &p, double &q) {
        const double t = fma(h * e, e, bw);
        p = fma(l, e, t);
        q = fma(-l, e, t);
    };
    two(ux, b1, h1, l1, out[1], out[3]);
    two(uy, b1, h1, l1, out[2], out[4]);
    two(ux + uy, b5, h5, l5, out[5], out[7]);
    two(uy - ux, b5, h5, l5, out[6], out[8]);
}

__device__ __forceinline__ void moments64(const double f[NQ], double &m0, double &m1, double &m2)
{
    const double d57 = f[5] - f[7], d68 = f[6] - f[8];
    m0 = f[0] + (f[1] + f[3]) + (f[2] + f[4]) + ((f[5] + f[7]) + (f[6] + f[8]));
    m1 = (f[1] - f[3]) + (d57 - d68);
    m2 = (f[2] - f[4]) + (d57 + d68);
}

template <int BX, int BY> struct Shape64 {
    static constexpr int LX = BX + 4, LY = BY + 4, LP = LX * LY;
    static constexpr int NXF = (BX + 1) * BY, NYF = BX * (BY + 1);
    static constexpr int XF = (NXF + 31) / 32 * 32, YF = (NYF + 31) / 32 * 32;
    static constexpr int NT = BX >= 16 ? 256 : (BX >= 8 ? 192 : 64);
    static constexpr int CTAS = BX >= 16 ? 2 : (BX >= 8 ? 4 : 8);
    static constexpr size_t SMEM = sizeof(double) * (size_t)(NQ * LP + 6 * (NXF + NYF));
    // FP64 warp instructions of a block (staging 53, face 94, cell 94): the cost model
    static constexpr int COST = (LP + 31) / 32 * 53 + (XF + YF) / 32 * 94 + (BX * BY + 31) / 32 * 94;
    static_assert(BX * BY <= NT, "one cell per thread");
};

// Face fluxes, times dt/V and unsigned, from the staged fbar+ f at the lower/left cell l
// (the other side is at l + S); S, T: staged strides along and across the axis.
template <int AX, int LP, int S, int T>
__device__ __forceinline__ void face64(double flux[6], const double *f, int l, const Cart64K &k)
{
    const double xo = AX == 0 ? k.xo : k.yo, xh = AX == 0 ? k.xh : k.yh, td = AX == 0 ? k.ydt : k.xdt;
    // velocities along +n, -n; (+n, +t) (-n, +t) (-n, -t) (+n, -t); tangential +t, -t
    constexpr int P = AX == 0 ? 1 : 2, M = AX == 0 ? 3 : 4, TP = AX == 0 ? 2 : 1, TM = AX == 0 ? 4 : 3;
    constexpr int PP = 5, MP = AX == 0 ? 6 : 8, MM = 7, PM = AX == 0 ? 8 : 6;
    auto at = [&](int a, int o) { return f[a * LP + l + o]; };
    auto low = [&](int a) { return fma(xo, at(a, S) - at(a, -S), at(a, 0)); };               // from the lower side
    auto high = [&](int a) { return fma(-xo, at(a, 2 * S) - at(a, 0), at(a, S)); };           // from the upper side
    auto tan = [&](int a) {          // both sides along the axis
        const double t = at(a, 0) + at(a, S), u = at(a, -S) + at(a, 2 * S);
        return fma(0.5 * xh, t - u, 0.5 * t);
    };
    auto across = [&](int a) {       // sum of both sides' differences across
        return (at(a, T) + at(a, S + T)) - (at(a, -T) + at(a, S - T));
    };
    double fb[NQ];
    fb[0] = tan(0);
    fb[P] = low(P);
    fb[M] = high(M);
    fb[TP] = fma(-0.5 * td, across(TP), tan(TP));
    fb[TM] = fma(0.5 * td, across(TM), tan(TM));
    fb[PP] = fma(-td, at(PP, T) - at(PP, -T), low(PP));
    fb[PM] = fma(td, at(PM, T) - at(PM, -T), low(PM));
    fb[MP] = fma(-td, at(MP, S + T) - at(MP, S - T), high(MP));
    fb[MM] = fma(td, at(MM, S + T) - at(MM, S - T), high(MM));
    double w0, w1, w2, fe[NQ];
    moments64(fb, w0, w1, w2);
    const double iv = recip64(w0);
    feq64<false>(k.bg[AX] * w0, w1 * iv, w2 * iv, fe);
#pragma unroll
    for (int q = 0; q < 6; q++) {
        const int a = AX == 0 ? XSLOT_A(q) : YSLOT_A(q);
        flux[q] = fma(k.g[AX], fb[a], fe[a]);
    }
}

// Boundary face in direction D (0 +x, 1 -x, 2 +y, 3 -y) of the cell staged at l with state
// (f^n, W^n) at g, on grid side `side`: its six fluxes as face64 gives them (Sec. III rules,
// as cart_boundary_face).
template <int D, int LP, int LX, bool DIAG>
__device__ __forceinline__ void boundary64(double flux[6], const double *f, int l, const CartInst &m, int side, int pos,
                                           const Cart64K &k, const double *__restrict__ fin, const double *__restrict__ Wn,
                                           int64_t g)
{
    constexpr int AX = D < 2 ? 0 : 1, S = AX == 0 ? 1 : LX, T = AX == 0 ? LX : 1;
    const int64_t np = m.npad;
    const double rho = Wn[g], iv = recip64(rho), ux = Wn[np + g] * iv, uy = Wn[2 * np + g] * iv;
    const int bk = m.side_kind[side];
    double rb = rho, ubx = 0.0, uby = 0.0;
    if (bk == BK_MOVING_WALL) { ubx = m.side_par[side][0]; uby = m.side_par[side][1]; }
    else if (bk == BK_FARFIELD) { rb = m.side_par[side][0]; ubx = m.side_par[side][1]; uby = m.side_par[side][2]; }
    else if (bk == BK_OUTLET) { ubx = ux; uby = uy; }
    double feqb[NQ], feqn[NQ];
    feq64<false>(rb, ubx, uby, feqb);
    feq64<false>(rho, ux, uy, feqn);
    const double xo = AX == 0 ? k.xo : k.yo, td = AX == 0 ? k.ydt : k.xdt;
    double px = 0.0, py = 0.0;
#pragma unroll
    for (int q = 0; q < 6; q++) {
        const int a = AX == 0 ? XSLOT_A(q) : YSLOT_A(q);
        const int n = AX == 0 ? EX(a) : EY(a), t = AX == 0 ? EY(a) : EX(a);
        const int out = (D == 0 || D == 2) ? n : -n;
        double fb;
        if (out < 0) fb = feqb[a] + (fin[a * np + g] - feqn[a]);         // non-equilibrium extrapolation
        else {
            const double *const c = f + a * LP + l;
            double A = fma(n > 0 ? xo : -xo, c[S] - c[-S], c[0]);
            if (t != 0) A = fma(t > 0 ? -td : td, c[T] - c[-T], A);
            fb = fma(k.b, feqb[a], A) * k.c;
        }
        flux[q] = k.lv[AX] * fb;
        if (DIAG) {
            px += (double)(EX(a) * out) * fb;
            py += (double)(EY(a) * out) * fb;
        }
    }
    if (DIAG) {
        const double len = AX == 0 ? m.dy : m.dx;
        cart_face_momentum(m, side, pos, len * px, len * py);
    }
}

// One block; s_f: shared memory of Shape64::SMEM bytes.  BOX (blocks whose ring lies inside the
// grid): f^n of the block and its ring has been copied to s_f, and W^n to where the fluxes go later.
template <int BX, int BY, bool DIAG, bool BOX>
__device__ __forceinline__ void cart64_block(const CartInst &m, const Cart64K &k, int par, double *s_f)
{
    using Sh = Shape64<BX, BY>;
    constexpr int LX = Sh::LX, LY = Sh::LY, LP = Sh::LP, NT = Sh::NT;
    double *const s_fx = s_f + NQ * LP, *const s_fy = s_fx + 6 * Sh::NXF;      // s_f [NQ][LY][LX]
    const double *__restrict__ fin = static_cast<const double *>(m.f[par]);
    double *__restrict__ fout = static_cast<double *>(m.f[1 - par]);
    const double *__restrict__ Wn = m.W[par];
    double *__restrict__ Wout = m.W[1 - par];
    const int x0 = blockIdx.x * BX, y0 = blockIdx.y * BY, nx = m.nx, ny = m.ny, tid = threadIdx.x;
    const int64_t np = m.npad, pitch = m.pitch;
    const bool px = m.periodic_x != 0, py = m.periodic_y != 0;
    const bool symL = !px && m.side_kind[3] == BK_SYMMETRY, symR = !px && m.side_kind[1] == BK_SYMMETRY;
    const bool symB = !py && m.side_kind[0] == BK_SYMMETRY, symT = !py && m.side_kind[2] == BK_SYMMETRY;

    // ---- phase 1: fbar+ of the block and its ring (periodic sides wrap, symmetry sides
    // mirror; positions past a wall are left to the ghosts below)
    for (int p = tid; p < LP; p += NT) {
        int gi = x0 + p % LX - 2, gj = y0 + p / LX - 2, mir = 0;
        bool in = true;
        if (!BOX && (gi < 0 || gi >= nx)) {
            if (px) { gi %= nx; if (gi < 0) gi += nx; }
            else if (gi < 0 ? symL : symR) { gi = gi < 0 ? -1 - gi : 2 * nx - 1 - gi; mir |= 1; }
            in = gi >= 0 && gi < nx;
        }
        if (!BOX && (gj < 0 || gj >= ny)) {
            if (py) { gj %= ny; if (gj < 0) gj += ny; }
            else if (gj < 0 ? symB : symT) { gj = gj < 0 ? -1 - gj : 2 * ny - 1 - gj; mir |= 2; }
            in = in && gj >= 0 && gj < ny;
        }
        if (!in) continue;
        const int64_t g = gi + pitch * gj;
        double fv[NQ], fe[NQ];
        const double *const w = BOX ? s_fx + p : Wn + g, *const fs = BOX ? s_f + p : fin + g;
        const int64_t ws = BOX ? LP : np;
        const double w0 = w[0], w1 = w[ws], w2 = w[2 * ws];
#pragma unroll
        for (int a = 0; a < NQ; a++) fv[a] = fs[a * ws];
        const double iv = recip64(w0);
        feq64<true>(w0, w1 * iv, w2 * iv, fe);
#pragma unroll
        for (int a = 0; a < NQ; a++) {
            const int d = mir == 0 ? a : (mir == 1 ? MIRROR_X(a) : (mir == 2 ? MIRROR_Y(a) : MIRROR_X(MIRROR_Y(a))));
            s_f[d * LP + p] = fma(k.b, fe[a] - fv[a], fv[a]);
        }
    }
    __syncthreads();
    // ---- beside a wall: the missing neighbour as the linear extrapolation of the first two
    // cells (their difference across the wall cell is then twice the one-sided one)
    {
        const int lr = nx - x0 + 2, lt = ny - y0 + 2;              // staged column / row past the last cells
        const bool wl = !px && !symL && x0 == 0, wr = !px && !symR && lr < LX;
        const bool wb = !py && !symB && y0 == 0, wt = !py && !symT && lt < LY;
        if (wl || wr || wb || wt) {
            for (int q = tid; q < NQ * LY; q += NT) {
                double *const row = s_f + q * LX;                   // plane q / LY, row q % LY
                if (wl) row[1] = 2.0 * row[2] - row[3];
                if (wr) row[lr] = 2.0 * row[lr - 1] - row[lr - 2];
            }
            for (int q = tid; q < NQ * LX; q += NT) {
                double *const col = s_f + (q / LX) * LP + q % LX;
                if (wb) col[LX] = 2.0 * col[2 * LX] - col[3 * LX];
                if (wt) col[lt * LX] = 2.0 * col[(lt - 1) * LX] - col[(lt - 2) * LX];
            }
            __syncthreads();
        }
    }

    // ---- phase 2: faces of constant x (whole warps), then of constant y, then a warp for
    // the faces of the block on each wall (a few lanes of one warp in the place of some lanes
    // of every cell warp)
    for (int t = tid; t < Sh::XF + Sh::YF + 128; t += NT) {
        double fl[6];
        if (t < Sh::XF) {
            const int fi = t % (BX + 1), fj = t / (BX + 1), c = x0 + fi;
            if (t >= Sh::NXF || y0 + fj >= ny || c > nx || (c == 0 && !px && !symL) || (c == nx && !px && !symR)) continue;
            face64<0, LP, 1, LX>(fl, s_f, (fj + 2) * LX + fi + 1, k);
#pragma unroll
            for (int q = 0; q < 6; q++) s_fx[q * Sh::NXF + t] = fl[q];
        } else if (t < Sh::XF + Sh::YF) {
            const int u = t - Sh::XF, fi = u % BX, fj = u / BX, c = y0 + fj;
            if (u >= Sh::NYF || x0 + fi >= nx || c > ny || (c == 0 && !py && !symB) || (c == ny && !py && !symT)) continue;
            face64<1, LP, LX, 1>(fl, s_f, (fj + 1) * LX + fi + 2, k);
#pragma unroll
            for (int q = 0; q < 6; q++) s_fy[q * Sh::NYF + u] = fl[q];
        } else {
            const int w = (t - Sh::XF - Sh::YF) >> 5, i = t & 31;       // right, left, top, bottom
            const int ic = w == 0 ? nx - 1 - x0 : w == 1 ? 0 : i, jc = w == 2 ? ny - 1 - y0 : w == 3 ? 0 : i;
            const bool wall = w == 0 ? !px && !symR && ic < BX : w == 1 ? !px && !symL && x0 == 0
                              : w == 2 ? !py && !symT && jc < BY : !py && !symB && y0 == 0;
            if (!wall || ic >= BX || jc >= BY || x0 + ic >= nx || y0 + jc >= ny) continue;
            const int l = (jc + 2) * LX + ic + 2;
            const int64_t g = x0 + ic + pitch * (y0 + jc);
            double *dst;
            if (w == 0) boundary64<0, LP, LX, DIAG>(fl, s_f, l, m, 1, y0 + jc, k, fin, Wn, g);
            else if (w == 1) boundary64<1, LP, LX, DIAG>(fl, s_f, l, m, 3, y0 + jc, k, fin, Wn, g);
            else if (w == 2) boundary64<2, LP, LX, DIAG>(fl, s_f, l, m, 2, x0 + ic, k, fin, Wn, g);
            else boundary64<3, LP, LX, DIAG>(fl, s_f, l, m, 0, x0 + ic, k, fin, Wn, g);
            dst = w < 2 ? s_fx + jc * (BX + 1) + ic + (w == 0) : s_fy + (jc + (w == 2)) * BX + ic;
#pragma unroll
            for (int q = 0; q < 6; q++) dst[q * (w < 2 ? Sh::NXF : Sh::NYF)] = fl[q];
        }
    }
    __syncthreads();

    // ---- phase 3: cells
    const int ti = tid % BX, tj = tid / BX, gi = x0 + ti, gj = y0 + tj;
    if (tj >= BY || gi >= nx || gj >= ny) return;
    const int64_t g = gi + pitch * gj;
    double fn[NQ];
#pragma unroll
    for (int a = 0; a < NQ; a++) fn[a] = fin[a * np + g];
    const double w0 = Wn[g], w1 = Wn[np + g], w2 = Wn[2 * np + g];
    const int fW = tj * (BX + 1) + ti, fE = fW + 1, fS = tj * BX + ti, fN = fS + BX;
    // the unsigned fluxes: out through one side minus in through the other, times the sign
    // of the velocity's component
    double F[NQ];
#pragma unroll
    for (int a = 0; a < NQ; a++) F[a] = 0.0;
#pragma unroll
    for (int q = 0; q < 6; q++) {
        const double d = s_fx[q * Sh::NXF + fE] - s_fx[q * Sh::NXF + fW];
        F[XSLOT_A(q)] = EX(XSLOT_A(q)) > 0 ? d : -d;
    }
#pragma unroll
    for (int q = 0; q < 6; q++) {
        const double d = s_fy[q * Sh::NYF + fN] - s_fy[q * Sh::NYF + fS];
        F[YSLOT_A(q)] += EY(YSLOT_A(q)) > 0 ? d : -d;
    }
    if (DIAG) {
        // symmetry sides are staged as mirror ghosts: the momentum leaving through such a
        // face is the moment of its flux
        auto sym_face = [&](int side, int pos, const double *fl, int stride, bool y_face, double sgn) {
            double qx = 0.0, qy = 0.0;
#pragma unroll
            for (int r = 0; r < 6; r++) {
                const int a = y_face ? YSLOT_A(r) : XSLOT_A(r);
                const double v = (double)(y_face ? EY(a) : EX(a)) * fl[r * stride];
                qx += (double)EX(a) * v;
                qy += (double)EY(a) * v;
            }
            cart_face_momentum(m, side, pos, sgn * k.rdtV * qx, sgn * k.rdtV * qy);
        };
        if (symL && gi == 0) sym_face(3, gj, s_fx + fW, Sh::NXF, false, -1.0);
        if (symR && gi == nx - 1) sym_face(1, gj, s_fx + fE, Sh::NXF, false, 1.0);
        if (symB && gj == 0) sym_face(0, gi, s_fy + fS, Sh::NYF, true, -1.0);
        if (symT && gj == ny - 1) sym_face(2, gi, s_fy + fN, Sh::NYF, true, 1.0);
    }
    double m0, m1, m2, fe[NQ];
    moments64(F, m0, m1, m2);
    const double W0 = w0 - m0, W1 = w1 - m1, W2 = w2 - m2;
    Wout[g] = W0;
    Wout[np + g] = W1;
    Wout[2 * np + g] = W2;
    const double iv = recip64(W0);
    feq64<true>(W0, W1 * iv, W2 * iv, fe);
#pragma unroll
    for (int a = 0; a < NQ; a++) {
        const double t = a == 0 ? fn[a] : fn[a] - F[a];
        fout[a * np + g] = fma(k.ri, fe[a] - t, t);
    }
}

template <int BX, int BY, bool DIAG>
__global__ void __launch_bounds__(Shape64<BX, BY>::NT, Shape64<BX, BY>::CTAS)
k_step_cart64(const CartInst m, const Cart64K k, int par)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    step_dependency_wait();
    cart64_block<BX, BY, DIAG, false>(m, k, par, reinterpret_cast<double *>(smem_raw));
}

// TMA staging: f^n and W^n of the blocks whose ring lies inside the grid come by two tensor
// copies (tf, tw: the maps of buffer par), f^n straight to where its fbar+ goes, each thread replacing
// what it read.  The arithmetic is that of the other blocks: the same bits as with plain loads.
using Sh64T = Shape64<16, 16>;
static_assert(CartTmaBox<P_FP64, 16, 16>::F_BYTES == sizeof(double) * NQ * Sh64T::LP, "the f box is s_f");
static_assert(CartTmaBox<P_FP64, 16, 16>::F_BYTES % 128 == 0, "the W box starts on a 128-byte boundary");
static_assert(CartTmaBox<P_FP64, 16, 16>::W_BYTES <= sizeof(double) * 6 * (Sh64T::NXF + Sh64T::NYF), "the W box fits the fluxes' place");
constexpr size_t SMEM64T = Sh64T::SMEM + 16 + 128;           // the barrier; 128 bytes of slack align the base
__global__ void __launch_bounds__(Sh64T::NT, Sh64T::CTAS)
k_step_cart64_tma(const CartInst m, const Cart64K k, int par, const __grid_constant__ CUtensorMap tf,
                  const __grid_constant__ CUtensorMap tw)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    step_dependency_wait();
    uint32_t sa;
    unsigned char *const sm = aligned_smem(smem_raw, sa);
    double *const s_f = reinterpret_cast<double *>(sm);
    if (cart_block_interior<16, 16>(m, blockIdx.x, blockIdx.y)) {
        const uint32_t bar = sa + (uint32_t)Sh64T::SMEM;
        if (threadIdx.x == 0) mbar_init(bar);
        __syncthreads();
        if (threadIdx.x == 0)
            tma_issue_block<P_FP64, 16, 16>(bar, sa, sa + (uint32_t)CartTmaBox<P_FP64, 16, 16>::F_BYTES, &tf, &tw,
                                            blockIdx.x * 16, blockIdx.y * 16);
        if (!cta_wait_staged(m, bar, 0)) return;
        cart64_block<16, 16, false, true>(m, k, par, s_f);
    } else {
        cart64_block<16, 16, false, false>(m, k, par, s_f);
    }
}

Cart64K coefs64(const CartInst &m)
{
    Cart64K k;
    // parts of one whole, the larger rounded and the smaller what it leaves: rounded each by itself
    // the whole is off, alike in every step
    auto parts = [](double q, double whole, double &p, double &r) {      // q of the whole in r, the rest in p
        if (q > 0.5 * whole) { r = q; p = whole - q; }
        else { p = whole - q; r = whole - p; }
    };
    k.b = m.b;
    k.ri = m.r / (1.0 + m.r);
    k.c = 1.0 / (1.0 + k.b);
    k.dtV = m.dtV; k.rdtV = 1.0 / m.dtV;
    k.lv[0] = m.dy * m.dtV; k.lv[1] = m.dx * m.dtV;
    for (int x = 0; x < 2; x++) parts(k.lv[x] * (k.b * k.c), k.lv[x], k.g[x], k.bg[x]);
    const double ax = 0.5 * m.ihx, ay = 0.5 * m.ihy;
    k.xdt = m.dt * ax; k.xh = 0.25; k.xo = 0.25 - k.xdt;
    k.ydt = m.dt * ay; k.yh = 0.25; k.yo = 0.25 - k.ydt;
    return k;
}

template <int BX, int BY> cudaError_t launch64(const CartInst &m, int parity, cudaStream_t st)
{
    using Sh = Shape64<BX, BY>;
    const dim3 grid((m.nx + BX - 1) / BX, (m.ny + BY - 1) / BY);
    // no early start: the blocks have to lie evenly on the SMs' FP64 pipes (256^2, in this kernel's
    // first form: 62.8 us, with it 87.3; then 54, now 56)
    if (m.force || m.bface)
        return launch_step_kernel(false, k_step_cart64<BX, BY, true>, grid, dim3(Sh::NT), Sh::SMEM, st, m, coefs64(m), parity);
    return launch_step_kernel(false, k_step_cart64<BX, BY, false>, grid, dim3(Sh::NT), Sh::SMEM, st, m, coefs64(m), parity);
}

template <int BX, int BY> cudaError_t prepare64()
{
    cudaError_t e = cudaFuncSetAttribute(k_step_cart64<BX, BY, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)Shape64<BX, BY>::SMEM);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_step_cart64<BX, BY, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)Shape64<BX, BY>::SMEM);
    return e;
}

// FP64 warp instructions on the fullest SM.
template <int BX, int BY> int64_t cost64(int nx, int ny, int n_sm)
{
    const int64_t blocks = (int64_t)((nx + BX - 1) / BX) * ((ny + BY - 1) / BY);
    if ((ny + BY - 1) / BY > 65535) return INT64_MAX;
    return (blocks + n_sm - 1) / n_sm * Shape64<BX, BY>::COST;
}

}  // namespace

int cart64_shape(int nx, int ny, int n_sm)          // an index of CART64_BLOCK
{
    const int64_t c[3] = {cost64<16, 14>(nx, ny, n_sm), cost64<8, 8>(nx, ny, n_sm), cost64<4, 4>(nx, ny, n_sm)};
    return c[0] <= c[1] && c[0] <= c[2] ? 0 : (c[1] <= c[2] ? 1 : 2);
}

cudaError_t prepare_cart64()
{
    cudaError_t e = prepare64<16, 14>();
    if (e == cudaSuccess) e = prepare64<8, 8>();
    if (e == cudaSuccess) e = prepare64<4, 4>();
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_step_cart64_tma, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SMEM64T);
    return e;
}

cudaError_t launch_step_cart64_tma(const CartInst &m, const CartTma &tma, int parity, cudaStream_t st)
{
    const dim3 grid((m.nx + 15) / 16, (m.ny + 15) / 16);
    return launch_step_kernel(false, k_step_cart64_tma, grid, dim3(Sh64T::NT), SMEM64T, st, m, coefs64(m), parity,
                              tma.f[parity], tma.W[parity]);
}

cudaError_t launch_step_cart64(const CartInst &m, int shape, int parity, cudaStream_t st)
{
    if (shape == 1) return launch64<8, 8>(m, parity, st);
    if (shape == 2) return launch64<4, 4>(m, parity, st);
    return launch64<16, 14>(m, parity, st);
}

}  // namespace sdugks
