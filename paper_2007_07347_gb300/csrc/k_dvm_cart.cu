// k_dvm_cart.cu -- the rarefied S-DUGKS step (k_dvm.cu) on uniform Cartesian grids.
//
// The interface states need moments over all Q velocities of the reconstructed
// distribution, which k_dvm.cu forms from the five rows of each upwind stencil of every face,
// writing the face fluxes (twice the size of f) to memory for its cell kernel.  Here the
// reconstruction's linearity takes the stencil out of that pass.  Towards the face at +h/2
//     fbar = phi + (h/2 - xi_x dt) dphi/dx - xi_y dt dphi/dy,      phi = fbar+,
// with differences of neighbouring cells as derivatives, so a moment of fbar over the
// velocities of one sign is a combination of the same half-range moments of phi, of one
// degree more, in the cell and its neighbours.
//
// phi, not f, is what is kept from step to step: phi = a f + b feq (a + b = 1), and Eq. fn+1
// for f is
//     phi^{n+1} = (phi - b feq - a F) / (1 + dt/tau) + (a r / (1 + r) + b) feq^{n+1},   r = dt/tau,
// without a division by a: each phi is read where a neighbour needs it without a Maxwellian of
// that neighbour.  f = (phi - b feq) / a when the caller asks for it; a >= 1/2 (dt <= tau)
// is this path's condition, so that no more than a bit of f is lost.
//
// One step:
//   k_dvc_moments  per cell: quadrant moments (degree <= 4) of its phi, one pass
//   k_dvc_states   per cell: its four interface states and macroscopic fluxes from the
//                  moments (Eqs. Macro, MacroFlux; diffuse walls), W^{n+1} in FP64 (Eq.
//                  MacroUpdate), and the one-axis factors of the interface equilibria and of
//                  feq(W^{n+1}) (the velocity grid is a tensor product)
//   k_dvc_update   phi^{n+1} into the other buffer, marching along lines of cells
// Moments are taken of phi less one resting Maxwellian (wall temperature, unit density), the
// same for every cell: it has no gradient and no net flux, and FP32 sums of the small rest
// keep the precision that the differences of neighbouring moments need.
//
// A step of the 40 x 40 x 100^2 micro cavity in FP32: 90 us where k_dvm.cu takes 171 (23 x 23 x 50^2:
// 19.1 / 36.5; 32 x 32 x 99^2: 68 / 212; FP64 30 x 30 x 64^2: 326 / 1285), of which the three kernels,
// each by itself with cold caches, are 24, 15 and 68.  With f kept, and so a Maxwellian
// for every cell read, a step took 140; with an update of single cells, ten reads each, 153.
#include "d2q9.cuh"
#include <algorithm>
#include <type_traits>

namespace sdugks {
namespace {

constexpr int NMOM = 15;                       // monomials x^a y^b with a + b <= 4
__host__ __device__ constexpr int mono(int a, int b) { return (a + b) * (a + b + 1) / 2 + b; }
constexpr int MOM_THREADS = 256, STATE_THREADS = 128, UPD_THREADS = 64;

// The step's constants in the compute precision.
template <class R> __device__ __forceinline__ const DvmCartK<R> &consts(const DvmCart &m);
template <> __device__ __forceinline__ const DvmCartK<float> &consts<float>(const DvmCart &m) { return m.kf; }
template <> __device__ __forceinline__ const DvmCartK<double> &consts<double>(const DvmCart &m) { return m.kd; }

// exp(-(x - u)^2 beta); FP32: beta times log2 e.  In FP32 to about one ulp: the rounding errors of the
// difference and of the products are carried along, and 2^r on |r| <= 1/2 is its Taylor
// series (the term of degree 8 is below 6e-9): the errors of a table of nv nodes average out less than
// those of nv^2 Maxwellians would.  A run that breaks down (R T, and with it beta, below zero) has to
// show it: the exponential's overflow is infinity and an undefined exponent NaN, as exp gives them.
// ul, bl: what u and beta leave out (FP32).
template <class R> __device__ __forceinline__ R gauss(R x, R u, R beta, R ul = R(0), R bl = R(0));
template <> __device__ __forceinline__ float gauss<float>(float x, float u, float beta, float ul, float bl)
{
    const float d = x - u, v = d - x, dl = (x - (d - v)) + (-u - v) - ul;
    const float hi = d * d, lo = fmaf(d, d, -hi) + 2.0f * d * dl, t = hi * beta;
    const float tl = fmaf(hi, beta, -t) + fmaf(lo, beta, hi * bl);
    const float n = rintf(fmaxf(fminf(t, 140.0f), -128.0f)), r = n - t;   // 2^-t = 2^-n 2^r
    float q = 1.5252734e-5f;                                              // (ln 2)^k / k!, k = 7 .. 1
    q = fmaf(q, r, 1.5403530e-4f);
    q = fmaf(q, r, 1.3333558e-3f);
    q = fmaf(q, r, 9.6181291e-3f);
    q = fmaf(q, r, 5.5504109e-2f);
    q = fmaf(q, r, 2.4022651e-1f);
    q = fmaf(q, r, 6.9314718e-1f);
    const float g = 1.0f + fmaf(q, r, -0.69314718f * tl * fmaf(q, r, 1.0f));
    if (!(t > -128.0f)) return t != t ? t : INFINITY;
    return t < 120.0f ? g * __int_as_float((127 - (int)n) << 23) : 0.0f;
}
template <> __device__ __forceinline__ double gauss<double>(double x, double u, double beta, double, double)
{
    return exp(-(x - u) * (x - u) * beta);
}

// Pairs of velocities (two columns in the moments, two rows in the update): paired FP32
// instructions, or two FP64 ones.
template <class R> struct PairT;
template <> struct PairT<float> { using T = float2; };
template <> struct PairT<double> { using T = double2; };
__device__ __forceinline__ float2 pset(float a, float b) { return make_float2(a, b); }
__device__ __forceinline__ double2 pset(double a, double b) { return make_double2(a, b); }
__device__ __forceinline__ float2 pfma(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 pmul(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 psub(float2 a, float2 b) { return __ffma2_rn(b, make_float2(-1.0f, -1.0f), a); }
__device__ __forceinline__ double2 pfma(double2 a, double2 b, double2 c) { return make_double2(fma(a.x, b.x, c.x), fma(a.y, b.y, c.y)); }
__device__ __forceinline__ double2 pmul(double2 a, double2 b) { return make_double2(a.x * b.x, a.y * b.y); }
__device__ __forceinline__ double2 psub(double2 a, double2 b) { return make_double2(a.x - b.x, a.y - b.y); }
template <class R> __device__ __forceinline__ typename PairT<R>::T pdup(R v) { return pset(v, v); }

// The columns of the velocity grid in pairs: those of xi_x < 0, then the others (the zero
// column of an odd grid among them).  n: 2, or 1 for the last of an odd number.
struct ColPair {
    int j, n, positive;
    __device__ __forceinline__ ColPair(int nv, int g)
    {
        const int neg = nv / 2, gn = (neg + 1) / 2;
        positive = g >= gn;
        j = positive ? neg + 2 * (g - gn) : 2 * g;
        n = min(2, (positive ? nv : neg) - j);
    }
};
__host__ __device__ constexpr int col_pairs(int nv) { return (nv / 2 + 1) / 2 + (nv - nv / 2 + 1) / 2; }
// ALIGNED (nv a multiple of 4): every pair is full and starts at an even column of a row that
// starts at an even offset, one vector access; otherwise two, the missing second column
// repeating the first.
template <class R, bool ALIGNED> __device__ __forceinline__ typename PairT<R>::T pload(const R *p, int n)
{
    if constexpr (ALIGNED) return *reinterpret_cast<const typename PairT<R>::T *>(p);
    else return pset(p[0], p[n - 1]);
}
template <class R, bool ALIGNED> __device__ __forceinline__ void pstore(R *p, typename PairT<R>::T v, int n)
{
    if constexpr (ALIGNED) *reinterpret_cast<typename PairT<R>::T *>(p) = v;
    else {
        p[0] = v.x;
        if (n == 2) p[1] = v.y;
    }
}

// A table of one-axis factors: [nv] along x, then along y the nodes < 0 and the others, each half
// padded so that a thread's rows are one aligned vector.
__host__ __device__ constexpr int tab_y(int nv) { return (nv + 7) / 8 * 8; }
__host__ __device__ constexpr int tab_half(int nv) { return (nv - nv / 2 + 7) / 8 * 8; }
__host__ __device__ constexpr int tab_size(int nv) { return tab_y(nv) + 2 * tab_half(nv); }
__device__ __forceinline__ int tab_row(int nv, int i) { return tab_y(nv) + (i >= nv / 2 ? tab_half(nv) - nv / 2 : 0) + i; }

// 2 RP values from an aligned place
template <class R, int RP> __device__ __forceinline__ void load_rows(const R *p, typename PairT<R>::T v[RP])
{
    if constexpr (sizeof(R) == 4 && RP % 2 == 0) {
#pragma unroll
        for (int k = 0; k < RP / 2; k++) {
            const float4 q = reinterpret_cast<const float4 *>(p)[k];
            v[2 * k] = make_float2(q.x, q.y);
            v[2 * k + 1] = make_float2(q.z, q.w);
        }
    } else {
#pragma unroll
        for (int k = 0; k < RP; k++) v[k] = reinterpret_cast<const typename PairT<R>::T *>(p)[k];
    }
}

// Rows (or columns) of one sign: [lo, hi), and the zero node (odd nv), which belongs to
// both halves with weight 1/2.
__device__ __forceinline__ void half_range(int nv, int positive, int &lo, int &hi)
{
    lo = positive ? nv - nv / 2 : 0;
    hi = positive ? nv : nv / 2;
}

// Half-range sum of t(x) xp(x) over the nodes of one sign (the zero node with weight 1/2), by
// four lanes (u = lane & 3), the result on all four.
template <class R> __device__ __forceinline__ R half_sum(const R *t, const R *xp, int nv, int positive, int u)
{
    int lo, hi;
    half_range(nv, positive, lo, hi);
    R s = R(0);
#pragma unroll 4
    for (int j = lo + u; j < hi; j += 4) s += t[j] * xp[j];
    if ((nv & 1) && u == 0) s += R(0.5) * (t[nv / 2] * xp[nv / 2]);
    s += __shfl_xor_sync(0xffffffffu, s, 1);
    s += __shfl_xor_sync(0xffffffffu, s, 2);
    return s;
}

// Parameters of feq of a cell's W.  In FP32 each is the sum of two numbers (_l: the second).
// Rounded to one, the factor and the temperature put all of a cell's Maxwellian off alike, in
// every step: R T was off by 2.3e-8 (root mean square, 40 x 40 x 100^2, 50 steps) where the general
// kernels are by 0.8e-8.
template <class R> struct Maxwell {
    R amp, amp_l, u[2], u_l[2], beta, beta_l;
};
struct FF {                                    // h + l, |l| <= ulp(h) / 2
    float h, l;
};
__device__ __forceinline__ FF ff_norm(float h, float l)
{
    const float s = h + l;
    return {s, l - (s - h)};
}
__device__ __forceinline__ FF ff_add(FF a, FF b)
{
    const float s = a.h + b.h, v = s - a.h;
    return ff_norm(s, ((a.h - (s - v)) + (b.h - v)) + (a.l + b.l));
}
__device__ __forceinline__ FF ff_mul(FF a, FF b)
{
    const float p = a.h * b.h;
    return ff_norm(p, fmaf(a.h, b.h, -p) + fmaf(a.h, b.l, a.l * b.h));
}
__device__ __forceinline__ FF ff_inv(FF a)
{
    const float q = recip<float>(a.h);
    return ff_norm(q, q * (fmaf(-a.h, q, 1.0f) - a.l * q));
}

// w: W, and in FP32 what that leaves out of it.  (FP32: no FP64 divisions, for which the block would wait.)
__device__ __forceinline__ void maxwell_of(Maxwell<float> &p, const float w[8], const DvmCartK<float> &K)
{
    constexpr double L = 0.5 * 1.4426950408889634;              // log2 e / 2
    const FF r{w[0], w[4]}, ir = ff_inv(r), ux = ff_mul({w[1], w[5]}, ir), uy = ff_mul({w[2], w[6]}, ir);
    const FF uu = ff_add(ff_mul(ux, ux), ff_mul(uy, uy));
    const FF iRT = ff_inv(ff_add(ff_mul({w[3], w[7]}, ir), {-0.5f * uu.h, -0.5f * uu.l}));
    const FF amp = ff_mul(ff_mul(r, iRT), {K.amp, K.amp_l}), beta = ff_mul(iRT, {(float)L, (float)(L - (double)(float)L)});
    p = {amp.h, amp.l, {ux.h, uy.h}, {ux.l, uy.l}, beta.h, beta.l};
}
__device__ __forceinline__ void maxwell_of(Maxwell<double> &p, const double w[8], const DvmCartK<double> &K)
{
    const double ir = 1.0 / w[0], ux = w[1] * ir, uy = w[2] * ir, iRT = 1.0 / (w[3] * ir - 0.5 * (ux * ux + uy * uy));
    p = {w[0] * iRT * K.amp, 0.0, {ux, uy}, {0.0, 0.0}, 0.5 * iRT, 0.0};
}
// By one warp, whose lanes 0 to 3 hold W in v.
template <class R> __device__ __forceinline__ Maxwell<R> warp_maxwell(double v, const DvmCartK<R> &K)
{
    const R h = (R)v, l = sizeof(R) == 4 ? (R)(v - (double)h) : R(0);
    R w[8];
#pragma unroll
    for (int k = 0; k < 4; k++) {
        w[k] = __shfl_sync(0xffffffffu, h, k);
        w[4 + k] = __shfl_sync(0xffffffffu, l, k);
    }
    Maxwell<R> p;
    maxwell_of(p, w, K);
    return p;
}
// its one-axis factors (those along y with the density and node weight), by all threads of the block
template <class R> __device__ __forceinline__ void cell_tables(const DvmCart &m, const Maxwell<R> &p, R *tab)
{
    const int nv = m.nv;
    for (int j = threadIdx.x; j < nv; j += blockDim.x) {
        const R x = static_cast<const R *>(m.vnode)[j], gy = gauss<R>(x, p.u[1], p.beta, p.u_l[1], p.beta_l);
        tab[j] = gauss<R>(x, p.u[0], p.beta, p.u_l[0], p.beta_l);
        tab[tab_row(nv, j)] = fma(p.amp, gy, p.amp_l * gy);
    }
}

// ---- initial state: f = feq(W) = phi, its tables
template <class R>
__global__ void __launch_bounds__(STATE_THREADS) k_dvc_init(const DvmCart m, const double *__restrict__ W, R *__restrict__ phi,
                                                           R *__restrict__ tab)
{
    __shared__ Maxwell<R> par;
    const int64_t c = blockIdx.x;
    R *const t = tab + c * tab_size(m.nv);
    if (threadIdx.x < 32) {
        const Maxwell<R> p = warp_maxwell<R>(W[4 * c + (threadIdx.x & 3)], consts<R>(m));
        if (threadIdx.x == 0) par = p;
    }
    __syncthreads();
    cell_tables<R>(m, par, t);
    __syncthreads();
    for (int q = threadIdx.x; q < m.nv * m.nv; q += blockDim.x) phi[c * m.Q + q] = t[q % m.nv] * t[tab_row(m.nv, q / m.nv)];
}

// ---- f of the present state
template <class R>
__global__ void __launch_bounds__(STATE_THREADS) k_dvc_f(const DvmCart m, const R *__restrict__ phi, const R *__restrict__ tab,
                                                        R *__restrict__ f)
{
    const DvmCartK<R> &K = consts<R>(m);
    const int64_t c = blockIdx.x;
    const R *const t = tab + c * tab_size(m.nv);
    const R ia = R(1) / K.a;
    for (int q = threadIdx.x; q < m.nv * m.nv; q += blockDim.x)
        f[c * m.Q + q] = (phi[c * m.Q + q] - K.b * (t[q % m.nv] * t[tab_row(m.nv, q / m.nv)])) * ia;
}

// ---- quadrant moments of phi less the reference, per cell: mom[c][sx + 2 sy][NMOM].
// A thread owns a pair of columns of the velocity grid and some of its rows, so that only powers of
// y multiply in the loop; columns are weighted with powers of x at the end.
template <class R, bool ALIGNED>
__global__ void __launch_bounds__(MOM_THREADS) k_dvc_moments(const DvmCart m, const R *__restrict__ f,
                                                            R *__restrict__ mom)
{
    using P = typename PairT<R>::T;
    extern __shared__ __align__(16) unsigned char dyn[];
    const int nv = m.nv, CG = col_pairs(nv), CT = min(CG, MOM_THREADS), NR = MOM_THREADS / CT;
    // yp [row][6]: the reference's factor and powers 1..4 of y, each twice (one operand of a paired
    // instruction); xp [5][nv]: powers of x; S [2][NR][5][nv]
    P *const yp = reinterpret_cast<P *>(dyn);
    R *const xp = reinterpret_cast<R *>(yp + 6 * nv), *const S = xp + 5 * nv;
    for (int j = threadIdx.x; j < nv; j += blockDim.x) {
        const R x = static_cast<const R *>(m.vnode)[j], x2 = x * x;
        const R q[5] = {R(1), x, x2, x * x2, x2 * x2};
        yp[6 * j] = pdup(static_cast<const R *>(m.m0)[nv + j]);
#pragma unroll
        for (int k = 0; k < 5; k++) {
            xp[k * nv + j] = q[k];
            if (k > 0) yp[6 * j + k] = pdup(q[k]);
        }
    }
    const int r = threadIdx.x / CT;
    step_dependency_wait();
    __syncthreads();
    const int64_t c = blockIdx.x;
    const R *fr = f + c * m.Q;
    if (r < NR) {
        for (int cg = threadIdx.x % CT; cg < CG; cg += CT) {
            const ColPair cp(nv, cg);
            const R *m0x = static_cast<const R *>(m.m0) + cp.j;
            const P mx = pset(-m0x[0], -m0x[cp.n - 1]);
#pragma unroll
            for (int half = 0; half < 2; half++) {
                int lo, hi;
                half_range(nv, half, lo, hi);
                P a[5];
#pragma unroll
                for (int k = 0; k < 5; k++) a[k] = pdup(R(0));
                auto add = [&](int i, P fv, R wt) {
                    P y[6];
                    load_rows<R, 6>(reinterpret_cast<const R *>(yp + 6 * i), y);
                    P d = pfma(mx, y[0], fv);
                    if (wt != R(1)) d = pmul(pdup(wt), d);
                    a[0] = pfma(pdup(R(1)), d, a[0]);
#pragma unroll
                    for (int k = 1; k < 5; k++) a[k] = pfma(y[k], d, a[k]);
                };
                const R *q = fr + (lo + r) * nv + cp.j;
                int i = lo + r;
                // five rows' loads ahead of their sums
                for (; i + 4 * NR < hi; i += 5 * NR, q += 5 * NR * nv) {
                    P v[5];
#pragma unroll
                    for (int u = 0; u < 5; u++) v[u] = pload<R, ALIGNED>(q + u * NR * nv, cp.n);
#pragma unroll
                    for (int u = 0; u < 5; u++) add(i + u * NR, v[u], R(1));
                }
                for (; i < hi; i += NR, q += NR * nv) add(i, pload<R, ALIGNED>(q, cp.n), R(1));
                if ((nv & 1) && r == 0) add(nv / 2, pload<R, ALIGNED>(fr + (nv / 2) * nv + cp.j, cp.n), R(0.5));
#pragma unroll
                for (int k = 0; k < 5; k++) pstore<R, false>(&S[((half * NR + r) * 5 + k) * nv + cp.j], a[k], cp.n);
            }
        }
    }
    __syncthreads();
    // rows' slices together
    for (int t = threadIdx.x; t < 10 * nv; t += blockDim.x) {
        const int half = t >= 5 * nv, q = t - half * 5 * nv;
        R *const p = S + half * NR * 5 * nv + q;
        R s = p[0];
        for (int k = 1; k < NR; k++) s += p[k * 5 * nv];
        p[0] = s;
    }
    __syncthreads();
    // quadrant moments: four lanes share a moment's columns
    const int t = min((int)threadIdx.x >> 2, 59), u = threadIdx.x & 3;
    const int qd = t / NMOM, k = t % NMOM, sx = qd & 1, sy = qd >> 1;
    const int n = k < 1 ? 0 : k < 3 ? 1 : k < 6 ? 2 : k < 10 ? 3 : 4, b = k - n * (n + 1) / 2, a = n - b;
    const R s = half_sum<R>(S + (sy * NR * 5 + b) * nv, xp + a * nv, nv, sx, u);
    if (threadIdx.x < 240 && u == 0) mom[c * 60 + t] = s;
}

// Directions of the neighbour table: 0 E, 1 W, 2 N, 3 S.
// Half-range moment (velocities of sign `pos` along axis ax) of fbar+ of a cell.
template <class R>
__device__ __forceinline__ R half_moment(const R *__restrict__ mom, int c, int ax, int pos, int k)
{
    const R *q = mom + (int64_t)c * 60 + k;
    return ax == 0 ? q[pos * NMOM] + q[(pos + 2) * NMOM] : q[(2 * pos) * NMOM] + q[(2 * pos + 1) * NMOM];
}

// Moment (a, b) of the reconstruction from cell c through its face in the direction of
// sign `pos` along axis ax, over the velocities that go that way.
template <class R>
__device__ __forceinline__ R face_moment(const DvmCart &m, const R *__restrict__ mom, int c, int ax, int pos, int a, int b)
{
    const int32_t *nb = m.nb + 4 * c;
    auto M = [&](int cell, int da, int db) { return half_moment<R>(mom, cell, ax, pos, mono(a + da, b + db)); };
    auto diff = [&](int axis, int da, int db) {          // central, or twice the one-sided difference
        const int p = nb[2 * axis], q = nb[2 * axis + 1];
        const R d = M(p >= 0 ? p : c, da, db) - M(q >= 0 ? q : c, da, db);
        return p >= 0 && q >= 0 ? d : d + d;
    };
    const DvmCartK<R> &K = consts<R>(m);
    const R hn = ax == 0 ? K.kh[0] : K.kh[1], dn = ax == 0 ? K.kdt[0] : K.kdt[1], dtt = ax == 0 ? K.kdt[1] : K.kdt[0];
    const int na = ax == 0 ? 1 : 0, nbb = ax == 0 ? 0 : 1;
    return M(c, 0, 0) + (pos ? hn : -hn) * diff(ax, 0, 0) - dn * diff(ax, na, nbb) - dtt * diff(1 - ax, nbb, na);
}

// ---- interface states, macroscopic fluxes, W^{n+1} and the tables of exponentials.
// One warp per face (E, W, N, S) of the cell; a face is evaluated by both of its cells with the
// same operands in the same order.
template <class R>
__global__ void __launch_bounds__(STATE_THREADS) k_dvc_states(const DvmCart m, const R *__restrict__ mom,
                                                             double *__restrict__ W, R *__restrict__ face_tab,
                                                             R *__restrict__ tab)
{
    extern __shared__ __align__(16) unsigned char dyn[];
    const int nv = m.nv;
    R *const x = reinterpret_cast<R *>(dyn);
    __shared__ double flux[4][4];             // macroscopic fluxes, outward, less the reference's
    const DvmCartK<R> &K = consts<R>(m);
    __shared__ Maxwell<R> par;
    for (int j = threadIdx.x; j < nv; j += blockDim.x) x[j] = static_cast<const R *>(m.vnode)[j];
    step_dependency_wait();
    __syncthreads();
    const int c = blockIdx.x, w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    {
        const int ax = w >> 1, out = !(w & 1);            // axis; the face lies on the cell's + side
        const int other = m.nb[4 * c + w];
        // moments of the axis' eight monomials (a along the axis, b across): from the lower
        // cell by lanes 0-7, from the upper by 8-15
        // (powers along 0 1 0 2 1 0 3 1, across 0 0 1 0 1 2 0 2, two bits each)
        const int k = lane & 7, upper = (lane >> 3) & 1;
        const int na = (0x7184 >> (2 * k)) & 3, nt = (0x8910 >> (2 * k)) & 3;
        const int a = ax == 0 ? na : nt, b = ax == 0 ? nt : na;
        const int cell = (upper != 0) == (out != 0) ? other : c;       // lower cell: c if the face is on its + side
        R v = R(0);
        if (lane < 16 && cell >= 0) v = face_moment<R>(m, mom, cell, ax, !upper, a, b);
        v += __shfl_xor_sync(0xffffffffu, v, 8);
        R d[8];
#pragma unroll
        for (int q = 0; q < 8; q++) d[q] = __shfl_sync(0xffffffffu, v, q);
        const R len = K.len[ax];
        R *ft = face_tab + ((int64_t)c * 4 + w) * tab_size(nv);
        if (other >= 0) {
            // {rho, n, t, E} of the interface: the reference's plus d
            const R *const m0 = K.m0f;
            const R r = m0[mono(0, 0)] + d[0], e = R(0.5) * ((m0[mono(2, 0)] + d[ax == 0 ? 3 : 5]) + (m0[mono(0, 2)] + d[ax == 0 ? 5 : 3]));
            const R mx = m0[mono(1, 0)] + d[ax == 0 ? 1 : 2], my = m0[mono(0, 1)] + d[ax == 0 ? 2 : 1];
            const R ir = R(1) / r, ux = mx * ir, uy = my * ir, RT = e * ir - R(0.5) * (ux * ux + uy * uy), iRT = R(1) / RT;
            const R pre = r * iRT * K.amp;
            const R beta = R(0.5) * iRT * (sizeof(R) == 4 ? R(1.4426950408889634) : R(1));
            // tables, and their sums of powers 1..3 along (n) and 0..2 across (t), less the reference's (whose
            // odd ones are zero): the fluxes below are small differences
            const R *const m0x = static_cast<const R *>(m.m0);
            R n1 = R(0), n2 = R(0), n3 = R(0), t0 = R(0), t1 = R(0), t2 = R(0);
            for (int j = lane; j < nv; j += 32) {
                const R xx = x[j], gx = gauss<R>(xx, ux, beta), gy = pre * gauss<R>(xx, uy, beta);
                ft[j] = gx;
                ft[tab_row(nv, j)] = gy;
                const R ex = gx - m0x[j], ey = gy - m0x[nv + j], gn = ax == 0 ? ex : ey, gt = ax == 0 ? ey : ex;
                const R x2 = xx * xx;
                n1 += xx * gn; n2 += x2 * gn; n3 += xx * x2 * gn;
                t0 += gt; t1 += xx * gt; t2 += x2 * gt;
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                n1 += __shfl_xor_sync(0xffffffffu, n1, o); n2 += __shfl_xor_sync(0xffffffffu, n2, o);
                n3 += __shfl_xor_sync(0xffffffffu, n3, o); t0 += __shfl_xor_sync(0xffffffffu, t0, o);
                t1 += __shfl_xor_sync(0xffffffffu, t1, o); t2 += __shfl_xor_sync(0xffffffffu, t2, o);
            }
            // moments of xi_n times (1, n, t, (n^2 + t^2) / 2): fbar's in d, the equilibrium's less the reference's
            const R N2 = K.m0s[ax][1], T0 = K.m0s[1 - ax][0], T2 = K.m0s[1 - ax][1];
            const R f1 = n1 * (T0 + t0), f2 = N2 * t0 + n2 * (T0 + t0), f3 = n1 * t1;
            const R f4 = R(0.5) * (n3 * (T0 + t0) + n1 * (T2 + t2));
            const R s = len * K.c, bb = K.b, sg = out ? s : -s;
            if (lane == 0) {
                flux[w][0] = to_f64<R>(sg * (d[1] + bb * f1));
                flux[w][ax == 0 ? 1 : 2] = to_f64<R>(sg * (d[3] + bb * f2));
                flux[w][ax == 0 ? 2 : 1] = to_f64<R>(sg * (d[4] + bb * f3));
                flux[w][3] = to_f64<R>(sg * (R(0.5) * (d[6] + d[7]) + bb * f4));
            }
        } else {
            // diffuse wall (Sec. III) on this side: rho_w = 1 + dw so that no mass passes.  The
            // flux is the reference's share (DvmWall.z) plus c times what leaves of fbar beyond
            // the reference and dw's: small terms, whose rounding, alike in every step, adds
            // up to little (taken as the difference of whole fluxes, it put u off by 7e-14)
            const DvmWall &wl = m.wall[w];
            const R sg = out ? R(1) : R(-1);
            const double dw = -(wl.rest + double(sg * d[1])) / wl.g[0];
            const R *gw = static_cast<const R *>(m.wall_tab) + (int64_t)w * 2 * nv;
            for (int j = lane; j < nv; j += 32) {
                ft[j] = gw[j];
                const double gy = (double)gw[nv + j];
                ft[tab_row(nv, j)] = (R)fma(dw, gy, gy);
            }
            if (lane < 4) {
                const R dn = d[3], dt_ = d[4];
                const R o = lane == 0 ? d[1] : lane == 3 ? R(0.5) * (d[6] + d[7]) : ((lane == 1) == (ax == 0) ? dn : dt_);
                flux[w][lane] = lane == 0 ? 0.0 : m.kd.len[ax] * (wl.z[lane] + m.kd.c * (double(sg * o) + dw * wl.g[lane]));
            }
        }
    }
    __syncthreads();
    if (threadIdx.x < 32) {
        const int k = lane & 3;
        const double w1 = W[4 * (int64_t)c + k] - m.kd.dtV * ((flux[0][k] + flux[1][k]) + (flux[2][k] + flux[3][k]));
        __syncwarp();
        if (lane < 4) W[4 * (int64_t)c + k] = w1;
        const Maxwell<R> p = warp_maxwell<R>(w1, K);
        if (lane == 0) par = p;
    }
    __syncthreads();
    cell_tables<R>(m, par, tab + (int64_t)c * tab_size(nv));
}

// ---- cell update.  A CTA takes velocities of one quadrant and marches along a line of cells, in
// x from the side the velocities come from; a thread owns a column and 2 RP rows of the
// velocity grid.  In the coordinates u, v of the march (the flow goes towards larger ones) the
// cell C = (u, v) needs phi of E (u + 1, v), N (u, v + 1), SE (u + 1, v - 1) and SS (u, v - 2) from memory; the
// cell behind and its neighbours, and the flux through the face behind, come along in
// registers.  So phi is read four times (256 MB a step on the 40 x 40 x 100^2 cavity) where the
// stencil of a cell by itself is ten reads.  A missing neighbour (wall) is extrapolated from the two
// cells before it, which makes the central difference the one-sided one.  The flux of a face
// is c l xi_n (fbar + b feq); a wall gives T with 1 / c in the place of b.
// Bound by latency: 124 registers, 14 warps per SM, half of a warp's wait on loads from L2
// (which move 44 % of their peak).  One pair of rows for a thread, at 64 registers, took
// 144 us a step where two take 90; 6 CTAs per SM 101; the loop unrolled twice 97.
// a value at a 32-bit offset in bytes
template <class T> __device__ __forceinline__ const T *at32(const T *p, uint32_t b)
{
    return reinterpret_cast<const T *>(reinterpret_cast<const char *>(p) + b);
}
template <class T> __device__ __forceinline__ T *at32(T *p, uint32_t b)
{
    return reinterpret_cast<T *>(reinterpret_cast<char *>(p) + b);
}
template <class R, int RP>
__global__ void __launch_bounds__(UPD_THREADS, sizeof(R) == 4 ? 8 : 6)
k_dvc_update(const DvmCart m, const R *__restrict__ fin, R *__restrict__ fout, const R *__restrict__ tab0,
             const R *__restrict__ tab1, const R *__restrict__ face_tab)
{
    using P = typename PairT<R>::T;
    extern __shared__ __align__(16) unsigned char dyn[];
    int *const line = reinterpret_cast<int *>(dyn);          // [4][seg + 3] cells of rows v - 2 .. v + 1; -1: none
    const int nv = m.nv, seg = m.seg, ls = seg + 3;
    const int qd = blockIdx.y & 3, px = qd & 1, py = qd >> 1, v = blockIdx.z;
    const int u0 = (int)(blockIdx.y >> 2) * seg, n = min(seg, m.nx - u0);
    for (int t = threadIdx.x; t < 4 * ls; t += blockDim.x) {
        int u = u0 - 2 + t % ls, w = v - 2 + t / ls;
        if (m.per_x) u = (u + 2 * m.nx) % m.nx;
        if (m.per_y) w = (w + 2 * m.ny) % m.ny;
        int c = -1;
        if (u >= 0 && u < m.nx && w >= 0 && w < m.ny) c = m.at[(px ? u : m.nx - 1 - u) + (int64_t)m.nx * (py ? w : m.ny - 1 - w)];
        line[t] = c;
    }
    const int ncol = px ? nv - nv / 2 : nv / 2, nrow = py ? nv - nv / 2 : nv / 2;
    const int t = blockIdx.x * blockDim.x + threadIdx.x, g = t / ncol, j = (px ? nv / 2 : 0) + t % ncol;
    const int i0 = (py ? nv / 2 : 0) + g * 2 * RP, left = nrow - g * 2 * RP;       // rows i0 .. i0 + min(2 RP, left)
    const DvmCartK<R> &K = consts<R>(m);
    const R *const x = static_cast<const R *>(m.vnode);
    __syncthreads();
    if (left <= 0) {
        step_dependency_wait();
        return;
    }
    const R ax = px ? x[j] : -x[j];
    const P Qx = pdup(-ax * K.kdt[0]), Ox = pdup(K.kh[0] - ax * K.kdt[0]);
    const R sx0 = ax * (K.len[0] * (K.dtV * K.c));
    P ay[RP];
    uint32_t off[2 * RP];                                    // bytes from the start of a cell
#pragma unroll
    for (int k = 0; k < RP; k++) {
        const int a = i0 + min(2 * k, left - 1), b = i0 + min(2 * k + 1, left - 1);
        off[2 * k] = (uint32_t)(a * nv + j) * (uint32_t)sizeof(R);
        off[2 * k + 1] = (uint32_t)(b * nv + j) * (uint32_t)sizeof(R);
        ay[k] = py ? pset(x[a], x[b]) : pset(-x[a], -x[b]);
    }
    const P dty = pdup(-K.kdt[1]), khy = pdup(K.kh[1]), two = pdup(R(2)), neg = pdup(R(-1));
    constexpr uint32_t rs = sizeof(R);
    const uint32_t tb = (uint32_t)tab_size(nv) * rs, ty = (uint32_t)(tab_y(nv) + py * tab_half(nv) + g * 2 * RP) * rs;
    const uint32_t jx = (uint32_t)j * rs, cb = (uint32_t)m.Q * rs;
    const R b_ = K.b;
    step_dependency_wait();

    auto load = [&](int c, P f[RP]) {                        // phi of a cell (c >= 0)
        const uint32_t b = (uint32_t)c * cb;
#pragma unroll
        for (int k = 0; k < RP; k++) f[k] = pset(*at32(fin, b + off[2 * k]), *at32(fin, b + off[2 * k + 1]));
    };
    auto add = [&](const R *tab, int c, R scale, P e[RP]) {  // plus scale times the Maxwellian of table c
        const uint32_t b = (uint32_t)c * tb;
        const P gx = pdup(scale * *at32(tab, b + jx));
        P gy[RP];
        load_rows<R, RP>(at32(tab, b + ty), gy);
#pragma unroll
        for (int k = 0; k < RP; k++) e[k] = pfma(gx, gy[k], e[k]);
    };
    auto beyond = [&](P a, P b) { return pfma(two, a, pmul(neg, b)); };        // 2 a - b
    const int *const l0 = line + 2 * ls + 2, *const lm = line + ls + 2, *const lmm = line + 2, *const lp = line + 3 * ls + 2;
    const bool hasS = lm[0] >= 0, hasN = lp[0] >= 0, hasSS = lmm[0] >= 0, hasW = l0[-1] >= 0;
    // face tables of a cell: E, W, N, S
    const int tE = px ? 0 : 1, tW = 1 - tE, tN = py ? 2 : 3, tS = 5 - tN;
    P W[RP], C[RP], S[RP], SW[RP], xi[RP];
    load(l0[0], C);
#pragma unroll
    for (int k = 0; k < RP; k++) { W[k] = SW[k] = S[k] = C[k]; xi[k] = pdup(R(0)); }
    if (hasS) {
        load(lm[0], S);
        if (hasW) load(lm[-1], SW);
    }
    if (hasW) {
        P WW[RP], NW[RP];
        load(l0[-1], W);
#pragma unroll
        for (int k = 0; k < RP; k++) WW[k] = beyond(W[k], C[k]);
        if (l0[-2] >= 0) load(l0[-2], WW);
        if (hasN) load(lp[-1], NW);
#pragma unroll
        for (int k = 0; k < RP; k++) {
            P d = pdup(R(0));
            if (hasN && hasS) d = psub(NW[k], SW[k]);
            else if (hasN) d = pmul(two, psub(NW[k], W[k]));
            else if (hasS) d = pmul(two, psub(W[k], SW[k]));
            xi[k] = pfma(pmul(dty, ay[k]), d, pfma(Ox, psub(C[k], WW[k]), W[k]));
        }
    }
    if (!hasW) add(face_tab, 4 * l0[0] + tW, R(1), xi);     // 1 / c = 1 + b: the ratio to the other faces unrounded
    add(face_tab, 4 * l0[0] + tW, b_, xi);
    P E[RP], N[RP], SE[RP], SS[RP], nE[RP], nN[RP], nSE[RP], nSS[RP];
    const R s0 = -(K.inv1r * K.b), s1 = K.a * K.r * K.inv1r + K.b;
    // phi^{n+1} as a change of phi: the coefficients add up to 1 without a rounding of 1 / (1 + r).  An
    // error that acts alike in every step does not average out: with it, and with 1 / c and the
    // wall's density rounded for the fluxes of walls, u was off by 9.1e-6 after 200 steps of a
    // 20 x 20 x 100^2 cavity at Kn = 2; now 5.5e-7 (k_dvm.cu 1.5e-6).
    const P m1 = pdup(-(K.r * K.inv1r)), fx = pdup(-(K.inv1r * K.a) * sx0), fy = pdup(-(K.inv1r * K.a) * (K.len[1] * (K.dtV * K.c)));
    auto march = [&](auto inside) {                          // inside: the lines around the line are there
        constexpr bool IN = decltype(inside)::value;
        const bool N_ = IN || hasN, S_ = IN || hasS, SS_ = IN || hasSS;
        auto fetch = [&](int i) {
            const bool e = l0[i + 1] >= 0;
            if (e) load(l0[i + 1], nE);
            if (N_) load(lp[i], nN);
            if (S_ && e) load(lm[i + 1], nSE);
            if (SS_) load(lmm[i], nSS);
        };
        fetch(0);
#pragma unroll 1
        for (int i = 0; i < n; i++) {
            const int c = l0[i];
            const bool hasE = l0[i + 1] >= 0;
#pragma unroll
            for (int k = 0; k < RP; k++) { E[k] = nE[k]; N[k] = nN[k]; SE[k] = nSE[k]; SS[k] = nSS[k]; }
            if (i + 1 < n) fetch(i + 1);
            P xo[RP], yo[RP], yi[RP], r[RP];
#pragma unroll
            for (int k = 0; k < RP; k++) { xo[k] = C[k]; yo[k] = C[k]; yi[k] = S_ ? S[k] : pdup(R(0)); r[k] = pmul(m1, C[k]); }
            add(face_tab, 4 * c + tE, b_, xo);
            add(face_tab, 4 * c + tN, b_, yo);
            if (!S_) add(face_tab, 4 * c + tS, R(1), yi);
            add(face_tab, 4 * c + tS, b_, yi);
            add(tab0, c, s0, r);
            add(tab1, c, s1, r);
            if (!hasE) {
#pragma unroll
                for (int k = 0; k < RP; k++) { E[k] = beyond(C[k], W[k]); SE[k] = beyond(S[k], SW[k]); }
            }
            if (i == 0 && !hasW) {
#pragma unroll
                for (int k = 0; k < RP; k++) { W[k] = beyond(C[k], E[k]); SW[k] = beyond(S[k], SE[k]); }
            }
            if (!N_) {
#pragma unroll
                for (int k = 0; k < RP; k++) N[k] = beyond(C[k], S[k]);
            }
            if (!S_) {
#pragma unroll
                for (int k = 0; k < RP; k++) { S[k] = beyond(C[k], N[k]); SE[k] = E[k]; }
            }
            if (!SS_) {
#pragma unroll
                for (int k = 0; k < RP; k++) SS[k] = beyond(S[k], C[k]);
            }
            const uint32_t b = (uint32_t)c * cb;
#pragma unroll
            for (int k = 0; k < RP; k++) {
                const P Qy = pmul(dty, ay[k]), Oy = pfma(dty, ay[k], khy);
                const P dx = psub(E[k], W[k]), dy = psub(N[k], S[k]);
                xo[k] = pfma(Qy, dy, pfma(Ox, dx, xo[k]));
                yo[k] = pfma(Oy, dy, pfma(Qx, dx, yo[k]));
                if (S_) yi[k] = pfma(Oy, psub(C[k], SS[k]), pfma(Qx, psub(SE[k], SW[k]), yi[k]));
                r[k] = pfma(fx, psub(xo[k], xi[k]), pfma(pmul(fy, ay[k]), psub(yo[k], yi[k]), r[k]));
                r[k] = pfma(pdup(R(1)), C[k], r[k]);
                if (2 * k < left) *at32(fout, b + off[2 * k]) = r[k].x;
                if (2 * k + 1 < left) *at32(fout, b + off[2 * k + 1]) = r[k].y;
                xi[k] = xo[k];
                W[k] = C[k]; C[k] = E[k]; SW[k] = S[k]; S[k] = SE[k];
            }
        }
    };
    if (hasN && hasS && hasSS) march(std::true_type{});
    else march(std::false_type{});
}

template <class R> size_t mom_smem(int nv)
{
    const int CG = col_pairs(nv), CT = CG < MOM_THREADS ? CG : MOM_THREADS, NR = MOM_THREADS / CT;
    return sizeof(R) * ((size_t)17 * nv + (size_t)2 * NR * 5 * nv);
}
template <class R> constexpr int upd_pairs() { return sizeof(R) == 4 ? 2 : 1; }
size_t upd_smem(int seg) { return sizeof(int) * 4 * (size_t)(seg + 3); }
template <class R> size_t state_smem(int nv) { return sizeof(R) * (size_t)nv; }

template <class R, bool ALIGNED> cudaError_t prepare_v(int nv)
{
    cudaError_t e = cudaFuncSetAttribute(k_dvc_moments<R, ALIGNED>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)mom_smem<R>(nv));
    return e;
}

template <class R, bool ALIGNED>
cudaError_t step_v(const DvmCart &m, const DvmCartState &s, int par, cudaStream_t st)
{
    const R *fin = static_cast<const R *>(s.phi[par]);
    R *fout = static_cast<R *>(s.phi[1 - par]), *mom = static_cast<R *>(s.mom);
    const R *tab0 = static_cast<const R *>(s.tab[par]), *cmom = mom;
    R *tab1 = static_cast<R *>(s.tab[1 - par]), *ft = static_cast<R *>(s.face_tab);
    const R *ctab1 = tab1, *cft = ft;
    const dim3 cells((unsigned)m.nc);
    const int nv = m.nv;
    cudaError_t e = launch_step_kernel(true, k_dvc_moments<R, ALIGNED>, cells, dim3(MOM_THREADS), mom_smem<R>(nv), st, m, fin, mom);
    if (e == cudaSuccess)
        e = launch_step_kernel(true, k_dvc_states<R>, cells, dim3(STATE_THREADS), state_smem<R>(nv), st, m, cmom, s.W, ft, tab1);
    if (e == cudaSuccess)
        e = launch_step_kernel(true, k_dvc_update<R, upd_pairs<R>()>, dim3((unsigned)m.chunks, 4u * ((m.nx + m.seg - 1) / m.seg), (unsigned)m.ny),
                               dim3(UPD_THREADS), upd_smem(m.seg), st, m, fin, fout, tab0, ctab1, cft);
    return e;
}

template <class R> cudaError_t step_p(const DvmCart &m, const DvmCartState &s, int par, cudaStream_t st)
{
    return m.nv % 4 == 0 ? step_v<R, true>(m, s, par, st) : step_v<R, false>(m, s, par, st);
}

}  // namespace

// Small solves stay with k_dvm.cu, whose two or three launches are shorter than these three: with
// its 16-byte vectors (nv a multiple of 4) up to 2^18 values of f in FP32 (16 x 16 x 20^2: 8.4 us
// a step, here 11.0; 16 x 16 x 32^2: 10.1 / 10.6; 30 x 30 x 20^2: 19.9 / 16.7) and 2^15 in FP64 (10 x 10 x 16^2:
// 32 / 36; 14 x 14 x 16^2: 44 / 33), otherwise up to 2^16 (12 x 12 x 18^2: 9.1 / 10.0; 16 x 16 x 33^2: 16.1 / 12.8)
// and 2^14 (8 x 8 x 17^2: 48 / 43).
bool dvm_cart_fits(int prec, int64_t nc, int nv, int ny)
{
    const int64_t values = nc * nv * nv, rs = prec == P_FP64 ? 8 : 4;
    const int64_t least = (int64_t)1 << (nv % 4 == 0 ? (prec == P_FP64 ? 15 : 18) : (prec == P_FP64 ? 14 : 16));
    // 32-bit byte offsets
    const int64_t cell = std::max<int64_t>((int64_t)nv * nv, 4 * tab_size(nv)) * rs;
    return values > least && nc * cell < ((int64_t)1 << 32) && ny <= 65535 &&
           (prec == P_FP64 ? mom_smem<double>(nv) : mom_smem<float>(nv)) <= 100 * 1024;
}

size_t dvm_cart_table(int nv) { return (size_t)tab_size(nv); }

// The march's split: the length of a segment of a line, the one with the least (waves of CTAs) x (cells
// of a segment + 2 for its start): 20 on the 40 x 40 x 100^2 cavity (98 us a step; 102 with 10, 106 with
// 8), 6 on 23 x 23 x 50^2 (18.9; 20.6 with 3, 21.1 with 8).
template <class R> cudaError_t split_march(DvmCart &m)
{
    constexpr int RP = upd_pairs<R>();
    const int hv = m.nv - m.nv / 2, threads = hv * ((hv + 2 * RP - 1) / (2 * RP));
    m.chunks = (threads + UPD_THREADS - 1) / UPD_THREADS;
    int dev = 0, n_sm = 1, per = 1;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_dvc_update<R, RP>, UPD_THREADS, upd_smem(64));
    if (e != cudaSuccess) return e;
    const int64_t slots = (int64_t)n_sm * std::max(per, 1), ctas = (int64_t)m.chunks * 4 * m.ny;
    int64_t least = 0;
    for (int k = 1; k <= m.nx && k <= 4096; k++) {
        const int seg = (m.nx + k - 1) / k;
        if (seg > 1024) continue;
        const int64_t waves = (ctas * ((m.nx + seg - 1) / seg) + slots - 1) / slots, cost = waves * (seg + 2);
        if (least == 0 || cost < least) { least = cost; m.seg = seg; }
    }
    return cudaSuccess;
}

cudaError_t prepare_dvm_cart(int prec, DvmCart &m)
{
    cudaError_t e = prec == P_FP64 ? (m.nv % 4 == 0 ? prepare_v<double, true>(m.nv) : prepare_v<double, false>(m.nv))
                                   : (m.nv % 4 == 0 ? prepare_v<float, true>(m.nv) : prepare_v<float, false>(m.nv));
    if (e == cudaSuccess) e = prec == P_FP64 ? split_march<double>(m) : split_march<float>(m);
    return e;
}

cudaError_t launch_dvm_cart_init(int prec, const DvmCart &m, const DvmCartState &s, cudaStream_t st)
{
    if (prec == P_FP64)
        k_dvc_init<double><<<(unsigned)m.nc, STATE_THREADS, 0, st>>>(m, s.W, static_cast<double *>(s.phi[0]), static_cast<double *>(s.tab[0]));
    else
        k_dvc_init<float><<<(unsigned)m.nc, STATE_THREADS, 0, st>>>(m, s.W, static_cast<float *>(s.phi[0]), static_cast<float *>(s.tab[0]));
    return cudaGetLastError();
}

cudaError_t launch_dvm_cart_f(int prec, const DvmCart &m, const DvmCartState &s, int par, cudaStream_t st)
{
    if (prec == P_FP64)
        k_dvc_f<double><<<(unsigned)m.nc, STATE_THREADS, 0, st>>>(m, static_cast<const double *>(s.phi[par]),
                                                                 static_cast<const double *>(s.tab[par]), static_cast<double *>(s.phi[1 - par]));
    else
        k_dvc_f<float><<<(unsigned)m.nc, STATE_THREADS, 0, st>>>(m, static_cast<const float *>(s.phi[par]),
                                                                static_cast<const float *>(s.tab[par]), static_cast<float *>(s.phi[1 - par]));
    return cudaGetLastError();
}

cudaError_t launch_dvm_cart_step(int prec, const DvmCart &m, const DvmCartState &s, int par, cudaStream_t st)
{
    return prec == P_FP64 ? step_p<double>(m, s, par, st) : step_p<float>(m, s, par, st);
}

}  // namespace sdugks
