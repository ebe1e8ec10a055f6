// sdugks_internal.h -- launch interface between the host library (sdugks_host.cpp)
// and the CUDA translation units.  Plain structs of device pointers and sizes.
#pragma once
#include <cstdint>
#include <cuda.h>
#include <cuda_runtime.h>

namespace sdugks {

constexpr int NQ = 9;
constexpr int MAXF = 4;         // faces per cell (quads and triangles)
constexpr int MAXPATCH = 64;    // boundary patches
constexpr uint16_t NO_LOCAL = 0xFFFF;
// LLSR neighbour codes of a symmetry slot: the mirror image of the cell itself in a
// line of constant x (SYM_X) or constant y (SYM_Y)
constexpr uint16_t SYM_X = 0xFFFD, SYM_Y = 0xFFFE;

// Tiled kernel shape: one CTA per tile of up to TILE_MAX cells.
constexpr int TILE_MAX = 128;   // interior cells per tile
constexpr int TILED_THREADS = 256;
constexpr int LOC_MAX = 416;    // interior + two halo rings
constexpr int SIG_MAX = 272;    // interior + first halo ring (cells whose gradient is needed)
constexpr int LF_MAX = 320;     // faces with at least one interior cell of the tile

enum Prec : int32_t { P_FP64 = 0, P_FP32 = 1, P_BF16DEV = 2, P_FP16DEV = 3 };

enum BcKind : int32_t { BK_UNSET = 0, BK_PERIODIC = 1, BK_WALL = 2, BK_MOVING_WALL = 3,
                        BK_FARFIELD = 4, BK_OUTLET = 5, BK_SYMMETRY = 6 };

// Scalars of one step (host-computed in FP64 from tau and dt; FP32 copies for the
// FP32-compute kernels so that no thread converts them).
struct Coefs {
    double a_plus;   // (2 tau - dt) / (2 tau)
    double b_plus;   // dt / (2 tau)
    double c_face;   // 2 tau / (2 tau + dt)
    double r;        // dt / tau
    double inv1r;    // 1 / (1 + dt / tau)
    double dt;
    double tie;      // |xi . n l| <= tie counts as tangential
    float fa_plus, fb_plus, fc_face, fr, finv1r, fdt, ftie, fpad_;
    int32_t bc_kind[MAXPATCH];
    double bc_par[MAXPATCH][3];
    float fbc_par[MAXPATCH][3];
    float fbc_drho[MAXPATCH];     // rho_inf - 1 of far-field patches (FP32 compute works with rho - 1)
};

// Slot kinds of a cell's faces (slots in ascending face id).
constexpr uint8_t SK_NONE = 0xFE;      // cell has fewer faces than MAXF
constexpr uint8_t SK_INTERIOR = 0xFF;  // face shared with another cell (periodic pairs included)
                                       // any other value: boundary patch id

// Unstructured tiled mesh on the device.  Cells are in internal (tile-contiguous)
// order; arrays indexed by cell are padded to npad.  Each tile lists the faces that
// touch its interior cells ("local faces", evaluated once per tile), oriented from
// their first side (the face owner) to the second.
struct TiledMesh {
    int32_t n_tiles;
    int64_t n, npad;
    int64_t n_lf;             // local faces of all tiles with the padding (stride of lf_geo, a multiple of 4)
    const int32_t *tile_c0;   // [n_tiles+1] interior cell range of each tile
    const int32_t *tile_h0;   // [n_tiles+1] range into halo
    const int32_t *tile_nh1;  // [n_tiles]   cells of ring 1 (first in the tile's halo)
    const int32_t *tile_s0;   // [n_tiles+1] range into sig_nb (each tile's rows padded to a multiple of 4)
    const int32_t *tile_f0;   // [n_tiles+1] first local face of each tile, a multiple of 4 (the
                              //   ranges are padded so that each starts 16-byte aligned)
    const int32_t *tile_nlf;  // [n_tiles] local faces of each tile (the rest of its range is padding)
    const int32_t *halo;      // internal ids of ring 1 then ring 2 of each tile
    int64_t n_sig;            // gradient rows of all tiles (stride of sig_d and sig_ai)
    const uint16_t *sig_nb;   // [n_sig][MAXF] tile-local index of the cell across each slot
    const void *sig_d;        // [MAXF][2][n_sig] x_k - x_j across each slot of each gradient row
    const void *sig_ai;       // [3][n_sig] LLSR inverse (xx, xy, yy) of each gradient row
    const uint16_t *cell_lf;  // [MAXF][npad] local face of each slot, | LF_SECOND when the cell
                              //   is the face's second side; LF_NONE for no face
    const uint32_t *lf_ab;    // [n_lf] tile-local first side | second side << 16; a boundary
                              //   face's second side is LF_BOUNDARY | patch
    const void *lf_geo;       // [6][n_lf] n l from the first side to the second (2),
                              //   x_f - x_first (2), x_f - x_second (2)
    const void *dtV;          // [npad] dt / V (compute precision)
    const double *vol;        // [npad] V
    double *force;            // nullptr, or [MAXPATCH][2]: momentum flux out of the fluid per boundary patch
    const int32_t *lf_bface;  // [n_lf] boundary-face row of each local face (-1: interior or periodic)
    double *bface;            // nullptr, or [n_bfaces][2]: momentum flux out of the fluid per boundary face
    bool early;               // launches allow the early start (early_start)
};
constexpr uint16_t LF_SECOND = 0x8000, LF_NONE = 0xFFFF;
constexpr uint32_t LF_BOUNDARY = 0xC000;

// One uniform-grid solve as the Cartesian kernels see it: nx x ny rectangles
// dx x dy, cell (i, j) at i + pitch j; side boundary rules; step coefficients; and
// its ping-pong state f[2] ([NQ][npad]), W[2] ([3][npad] FP64).  Buffer p holds
// t_n when the launch parity is p.
struct CartInst {
    int32_t nx, ny, pitch, periodic_x, periodic_y;
    int32_t side_kind[4];     // BK_* of the bottom, right, top, left side (unused if periodic)
    int32_t item0, n_items;   // batched runs: this instance's range in the work list
    int64_t npad;             // >= pitch * ny, multiple of 32
    double dx, dy, dtV;       // dtV = dt / (dx dy)
    double ihx, ihy;          // 1 / dx, 1 / dy
    double a, b, c, r, dt;    // (2tau-dt)/2tau, dt/2tau, 2tau/(2tau+dt), dt/tau, dt
    double side_par[4][3];
    float fdx, fdy, fdtV, fa, fb, fc, fr, finv1r, fdt, fihx, fihy;
    float fside_par[4][3];
    float fside_drho[4];      // rho_inf - 1 of far-field sides (FP32 compute works with rho - 1)
    void *f[2];
    double *W[2];
    double *snap;             // [2][npad] residual snapshot (U0, V0)
    double *force;            // nullptr, or [4][2]: momentum flux out of the fluid per grid side
    int32_t *err;             // nullptr, or a device flag set to 1 when a bounded staging wait gave up
    uint64_t tma_wait_ns;     // TMA staging: wait limit of a block's copies (0: give up at once)
    const int32_t *bidx;      // [2 (nx + ny)] boundary-face row of each side face: bottom (by i), right
                              //   (by j), top (by i), left (by j); -1 on periodic sides
    double *bface;            // nullptr, or [n_bfaces][2]: momentum flux out of the fluid per boundary face
    int64_t early;            // launches allow the early start (early_start)
};

// Device state of one solver, ping-pong: f [2][NQ][npad] (element type by
// precision), W [2][3][npad] FP64.
struct State {
    void *f[2];
    double *W[2];
};

// fused step kernels (k_step_fp64.cu, k_step_fp32.cu); prepare_* sets the kernel
// attributes on the current device and is called once per solver creation
cudaError_t prepare_tiled_fp64();
cudaError_t launch_step_tiled_fp64(const TiledMesh &m, const Coefs &c, const void *f_in, void *f_out,
                                   const double *W_in, double *W_out, cudaStream_t st);
cudaError_t prepare_tiled_fp32(int prec);
int occ_tiled_fp64();
int occ_tiled_fp32(int prec);                              // resident tiles per SM
cudaError_t prepare_cart(int prec);
// block shapes of the FP32-compute Cartesian kernel: 0 = 16x16, 1 = 16x14, 2 = 16x8
constexpr int CART_SHAPES = 3;
// block of the batched kernel: 16 x BATCH_TY cells per (instance, block) work item (the
// 16x8 shape fits four CTAs per SM, the fastest shape of the single-solve kernel on
// grids of many waves)
constexpr int BATCH_TY = 8;
constexpr int CART_TY[CART_SHAPES] = {16, 14, 8};
// Tensor maps of one Cartesian state for the TMA staging of interior blocks:
// f[b] views f buffer b as (x, y, velocity), W[b] views W buffer b as (x, y, component);
// the boxes are the block with its two-cell halo, widened in x to 16-byte boundaries.
struct CartTma {
    CUtensorMap f[2], W[2];
};
cudaError_t make_cart_tma(int prec, int shape, const CartInst &m, CartTma &out);
// tma: nullptr stages every block with plain loads; general: every block on the general
// code path (no interior variant; ignored with TMA staging)
cudaError_t launch_step_cart(int prec, int shape, const CartInst &m, const CartTma *tma, bool general, int parity,
                             cudaStream_t st);
int cart_shape_occupancy(int prec, int shape, bool tma);   // resident CTAs per SM
// FP64: blocks of 16x14, 8x8 or 4x4 cells (shape 0, 1, 2), by grid size; 16x16 with TMA staging
cudaError_t prepare_cart64();
cudaError_t launch_step_cart64_tma(const CartInst &m, const CartTma &tma, int parity, cudaStream_t st);
cudaError_t launch_step_cart64(const CartInst &m, int shape, int parity, cudaStream_t st);
int cart64_shape(int nx, int ny, int n_sm);
constexpr int CART64_BLOCK[3][2] = {{16, 14}, {8, 8}, {4, 4}};
// One uniform-grid solve as the marching form and its block form see it (FP32 storage; no
// symmetry side, an even nx where x is periodic): the grid and its side rules, the ping-pong state, and
// the step's constants, each twice (one operand of a paired instruction).
struct StripInst {
    int32_t nx, ny, pitch, npad, periodic_x, periodic_y;
    int32_t side_kind[4];
    float side_par[4][3], side_drho[4];
    float sb, sc, len_dtV[2];                  // b, c; lengths of faces of constant x, y times dt / V
    float *f[2];
    double *W[2];
    float2 b, ri;                              // ri = r / (1 + r)
    float2 g[2], bg[2];                        // faces of constant x, y: c len dt/V, b c len dt/V
    float2 xdt[2], xh[2], xo[2];               // dt, h/2, h/2 - dt along x, times 1/(2 dx); [1] negated
    float2 ydt[2], yh[2], yo[2];
};
bool strip_fits(const CartInst &m, int prec);                // the marching form takes this solve
void fill_strip(const CartInst &m, StripInst &s);
int strip_count(int nx, bool periodic_x);                    // 60-column strips of a grid
// rows per warp for a set of grids (strips x rows, as counted by `items(rows)`) that fill
// `slots` resident warps best, and the model's time of a step in row units
template <class Items> inline int strip_rows(int64_t slots, int max_ny, Items &&items, double &cost)
{
    // A range of rows costs rows + 2 units (two rows' worth for its halo and its start).
    // A step is half whole waves, half work that fills the slots evenly: with items / slots
    // = r, (rows + 2) (ceil(r) + max(1, r)) / 2.  Fits 40 measured (size, rows) pairs from
    // 448^2 to 2048^2 within 6 % at 1.8 to 2.1 us a unit (GB300).
    int best = 0;
    cost = 1e300;
    for (int rows = 1; rows <= max_ny && rows <= 256; rows += 1 + rows / 16) {
        if ((max_ny + rows - 1) / rows > 32767) continue;
        const double r = (double)items(rows) / (double)slots;
        const double c = (rows + 2) * 0.5 * ((double)(int64_t)(r + 0.999999) + (r > 1.0 ? r : 1.0));
        if (c < cost) { cost = c; best = rows; }
    }
    return best;                               // 0: no range fits
}
cudaError_t prepare_strip();
cudaError_t launch_step_strip(const StripInst &s, int rows, bool early, int parity, cudaStream_t st);
int strip_slots();                                           // resident warps of the device
// batched: a group of instances, handed to the kernel by value (constant memory), and its
// (instance of the group, strip | range << 16) items in device memory, one warp each
constexpr int STRIP_GROUP = 96;
struct StripGroup {
    StripInst inst[STRIP_GROUP];
};
static_assert(sizeof(StripGroup) <= 32000, "a group is a kernel parameter");
cudaError_t prepare_strip_batch();
cudaError_t launch_strip_batch(const StripGroup &g, const int2 *items, int n_items, int rows, bool early, int parity,
                               cudaStream_t st);
// by blocks of 16 x BATCH_TY cells, one CTA per (instance, block) item, the records in device
// memory: the same bits as the marching warps.  wide: for lists within strip_block_slots(true)
cudaError_t launch_strip_blocks(const StripInst *insts, const int2 *items, int n_items, bool wide, bool early, int parity,
                                cudaStream_t st);
int strip_block_slots(bool wide);                            // resident CTAs of the device
// batched: every (instance, tile) item of the list, one per CTA (per_item: grid >= the
// item count) or grid-stride over a fixed grid
cudaError_t prepare_batch(int prec);
cudaError_t launch_step_batch(int prec, const CartInst *insts, const int2 *items, const int *n_items, int grid,
                              bool per_item, int parity, cudaStream_t st);
int batch_ctas_per_sm(int prec);
// batched residual: partial [max_items][4] per tile, out [n_inst][4] = (num, den, mass, non-finite)
cudaError_t launch_batch_residual(const CartInst *insts, int n_inst, const int2 *items, const int *n_items, int grid,
                                  int parity, double *partial, double *out, cudaStream_t st);
cudaError_t launch_batch_init(int prec, const CartInst *inst_host, const CartInst *inst_dev, int parity,
                              const double *rho, const double *u, cudaStream_t st);
cudaError_t launch_batch_macros(const CartInst *inst_host, const CartInst *inst_dev, int parity, double *rho, double *u,
                                cudaStream_t st);
cudaError_t launch_step_tiled_fp32(int prec, const TiledMesh &m, const Coefs &c, const void *f_in, void *f_out,
                                   const double *W_in, double *W_out, cudaStream_t st);

// Programmatic dependent launch of the step kernels: each step kernel lets the next
// launch in its stream be scheduled as soon as all of its CTAs are running
// (griddepcontrol.launch_dependents) and, before it touches memory that a step
// writes, waits until the previous grid has completed and its writes are visible
// (griddepcontrol.wait; a no-op when the launch did not allow an early start); what
// only the host writes (mesh data, work items) may be read before the wait.  The
// next step's CTAs therefore take the SM slots the moment the current step's CTAs
// retire, instead of after the launch latency.
//
// The early start suits grids whose fullest SM holds as many CTAs as fit anyway (more than
// all SMs' slots but one each), whose next CTAs take over slot by slot, and grids of a few CTAs.
// In between, the next step's CTAs are placed while the current ones still run, wherever there
// is room, and pile up on some SMs: the step then lasts as long as the fullest SM.  GB300, us
// per step with / without: 169 tiles of 608 slots 8.2 / 6.1, 441 tiles 8.45 / 8.07, 484 tiles 8.2 / 8.75,
// 1024 tiles 13.3 / 14.0; 4x1024 channel (128 blocks of 608) 4.1 / 3.1, 4x256 channel (19 blocks)
// 3.44 / 3.53; bf16 cavities of 144 blocks in 304 slots 4.52 / 4.46, 169 blocks 4.49 / 4.59, 196 blocks
// 4.50 / 4.68.  These are steps of a graph.  Launched one by one, a step without the early start takes
// 6.2 us at least (361 tiles 10.3), and with it 4.1 (8.8): it then always has it.
inline bool early_start(int64_t ctas, int64_t slots, int n_sm) { return 4 * ctas <= n_sm || ctas > slots - n_sm; }

#ifdef __CUDACC__
__device__ __forceinline__ void step_dependency_wait()
{
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
}

// early: allow the programmatic early start (see early_start)
template <class... P, class... A>
cudaError_t launch_step_kernel(bool early, void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st,
                               A &&...args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = early ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<A &&>(args)...);
}
#endif

// Rarefied solver on a discrete velocity grid (Q nodes): any face-based mesh, f and
// the scratch arrays cell- (or face-) major with the Q velocities contiguous.
struct DvmMesh {
    int64_t nc, nf, Q;
    const int32_t *cell_face;  // [nc][MAXF] face id, | DVM_SECOND when the cell is the face's
                               //   second side; -1 for no face
    const int32_t *cell_nb;    // [nc][MAXF] LLSR neighbour (periodic partners included), -1 none
    const void *cell_d;        // [nc][MAXF][2] x_k - x_j (compute precision)
    const void *ainv;          // [nc][3] LLSR inverse (xx, xy, yy)
    const double *dtV;         // [nc] dt / V
    const int32_t *face_own, *face_nbr;   // face_nbr: cell, or -1 - patch
    const void *face_geo;      // [nf][6] n l (first -> second side), x_f - x_first, x_f - x_second
    // velocity q = j + nv i (x fastest) sits at (vnode[j], vnode[i]) with weight w_node
    const void *vnode;         // [nv] nodes of one axis (compute precision)
    int32_t nv;
    double w_node;
};
constexpr int32_t DVM_SECOND = int32_t(0x40000000);
constexpr int DVM_THREADS = 256;
// one step; fbp_ready: fbp already holds this step's fbar+ (left there by the previous
// step's cell kernel), else it is formed first.  The step leaves the next step's fbar+ in fbp.
cudaError_t launch_dvm_step(int prec, const DvmMesh &m, const Coefs &c, double RTw, void *f, double *W, void *fbp,
                            void *flux, bool fbp_ready, cudaStream_t st);
cudaError_t launch_dvm_init(int prec, const DvmMesh &m, const double *W, void *f, cudaStream_t st);
cudaError_t prepare_dvm(int prec, int64_t Q, int nv);   // kernel attributes on the current device

// Rarefied solver on a uniform Cartesian grid (k_dvm_cart.cu).  A wall, from sums of xi_n
// (outward) times (1, x, y, (x^2 + y^2) / 2), with 1 + b = 1 / c:
struct DvmWall {
    double g[4];               // of its Maxwellian of unit density: b times over the leaving velocities plus
                               // 1 + b times over the entering ones
    double rest;               // g[0] plus the mass that leaves in the reference Maxwellian
    double z[4];               // c (leaving part of the reference + g) less the whole reference: the flux,
                               // less the reference's, for a cell that holds the reference
};
template <class R> struct DvmCartK {
    R amp, amp_l;              // node weight / (2 pi); what amp leaves out
    R a, b, c, r, inv1r, dtV;
    R len[2];                  // length of a face of constant x, y
    R kh[2], kdt[2];           // h / 2 and dt along x and y, times 1 / (2 h)
    R m0f[15], m0s[2][2];      // moments of the reference; of its factors along x and y (powers 0 and 2)
};
struct DvmCart {
    int32_t nc, nv, nx, ny, per_x, per_y;
    int32_t chunks, seg;       // the update: CTAs per line and quadrant, cells of a line per CTA
    int64_t Q;
    const int32_t *at;         // [ny][nx] cell of a lattice position
    const int32_t *nb;         // [nc][4] neighbour E, W, N, S; -1 a wall
    const void *vnode;         // [nv] nodes of one axis (compute precision)
    const void *m0;            // [2][nv] factors of the reference Maxwellian (x; y with the node weight)
    const void *wall_tab;      // [4][2][nv] factors of the wall Maxwellians of the E, W, N, S sides
    DvmCartK<double> kd;
    DvmCartK<float> kf;
    DvmWall wall[4];
};
struct DvmCartState {
    void *phi[2];              // [nc][Q] fbar+
    double *W;                 // [nc][4]
    void *tab[2];              // [nc][table] factors of feq(W)
    void *mom;                 // [nc][4][15] quadrant moments of fbar+
    void *face_tab;            // [nc][4][table] factors of the interface equilibria
};
bool dvm_cart_fits(int prec, int64_t nc, int nv, int ny);
size_t dvm_cart_table(int nv);          // values of one table
cudaError_t prepare_dvm_cart(int prec, DvmCart &m);
cudaError_t launch_dvm_cart_init(int prec, const DvmCart &m, const DvmCartState &s, cudaStream_t st);
// f of the state in phi[parity], into the other buffer
cudaError_t launch_dvm_cart_f(int prec, const DvmCart &m, const DvmCartState &s, int parity, cudaStream_t st);
cudaError_t launch_dvm_cart_step(int prec, const DvmCart &m, const DvmCartState &s, int parity, cudaStream_t st);

// state conversions between the caller's cell-major FP64 layout (user cell order)
// and the internal SoA layout: the q-th listed cell is user cell perm[q] stored at
// internal offset loc[q] (loc == nullptr: offset q).
cudaError_t launch_init_state(int prec, int64_t n, int64_t npad, const int32_t *perm, const int32_t *loc,
                              const double *rho, const double *u, void *f, double *W, cudaStream_t st);
cudaError_t launch_pack_state(int prec, int64_t n, int64_t npad, const int32_t *perm, const int32_t *loc, const void *f,
                              const double *W, double *f_out, double *W_out, cudaStream_t st);
cudaError_t launch_unpack_state(int prec, int64_t n, int64_t npad, const int32_t *perm, const int32_t *loc,
                                const double *f_in, const double *W_in, void *f, double *W, cudaStream_t st);
// rr: the density the stored W[0] is measured from (rho = rr + W[0]; 0 for FP64, 1 for
// the FP32-compute precisions)
cudaError_t launch_macros(int64_t n, int64_t npad, const int32_t *perm, const int32_t *loc, const double *W, double rr,
                          double *rho, double *u, cudaStream_t st);
// residual over the listed cells: snap [2][npad] (U0, V0); partial [blocks][4];
// out[4] = (num, den, mass, non-finite count)
cudaError_t launch_residual(int64_t n, int64_t npad, const int32_t *loc, const double *W, double rr, const double *vol,
                            double *snap, double *partial, int n_blocks, double *out, cudaStream_t st);
inline double rho_ref_of(int prec) { return prec == P_FP64 ? 0.0 : 1.0; }
int residual_blocks(int64_t n);

// records msg as the calling thread's sdugks_last_error() and returns code
int set_error(int code, const char *msg);

}  // namespace sdugks
