// k_strip.cu -- the marching-warp Cartesian step (FP32) of single solves and of batches, and
// its form by blocks for small batches.
#include "step_strip_block.cuh"

namespace sdugks {

// One warp per CTA and (strip, range of rows): what depends on the work item alone is
// then uniform to the compiler, and warps that share nothing need not end together.
__global__ void __launch_bounds__(32, STRIP_CTAS) k_step_strip(const StripInst m, int par, int rows)
{
    extern __shared__ __align__(128) unsigned char smem_raw[];
    step_dependency_wait();
    strip_item(m, par, blockIdx.x, blockIdx.y, rows, smem_raw);
}

// Batched: the instances' records are kernel parameters, so that their constants come from
// constant memory as in the single solve; the work list is written by the host only and
// may be read before the wait on the previous step.
__global__ void __launch_bounds__(32, STRIP_CTAS)
k_strip_batch(const __grid_constant__ StripGroup G, const int2 *__restrict__ items, int par, int rows)
{
    extern __shared__ __align__(128) unsigned char smem_raw[];
    const int2 it = items[blockIdx.x];
    step_dependency_wait();
    const int q = __shfl_sync(0xffffffffu, it.x, 0), y = __shfl_sync(0xffffffffu, it.y, 0);
    strip_item(G.inst[q], par, y & 0xFFFF, y >> 16, rows, smem_raw);
}

// Batched, by blocks (step_strip_block.cuh): one CTA per (instance, block x | block y << 16)
// item.  The items and the records are written by the host only and are read before the wait.
template <bool WIDE>
__global__ void __launch_bounds__(sb_threads<WIDE>(), sb_ctas<WIDE>())
k_strip_block_batch(const StripInst *__restrict__ insts, const int2 *__restrict__ items, int par)
{
    __shared__ __align__(16) StripBlockSmem S;
    const int2 it = items[blockIdx.x];
    static_assert(sizeof(StripInst) % 8 == 0 && sizeof(StripInst) / 8 <= sb_threads<WIDE>(), "the record in one round");
    if (threadIdx.x < sizeof(StripInst) / 8)
        reinterpret_cast<uint64_t *>(&S.m)[threadIdx.x] = reinterpret_cast<const uint64_t *>(insts + it.x)[threadIdx.x];
    step_dependency_wait();
    __syncthreads();
    const int x0 = (it.y & 0xFFFF) * 16, y0 = (it.y >> 16) * BATCH_TY;
    const bool inside = x0 >= 2 && x0 + 18 <= S.m.nx && y0 >= 2 && y0 + BATCH_TY + 2 <= S.m.ny;
    if (inside) strip_block<false, WIDE>(S, par, x0, y0);
    else strip_block<true, WIDE>(S, par, x0, y0);
}

bool strip_fits(const CartInst &m, int prec)
{
    if (prec != P_FP32 || m.npad > (int64_t)1 << 30 || (m.periodic_x && m.nx % 2 != 0)) return false;
    for (int k = 0; k < 4; k++)
        if (m.side_kind[k] == BK_SYMMETRY) return false;
    return true;
}

int strip_count(int nx, bool periodic_x)
{
    // strip k stages the columns from 60 k (60 k - 2 on a periodic grid); the last strip
    // of a grid with sides also updates its last columns
    if (periodic_x) return (nx + STRIP_STEP - 1) / STRIP_STEP;
    return nx <= STRIP_W ? 1 : (nx - (STRIP_W - STRIP_STEP) + STRIP_STEP - 1) / STRIP_STEP;
}

// The parts of one whole (a face's c + b c = 1 times its length and dt/V), for every cell and step the same:
// rounded each by itself, and from rounded factors, the whole is off by up to 1e-7, alike in every
// step.  The larger part is rounded and the smaller one is what it leaves of the whole (448^2, 300 steps, with
// the same for a + b and 1/(1+r) + r/(1+r), which the step has as 1 - b and 1 - r/(1+r): u off by 1.7e-7
// before, 0.8e-7 now, 1.1e-7 by blocks; 8 cavities of 32^2 to 128^2, 500 steps: 4.2e-6, 0.9e-6, 3.2e-6).
static float part_of(double part, double whole)
{
    return part > 0.5 * whole ? (float)part : (float)(whole - (double)(float)(whole - part));
}
static float whole_less(double part, double whole)
{
    return part > 0.5 * whole ? (float)(whole - (double)(float)part) : (float)(whole - part);
}

void fill_strip(const CartInst &m, StripInst &s)
{
    auto two = [](float v) { return make_float2(v, v); };
    auto signs = [&](float2 p[2], double v) { p[0] = two((float)v); p[1] = two(-(float)v); };
    s.nx = m.nx; s.ny = m.ny; s.pitch = m.pitch; s.npad = (int32_t)m.npad;
    s.periodic_x = m.periodic_x; s.periodic_y = m.periodic_y;
    for (int k = 0; k < 4; k++) {
        s.side_kind[k] = m.side_kind[k];
        for (int d = 0; d < 3; d++) s.side_par[k][d] = m.fside_par[k][d];
        s.side_drho[k] = m.fside_drho[k];
    }
    for (int b = 0; b < 2; b++) { s.f[b] = static_cast<float *>(m.f[b]); s.W[b] = m.W[b]; }
    s.b = two((float)m.b); s.ri = two((float)(m.r / (1.0 + m.r)));
    s.sc = (float)(1.0 / (1.0 + m.b)); s.sb = (float)(1.0 / (double)s.sc - 1.0);
    for (int x = 0; x < 2; x++) {
        const double lv = (x == 0 ? m.dy : m.dx) * m.dtV, bg = lv * m.b / (1.0 + m.b);
        s.len_dtV[x] = (float)lv;
        s.g[x] = two(whole_less(bg, lv)); s.bg[x] = two(part_of(bg, lv));
    }
    const double ax = 0.5 * m.ihx, ay = 0.5 * m.ihy;
    signs(s.xdt, m.dt * ax); signs(s.xh, STRIP_XH); signs(s.xo, 0.25 - m.dt * ax);
    signs(s.ydt, m.dt * ay); signs(s.yh, STRIP_XH); signs(s.yo, 0.25 - m.dt * ay);
}

cudaError_t prepare_strip()
{
    return cudaFuncSetAttribute(k_step_strip, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)STRIP_SMEM);
}

cudaError_t prepare_strip_batch()
{
    return cudaFuncSetAttribute(k_strip_batch, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)STRIP_SMEM);
}

cudaError_t launch_strip_batch(const StripGroup &g, const int2 *items, int n_items, int rows, bool early,
                               int parity, cudaStream_t st)
{
    return launch_step_kernel(early, k_strip_batch, dim3(n_items), dim3(32), STRIP_SMEM, st, g, items, parity, rows);
}

cudaError_t launch_strip_blocks(const StripInst *insts, const int2 *items, int n_items, bool wide, bool early, int parity,
                                cudaStream_t st)
{
    if (wide)
        return launch_step_kernel(early, k_strip_block_batch<true>, dim3(n_items), dim3(sb_threads<true>()), 0, st, insts, items, parity);
    return launch_step_kernel(early, k_strip_block_batch<false>, dim3(n_items), dim3(sb_threads<false>()), 0, st, insts, items, parity);
}

int strip_block_slots(bool wide)
{
    int dev = 0, n_sm = 1, n = 0;
    if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev);
    const cudaError_t e = wide ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_strip_block_batch<true>, sb_threads<true>(), 0)
                               : cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_strip_block_batch<false>, sb_threads<false>(), 0);
    return n_sm * (e != cudaSuccess || n < 1 ? 1 : n);
}

cudaError_t launch_step_strip(const StripInst &s, int rows, bool early, int parity, cudaStream_t st)
{
    return launch_step_kernel(early, k_step_strip, dim3(strip_count(s.nx, s.periodic_x != 0), (s.ny + rows - 1) / rows), dim3(32),
                              STRIP_SMEM, st, s, parity, rows);
}

int strip_slots()
{
    int dev = 0, n_sm = 1, n = 0;
    if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev);
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_step_strip, 32, STRIP_SMEM) != cudaSuccess || n < 1) n = 1;
    return n_sm * n;
}

}  // namespace sdugks
