// k_strip.cu -- the marching-warp Cartesian step (FP32) of single solves and of batches.
#include "step_strip.cuh"

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

void fill_strip(const CartInst &m, StripInst &s)
{
    auto two = [](float v) { return make_float2(v, v); };
    auto signs = [&](float2 p[2], float v) { p[0] = two(v); p[1] = two(-v); };
    s.nx = m.nx; s.ny = m.ny; s.pitch = m.pitch; s.npad = (int32_t)m.npad;
    s.periodic_x = m.periodic_x; s.periodic_y = m.periodic_y;
    for (int k = 0; k < 4; k++) {
        s.side_kind[k] = m.side_kind[k];
        for (int d = 0; d < 3; d++) s.side_par[k][d] = m.fside_par[k][d];
        s.side_drho[k] = m.fside_drho[k];
    }
    for (int b = 0; b < 2; b++) { s.f[b] = static_cast<float *>(m.f[b]); s.W[b] = m.W[b]; }
    s.sb = m.fb; s.sc = m.fc;
    s.a = two(m.fa); s.b = two(m.fb); s.inv = two(m.finv1r); s.ri = two(m.fr * m.finv1r);
    for (int x = 0; x < 2; x++) {
        s.len_dtV[x] = (x == 0 ? m.fdy : m.fdx) * m.fdtV;
        const float g = m.fc * s.len_dtV[x];
        s.g[x] = two(g); s.bg[x] = two(m.fb * g);
    }
    const float hx = 0.5f * m.fdx, hy = 0.5f * m.fdy, ax = 0.5f * m.fihx, ay = 0.5f * m.fihy;
    signs(s.xdt, m.fdt * ax); signs(s.xh, hx * ax); signs(s.xo, (hx - m.fdt) * ax);
    signs(s.ydt, m.fdt * ay); signs(s.yh, hy * ay); signs(s.yo, (hy - m.fdt) * ay);
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
