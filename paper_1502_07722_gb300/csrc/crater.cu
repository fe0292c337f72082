// Crater profile of the atomic-transport stage (paper: once the crater has solidified its width
// and depth are measured from the density map and compared with experiment; Eq. 5 turns the
// width into a threshold fluence). For every column of nodes the material missing from the
// original slab, as a thickness of solid-density material:
//     d(column) = dx * scale / n_atoms * sum_{k = 0..slab_k} (rho0 - rho)(k, column),
// rho0 the node sums at the start, rho the current ones (int64 node sums of the pair species),
// scale the factor from a node sum to a density in m^-3. The column sums are exact integers; one
// FP64 multiply per column turns them into metres.
#include "pic_internal.cuh"

namespace gbpic {

// A warp reads 32 neighbouring nodes of a row. A block's 16 warps are 2^lr that take every 2^lr-th row of the same 32
// columns, their integer sums meeting in shared memory, times groups of 32 columns: about eight rows per warp. (One thread
// per column, walking all rows, was one chain of dependent loads: 139 us for 1024 columns of 513 rows, 12 with 16 warps
// to a column whatever the rows; 512 x 512 columns of 7 rows 9 us by single threads, 13 by 16 warps, 9 now.)
constexpr int kProfileWarps = 16;
template <int LR>
__global__ void __launch_bounds__(32 * kProfileWarps)
    k_crater_profile(const u64* __restrict__ rho0, const u64* __restrict__ rho, int64_t ncol, int rows, double depth_scale,
                     double* __restrict__ out)
{
    __shared__ long long sh[kProfileWarps][32];
    constexpr int nr = 1 << LR;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, r = w & (nr - 1);
    const int64_t col = (blockIdx.x * (int64_t)(kProfileWarps >> LR) + (w >> LR)) * 32 + lane;
    long long s = 0;
    if (col < ncol) {
#pragma unroll 4
        for (int k = r; k < rows; k += nr) {
            const size_t q = (size_t)k * (size_t)ncol + (size_t)col;
            s += (long long)(__ldg(rho0 + q) - __ldg(rho + q));
        }
    }
    sh[w][lane] = s;
    __syncthreads();
    if (r == 0 && col < ncol) {
        for (int q = 1; q < nr; q++) s += sh[w + q][lane];
        out[col] = (double)s * depth_scale;
    }
}

void launch_crater_profile(Ctx& c, const u64* rho0, double depth_scale, double* out, cudaStream_t st)
{
    const int64_t ncol = (int64_t)c.nx * c.ny;
    const int rows = c.cfg.slab_k + 1 < c.nz + 1 ? c.cfg.slab_k + 1 : c.nz + 1;
    int lr = 0;
    while (1 << lr < kProfileWarps && 8 << lr < rows) lr++;
    const int64_t cols = 32 * (kProfileWarps >> lr);
    auto kernel = lr == 0 ? k_crater_profile<0>
                : lr == 1 ? k_crater_profile<1>
                : lr == 2 ? k_crater_profile<2>
                : lr == 3 ? k_crater_profile<3> : k_crater_profile<4>;
    kernel<<<(unsigned)((ncol + cols - 1) / cols), 32 * kProfileWarps, 0, st>>>(rho0, c.rho[c.cur], ncol, rows, depth_scale, out);
}

}  // namespace gbpic
