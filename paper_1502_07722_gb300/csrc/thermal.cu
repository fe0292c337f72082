// Coupling of the two stages (paper: the atomic-transport run starts from the lattice temperature
// the laser-interaction run leaves once electrons and lattice have equilibrated).
//  * Lattice temperature per cell of one species: T = m c^2 / (3 k_B) sum |u - mean u|^2 / (N - 1)
//    over the N particles of the cell (the thermal spread about the cell's mean flow); cells with
//    fewer than two particles get 0. Per-cell sums (FP64 atomics), then one thread per cell.
//  * Re-tempering to a map: momenta drawn at the uniform temperature T_from become the same draws
//    at the temperature of their cell, u -> u sqrt(T_cell / T_from).
//  * Regridding a cell map between stages of different cells: a conservative (volume-weighted)
//    remap on grids placed on each other by the slab's surface and the laser axis.
#include "pic_internal.cuh"
#include "pic_device.cuh"

namespace gbpic {

// momenta whose squares, or the rounding errors of these, leave FP32's range (or that are not finite)
static __device__ __noinline__ void add_wide_moments(double* acc, int64_t ncell, int at, float a, float b, float c)
{
    const double da = a, db = b, dc = c;
    atomicAdd(acc + at, 1.0);
    atomicAdd(acc + ncell + at, da);
    atomicAdd(acc + 2 * ncell + at, db);
    atomicAdd(acc + 3 * ncell + at, dc);
    atomicAdd(acc + 4 * ncell + at, da * da + db * db + dc * dc);
}

// Number, sums of u and of u^2 of each cell's particles. Lanes walk runs of particles of one cell
// (run_columns) and sum them in registers as three FP32 numbers: GB300's FP64 rate is 1/64 of its FP32
// rate, and the conversions and products of one FP64 reduction per particle took 189 us for 16.8 M
// particles on 1024^2 cells, 85 to 131 us now. A run that ends goes to the warp's queue; the queue is
// converted to FP64 and reduced into the cells 32 runs at a time (lanes end their runs at different turns,
// and an FP64 instruction costs the same for one lane as for 32).
constexpr int kMomWarps = 4, kMomWords = 14;
__global__ void __launch_bounds__(32 * kMomWarps)
    k_cell_moments(const int32_t* __restrict__ cell, const float* __restrict__ ux, const float* __restrict__ uy,
                   const float* __restrict__ uz, int64_t n, int64_t ncell, int cols, double* __restrict__ acc)
{
    __shared__ int queue_all[kMomWarps][kMomWords][64];      // at most 31 left over + 32 new per warp
    int(*queue)[64] = queue_all[threadIdx.x >> 5];
    const int lane = threadIdx.x & 31;
    const int64_t warp = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5, nwarp = ((int64_t)gridDim.x * blockDim.x) >> 5;
    const int64_t chunk = 32 * (int64_t)cols;
    int at = -1, num = 0, nq = 0;
    Sum3 v[4];            // u and u^2
    auto drain = [&](int count) {
        __syncwarp();
        nq -= count;
        if (lane < count) {
            const int e = nq + lane, c = queue[0][e];
            atomicAdd(acc + c, (double)queue[1][e]);
#pragma unroll
            for (int d = 0; d < 4; d++) {
                const Sum3 t = {__int_as_float(queue[2 + 3 * d][e]), __int_as_float(queue[3 + 3 * d][e]),
                                __int_as_float(queue[4 + 3 * d][e])};
                atomicAdd(acc + (d + 1) * ncell + c, t.value());
            }
        }
        __syncwarp();
    };
    // queues the run of every lane with `end` set (all lanes of the warp call it)
    auto close = [&](bool end) {
        const unsigned m = __ballot_sync(0xffffffffu, end);
        if (m == 0) return;
        if (end) {
            const int e = nq + __popc(m & ((1u << lane) - 1u));
            queue[0][e] = at;
            queue[1][e] = num;
#pragma unroll
            for (int d = 0; d < 4; d++) {
                queue[2 + 3 * d][e] = __float_as_int(v[d].s0);
                queue[3 + 3 * d][e] = __float_as_int(v[d].s1);
                queue[4 + 3 * d][e] = __float_as_int(v[d].s2);
                v[d].zero();
            }
            num = 0;
        }
        nq += __popc(m);
        if (nq >= 32) drain(32);
    };
    for (int d = 0; d < 4; d++) v[d].zero();
    for (int64_t base = warp * chunk; base < n; base += nwarp * chunk) {
        for (int q0 = 0; q0 < cols; q0 += kRunBatch) {
            int k[kRunBatch];
            float va[kRunBatch], vb[kRunBatch], vc[kRunBatch];
#pragma unroll
            for (int q = 0; q < kRunBatch; q++) {
                const int64_t p = base + 32 * (int64_t)(q0 + q) + lane;
                const bool in = q0 + q < cols && p < n;
                k[q] = in ? cell[p] : -1;
                va[q] = in ? ux[p] : 0.0f;
                vb[q] = in ? uy[p] : 0.0f;
                vc[q] = in ? uz[p] : 0.0f;
            }
#pragma unroll
            for (int q = 0; q < kRunBatch; q++) {
                close(k[q] >= 0 && k[q] != at && num > 0);
                if (k[q] < 0) continue;
                at = k[q];
                const float a = va[q], b = vb[q], c = vc[q];
                const float size = fabsf(a) + fabsf(b) + fabsf(c);       // a particle at rest has nothing to round
                if (!(size < 1e15f) || (size < 0x1p-40f && size > 0.0f)) {
                    add_wide_moments(acc, ncell, at, a, b, c);
                    continue;
                }
                num++;
                v[0].add(a);
                v[1].add(b);
                v[2].add(c);
                v[3].add_square(a);
                v[3].add_square(b);
                v[3].add_square(c);
            }
        }
        close(num > 0);
    }
    if (nq > 0) drain(nq);
}

// One FP64 reduction per particle and sum.
__global__ void k_cell_moments_direct(const int32_t* __restrict__ cell, const float* __restrict__ ux,
                                      const float* __restrict__ uy, const float* __restrict__ uz, int64_t n, int64_t ncell,
                                      double* __restrict__ acc)
{
    for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < n; p += (int64_t)gridDim.x * blockDim.x) {
        const int64_t q = cell[p];
        const double a = ux[p], b = uy[p], c = uz[p];
        atomicAdd(acc + q, 1.0);
        atomicAdd(acc + ncell + q, a);
        atomicAdd(acc + 2 * ncell + q, b);
        atomicAdd(acc + 3 * ncell + q, c);
        atomicAdd(acc + 4 * ncell + q, a * a + b * b + c * c);
    }
}

// Which of the two: the walk pays for its serial loads, queue and conversions with long runs and many of them. Whole
// call, us, walk / direct after 43 steps: 0.5 M particles at 8 per cell 28 / 23 (2D) and 31 / 23 (3D), at 64 per cell
// 27 / 23 and 28 / 25; 1 M at 16 per cell 31 / 27 and 37 / 29; 2 M at 32 per cell 39 / 40 and 45 / 45; 8 M at 8
// per cell 140 / 158 and 179 / 162, at 32 per cell 87 / 119 and 111 / 124; 24 M at 32 per cell 196 / 324 and 240 / 322.
// Lone particles have no runs (24 M: 1490 / 1243 in 2D), and below 12 per cell the rows of the layout have 8 records, which cut
// the runs of a count that does not divide 8 (24 M at 9 per cell: 489 / 435 and 518 / 435).
static bool direct_moments(const Ctx& c, const Species& S)
{
    return S.n < (c.dims == 3 ? 3 << 19 : 1 << 20) || S.ppc < 2 || (S.ppc < 12 && 8 % S.ppc != 0);
}

__global__ void k_cell_temperature(const double* __restrict__ acc, int64_t ncell, double mc2_3k, double* __restrict__ T)
{
    for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < ncell; q += (int64_t)gridDim.x * blockDim.x) {
        const double n = acc[q];
        if (n < 2.0) {
            T[q] = 0.0;
            continue;
        }
        const double sx = acc[ncell + q], sy = acc[2 * ncell + q], sz = acc[3 * ncell + q];
        T[q] = mc2_3k * (acc[4 * ncell + q] - (sx * sx + sy * sy + sz * sz) / n) / (n - 1.0);
    }
}

__global__ void k_set_temperature(const int32_t* __restrict__ cell, float* ux, float* uy, float* uz, int64_t n,
                                  const double* __restrict__ T, double T_from)
{
    for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < n; p += (int64_t)gridDim.x * blockDim.x) {
        const double f = sqrt(T[cell[p]] / T_from);
        ux[p] = (float)((double)ux[p] * f);
        uy[p] = (float)((double)uy[p] * f);
        uz[p] = (float)((double)uz[p] * f);
    }
}

static int grid_of(const Ctx& c, int64_t n)
{
    int64_t g = (n + 255) / 256;
    if (g > (int64_t)c.nsm * 16) g = (int64_t)c.nsm * 16;
    return g < 1 ? 1 : (int)g;
}

void launch_cell_temperature(Ctx& c, int s, double* work, double* T, cudaStream_t st)
{
    const Species& S = c.sp[s];
    const int64_t ncell = (int64_t)c.nx * c.ny * c.nz;
    cudaMemsetAsync(work, 0, sizeof(double) * 5 * (size_t)ncell, st);
    if (S.n > 0 && direct_moments(c, S)) {
        k_cell_moments_direct<<<grid_of(c, S.n), 256, 0, st>>>(S.a.cell, S.a.ux, S.a.uy, S.a.uz, S.n, ncell, work);
    } else if (S.n > 0) {
        const int cols = run_columns(c, S);
        k_cell_moments<<<2 * run_grid(c, S.n, cols), 32 * kMomWarps, 0, st>>>(S.a.cell, S.a.ux, S.a.uy, S.a.uz, S.n, ncell,
                                                                              cols, work);
    }
    k_cell_temperature<<<grid_of(c, ncell), 256, 0, st>>>(work, ncell, S.mass * kC * kC / (3.0 * kKb), T);
}

void launch_set_temperature(Ctx& c, int s, const double* T, double T_from, cudaStream_t st)
{
    const Species& S = c.sp[s];
    if (S.n > 0) k_set_temperature<<<grid_of(c, S.n), 256, 0, st>>>(S.a.cell, S.a.ux, S.a.uy, S.a.uz, S.n, T, T_from);
}

// One axis of the remap: destination cell d of a grid (n, dx, origin o: cell d spans
// [(d - o) dx, (d + 1 - o) dx]) against the source axis (ns, dxs, os); the source cells it overlaps
// are lo .. hi (empty when lo > hi), the overlap with source cell s is ov(s).
struct RegridAxis {
    double a0, a1, dxs, os;
    int lo, hi;
};
__device__ __forceinline__ RegridAxis regrid_axis(int d, double dx, double o, int ns, double dxs, double os)
{
    RegridAxis A;
    A.a0 = (d - o) * dx;
    A.a1 = (d + 1 - o) * dx;
    A.dxs = dxs;
    A.os = os;
    A.lo = max(0, (int)floor(A.a0 / dxs + os));
    A.hi = min(ns - 1, (int)ceil(A.a1 / dxs + os) - 1);
    return A;
}
__device__ __forceinline__ double regrid_overlap(const RegridAxis& A, int s)
{
    const double b0 = (s - A.os) * A.dxs, b1 = b0 + A.dxs;
    return fmax(0.0, fmin(A.a1, b1) - fmax(A.a0, b0));
}

struct RegridGrid {
    int nx, ny, nz;
    double dx, ox, oy, oz;      // origins: nx / 2, ny / 2, surface
};

__global__ void k_regrid_cells(int dims, const double* __restrict__ src, RegridGrid S, double* __restrict__ dst,
                               RegridGrid D, double fill)
{
    const int64_t nd = (int64_t)D.nx * D.ny * D.nz;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; c < nd; c += stride) {
        const int i = (int)(c % D.nx);
        const int64_t q = c / D.nx;
        const int j = (int)(q % D.ny), k = (int)(q / D.ny);
        const RegridAxis X = regrid_axis(i, D.dx, D.ox, S.nx, S.dx, S.ox);
        const RegridAxis Z = regrid_axis(k, D.dx, D.oz, S.nz, S.dx, S.oz);
        RegridAxis Y;
        if (dims == 3) Y = regrid_axis(j, D.dx, D.oy, S.ny, S.dx, S.oy);
        double sum = 0.0, covered = 0.0;
        for (int sk = Z.lo; sk <= Z.hi; sk++) {
            const double wz = regrid_overlap(Z, sk);
            for (int sj = dims == 3 ? Y.lo : 0; sj <= (dims == 3 ? Y.hi : 0); sj++) {
                const double wzy = dims == 3 ? wz * regrid_overlap(Y, sj) : wz;
                for (int si = X.lo; si <= X.hi; si++) {
                    const double w = wzy * regrid_overlap(X, si);
                    sum += w * src[((int64_t)sk * S.ny + sj) * S.nx + si];
                    covered += w;
                }
            }
        }
        const double vol = dims == 3 ? D.dx * D.dx * D.dx : D.dx * D.dx;
        dst[c] = (sum + fill * (vol - covered)) / vol;
    }
}

}  // namespace gbpic

extern "C" PIC_API int pic_regrid_cells(int32_t dims, const double* dev_src, int32_t src_nx, int32_t src_ny,
                                        int32_t src_nz, double src_dx, int32_t src_surface, double* dev_dst,
                                        int32_t dst_nx, int32_t dst_ny, int32_t dst_nz, double dst_dx,
                                        int32_t dst_surface, double fill, void* stream)
{
    using namespace gbpic;
    if (!dev_src || !dev_dst || (dims != 2 && dims != 3)) return PIC_EINVAL;
    if (dims == 2) src_ny = dst_ny = 1;
    if (src_nx < 1 || src_ny < 1 || src_nz < 1 || dst_nx < 1 || dst_ny < 1 || dst_nz < 1) return PIC_EINVAL;
    if (!(src_dx > 0.0) || !(dst_dx > 0.0)) return PIC_EINVAL;
    if (src_surface < 0 || src_surface > src_nz || dst_surface < 0 || dst_surface > dst_nz) return PIC_EINVAL;
    const RegridGrid S = {src_nx, src_ny, src_nz, src_dx, 0.5 * src_nx, 0.5 * src_ny, (double)src_surface};
    const RegridGrid D = {dst_nx, dst_ny, dst_nz, dst_dx, 0.5 * dst_nx, 0.5 * dst_ny, (double)dst_surface};
    const int64_t nd = (int64_t)dst_nx * dst_ny * dst_nz;
    int64_t g = (nd + 255) / 256;
    if (g > 65536) g = 65536;
    k_regrid_cells<<<(int)g, 256, 0, (cudaStream_t)stream>>>(dims, dev_src, S, dev_dst, D, fill);
    return cudaGetLastError() == cudaSuccess ? PIC_OK : PIC_ECUDA;
}

