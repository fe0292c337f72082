// Stand-alone entry kernels: node density of the pair species at the current positions (paper:
// weights interpolated to the nearest surrounding nodes) and the per-atom pair force from that
// density (Eqs. 1-3), without advancing the particles.
#include "pic_device.cuh"

namespace gbpic {

// A warp takes chunks of 32 x cols records; lane l walks records l, l + 32, ... of its chunk. The sort
// stores a block of the cell order as a 32-row matrix column by column, so these are consecutive
// particles of the cell order (between sorts they have barely moved): the lane sums a run of particles of one
// cell in registers and issues the four corner reductions once per run (any order stays exact; only
// the runs get shorter). One set of reductions per particle was bound by them: 128 us for 16.8 M ions on
// 1024^2 cells, 36 us now.
__global__ void __launch_bounds__(256) k_deposit_density(const int32_t* __restrict__ cell, const float* __restrict__ fx,
                                                         const float* __restrict__ fz, int64_t n, int nx, unsigned magic,
                                                         int shift, int cols, u64* out)
{
    const int lane = threadIdx.x & 31;
    const int64_t warp = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5, nwarp = ((int64_t)gridDim.x * blockDim.x) >> 5;
    const int64_t chunk = 32 * (int64_t)cols;
    for (int64_t base = warp * chunk; base < n; base += nwarp * chunk) {
        int at = -1;
        u64 s00 = 0, s10 = 0, s01 = 0, s11 = 0;
        auto flush = [&]() {
            const int k = (int)(__umulhi((unsigned)at, magic) >> shift), i = at - k * nx;
            u64* r = out + at;
            const int d1 = i + 1 == nx ? 1 - nx : 1;
            if (s00) atomicAdd(r, s00);
            if (s10) atomicAdd(r + d1, s10);
            if (s01) atomicAdd(r + nx, s01);
            if (s11) atomicAdd(r + nx + d1, s11);
            s00 = s10 = s01 = s11 = 0;
        };
        for (int q0 = 0; q0 < cols; q0 += kRunBatch) {
            int c[kRunBatch];
            float ox[kRunBatch], oz[kRunBatch];
#pragma unroll
            for (int q = 0; q < kRunBatch; q++) {
                const int64_t p = base + 32 * (int64_t)(q0 + q) + lane;
                const bool in = q0 + q < cols && p < n;
                c[q] = in ? cell[p] : -1;
                ox[q] = in ? fx[p] : 0.0f;
                oz[q] = in ? fz[p] : 0.0f;
            }
#pragma unroll
            for (int q = 0; q < kRunBatch; q++) {
                if (c[q] < 0) continue;
                if (c[q] != at) {
                    if (at >= 0) flush();
                    at = c[q];
                }
                const unsigned x = (unsigned)qoff(ox[q]), z = (unsigned)qoff(oz[q]), ax = kQOne - x, az = kQOne - z;
                s00 += (u64)ax * az;
                s10 += (u64)x * az;
                s01 += (u64)ax * z;
                s11 += (u64)x * z;
            }
        }
        if (at >= 0) flush();
    }
}

__global__ void k_pair_force(const int32_t* __restrict__ cell, const float* __restrict__ fx,
                             const float* __restrict__ fz, int64_t n, int nx, int nz, const u64* __restrict__ rho,
                             float rho_s, float h_coef, int pot_mode, float c_att, float s_rep, float f_unit,
                             EamP eam, float* __restrict__ out)
{
    for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < n; p += (int64_t)gridDim.x * blockDim.x) {
        const int c = cell[p];
        const int k = c / nx, i = c - k * nx;
        float dens, dnx, dnz;
        gather_density(rho, nx, nz, rho_s, i, k, fx[p], fz[p], dens, dnx, dnz);
        float Fx, Fz;
        pair_force_xz(dens, dnx, dnz, h_coef, pot_mode, c_att, s_rep, Fx, Fz, eam);
        out[3 * p + 0] = f_unit * Fx;
        out[3 * p + 1] = 0.0f;
        out[3 * p + 2] = f_unit * Fz;
    }
}

// Pair force at probe positions that add nothing to the density (the calibration of the attractive
// factor follows one atom out of the target). A probe outside the grid or with an offset outside
// [0, 1) x [0, 1] reads nothing and gets NaN.
__global__ void k_pair_force_probe(const int32_t* __restrict__ cell, const float* __restrict__ fx,
                                   const float* __restrict__ fz, int64_t n, int nx, int nz,
                                   const u64* __restrict__ rho, float rho_s, float h_coef, int pot_mode,
                                   float c_att, float s_rep, float f_unit, EamP eam, float* __restrict__ out)
{
    for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < n; p += (int64_t)gridDim.x * blockDim.x) {
        const int c = cell[p];
        const float a = fx[p], b = fz[p];
        if (c < 0 || c >= nx * nz || !(a >= 0.0f && a < 1.0f && b >= 0.0f && b <= 1.0f)) {
            out[3 * p + 0] = out[3 * p + 1] = out[3 * p + 2] = __int_as_float(0x7fc00000);
            continue;
        }
        const int k = c / nx, i = c - k * nx;
        float dens, dnx, dnz;
        gather_density(rho, nx, nz, rho_s, i, k, a, b, dens, dnx, dnz);
        float Fx, Fz;
        pair_force_xz<true>(dens, dnx, dnz, h_coef, pot_mode, c_att, s_rep, Fx, Fz, eam);
        out[3 * p + 0] = f_unit * Fx;
        out[3 * p + 1] = 0.0f;
        out[3 * p + 2] = f_unit * Fz;
    }
}

// Flags particles outside the grid or with offsets outside [0,1) x [0,1] (bit 0 of *bad).
__global__ void k_validate(const int32_t* __restrict__ cell, const float* __restrict__ fx,
                           const float* __restrict__ fy, const float* __restrict__ fz, int64_t n, int64_t ncell,
                           unsigned* bad)
{
    for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < n; p += (int64_t)gridDim.x * blockDim.x) {
        const int c = cell[p];
        const float a = fx[p], b = fz[p], y = fy ? fy[p] : 0.0f;
        if (c < 0 || c >= ncell || !(a >= 0.0f && a < 1.0f && b >= 0.0f && b <= 1.0f && y >= 0.0f && y < 1.0f))
            atomicOr(bad, 1u);
    }
}

static int grid_for(const Ctx& c, int64_t n)
{
    int64_t g = (n + 255) / 256;
    const int64_t cap = (int64_t)c.nsm * 8;
    if (g > cap) g = cap;
    return g < 1 ? 1 : (int)g;
}

void launch_deposit_density(Ctx& c, u64* out, cudaStream_t st)
{
    cudaMemsetAsync(out, 0, sizeof(u64) * c.nn, st);
    const Species& S = c.sp[0];
    if (S.n == 0) return;
    unsigned magic;
    int shift;
    magic_div(c.nx, magic, shift);
    const int cols = run_columns(c, S);
    k_deposit_density<<<run_grid(c, S.n, cols), 256, 0, st>>>(S.a.cell, S.a.fx, S.a.fz, S.n, c.nx, magic, shift, cols,
                                                              out);
}

void launch_validate(Ctx& c, const SpeciesBuf& b, int64_t n, unsigned* bad, cudaStream_t st)
{
    if (n == 0) return;
    k_validate<<<grid_for(c, n), 256, 0, st>>>(b.cell, b.fx, c.dims == 3 ? b.fy : nullptr, b.fz, n,
                                               (int64_t)c.nx * c.ny * c.nz, bad);
}

void launch_pair_force_probe(Ctx& c, int64_t n, const int32_t* cell, const float* fx, const float* fz, int pot_mode,
                             double c_att, double s_rep, float* out, cudaStream_t st)
{
    if (n == 0) return;
    k_pair_force_probe<<<grid_for(c, n), 256, 0, st>>>(cell, fx, fz, n, c.nx, c.nz, c.rho[c.cur], (float)c.rho_scale,
                                                      (float)(c.r0 / (6.0 * c.cfg.dx)), pot_mode, (float)c_att,
                                                      (float)s_rep, (float)(c.D / c.r0), eam_params(c.cfg), out);
}

void launch_pair_force(Ctx& c, float* out, cudaStream_t st)
{
    const Species& S = c.sp[0];
    if (S.n == 0) return;
    k_pair_force<<<grid_for(c, S.n), 256, 0, st>>>(S.a.cell, S.a.fx, S.a.fz, S.n, c.nx, c.nz, c.rho[c.cur],
                                                   (float)c.rho_scale, (float)(c.r0 / (6.0 * c.cfg.dx)),
                                                   pot_code(c.cfg), pot_param(c.cfg), (float)c.cfg.s_rep,
                                                   (float)(c.D / c.r0), eam_params(c.cfg), out);
}

}  // namespace gbpic
