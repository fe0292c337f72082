// Energy diagnostics in FP64 (paper: the pair-potential cycle is energy conserving):
// kinetic energy per species, electric and magnetic field energy, pair-potential energy.
// Each block reduces its share into a fixed slot of a partials array; a single block then adds
// the partials in block order, so the result does not depend on scheduling.
#include "pic_device.cuh"

namespace gbpic {

constexpr int kEBlock = 256;
constexpr int kBatch = 4;   // particles of a thread whose loads are in flight together
constexpr int kSlots = 5;   // 0 KE ions, 1 KE electrons, 2 field E, 3 field B, 4 pair

// lanes of a warp, a fixed-shape tree (the result in lane 0)
__device__ __forceinline__ double warp_sum(double v)
{
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    return v;
}

struct EnergyArgs {
    int nx, nz, nsp;
    unsigned nx_magic;
    int nx_shift;
    SpeciesBuf sp[2];
    int64_t n[2];
    const float* F[6];
    const u64* rho;
    float rho_s, h_coef, c_att, s_rep;
    int pot_mode;
    EamP eam;
    double* partials;   // gridDim.x * kSlots
};

// LJ: Eq. (3) on the cubic lattice compiled in (the run-time potential code costs the other forms' branches).
template <bool LJ>
__global__ void __launch_bounds__(kEBlock) k_energy(const EnergyArgs a)
{
    __shared__ double sh[kSlots][kEBlock];
    const int64_t tid = blockIdx.x * (int64_t)kEBlock + threadIdx.x;
    const int64_t stride = (int64_t)gridDim.x * kEBlock;
    LongSum ke[2], pe;
    double fe = 0.0, fb = 0.0;
#pragma unroll
    for (int s = 0; s < 2; s++) {
        if (s >= a.nsp) break;
        const SpeciesBuf& S = a.sp[s];
        int terms = 0;
        for (int64_t p0 = tid; p0 < a.n[s]; p0 += kBatch * stride) {
            float ux[kBatch], uy[kBatch], uz[kBatch], fx[kBatch], fz[kBatch];
            int cell[kBatch];
#pragma unroll
            for (int q = 0; q < kBatch; q++) {
                const int64_t p = p0 + q * stride;
                const bool in = p < a.n[s];
                ux[q] = in ? S.ux[p] : 0.0f;
                uy[q] = in ? S.uy[p] : 0.0f;
                uz[q] = in ? S.uz[p] : 0.0f;
                if (s == 0) {            // the kinetic energy of the electrons needs no cell
                    cell[q] = in ? S.cell[p] : 0;
                    fx[q] = in ? S.fx[p] : 0.0f;
                    fz[q] = in ? S.fz[p] : 0.0f;
                }
            }
            float n[kBatch], dnx[kBatch], dnz[kBatch];
            if (s == 0) {
#pragma unroll
                for (int q = 0; q < kBatch; q++) {
                    const int c = cell[q], k = (int)(__umulhi((unsigned)c, a.nx_magic) >> a.nx_shift), i = c - k * a.nx;
                    gather_density<true>(a.rho, a.nx, a.nz, a.rho_s, i, k, fx[q], fz[q], n[q], dnx[q], dnz[q]);
                }
            }
#pragma unroll
            for (int q = 0; q < kBatch; q++) {
                if (p0 + q * stride >= a.n[s]) continue;
                const float u2 = ux[q] * ux[q] + uy[q] * uy[q] + uz[q] * uz[q];
                ke[s].add(u2 / (sqrtf(1.0f + u2) + 1.0f));
                if (s == 0 && n[q] > 0.0f) {
                    const float cr = fast_cbrt(n[q]);
                    const float inv43 = fast_rcp(n[q] * cr);
                    pe.add(pair_energy_xz(cr, inv43, dnx[q], dnz[q], a.h_coef, LJ ? 0 : a.pot_mode, a.c_att, a.s_rep, a.eam));
                }
            }
            if ((terms += kBatch) == kFold) {
                terms = 0;
                ke[s].fold();
                if (s == 0) pe.fold();
            }
        }
    }
    const int64_t nn = (int64_t)(a.nz + 1) * a.nx;
    for (int64_t c = tid; c < nn; c += stride) {
        const int k = (int)(c / a.nx);
        const double wn = (k == 0 || k == a.nz) ? 0.5 : 1.0;
        const double ex = a.F[0][c], ey = a.F[1][c], bz = a.F[5][c];
        fe += wn * (ex * ex + ey * ey);
        fb += wn * bz * bz;
        if (k < a.nz) {
            const double ez = a.F[2][c], bx = a.F[3][c], by = a.F[4][c];
            fe += ez * ez;
            fb += bx * bx + by * by;
        }
    }
    // Warp s adds up slot s. (A shuffle tree in every warp for every slot took 60 FP64 instructions per warp, about
    // 15 us whatever the size on 2 FP64 lanes per SM; this takes 13 per slot and block.)
    sh[0][threadIdx.x] = ke[0].value();
    sh[1][threadIdx.x] = ke[1].value();
    sh[2][threadIdx.x] = fe;
    sh[3][threadIdx.x] = fb;
    sh[4][threadIdx.x] = pe.value();
    __syncthreads();
    const int s = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (s < kSlots) {
        double v = sh[s][lane];
        for (int w = 1; w < kEBlock / 32; w++) v += sh[s][lane + 32 * w];
        v = warp_sum(v);
        if (lane == 0) a.partials[(size_t)blockIdx.x * kSlots + s] = v;
    }
}

// one warp per slot, blocks assigned to lanes in a fixed way
__device__ __forceinline__ double sum_slot(const double* __restrict__ partials, int nb, int s, int lane)
{
    double v = 0.0;
    for (int b = lane; b < nb; b += 32) v += partials[(size_t)b * kSlots + s];
    return warp_sum(v);
}

__global__ void __launch_bounds__(32 * kSlots) k_energy_final(const double* __restrict__ partials, int nb, double* out)
{
    const int s = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const double r = sum_slot(partials, nb, s, lane);
    if (lane == 0) out[s] = r;
}

// Sums of FP32 terms in three FP32 numbers (LongSum) and the FP64 conversions kept off the common way: a call on the
// 33.5 M particles and 1 M nodes of the 1024^2 slab 520 -> 287 us (8 FP64-pipe instructions per particle were its bound).
// Small states take as many blocks as give every thread a particle or a node: each block costs its share of
// FP64 adds at the end (64^2 cells, 16384 ions: 23.1 us with every block and shuffle trees, 7.2 now; the final sum
// 8.4 -> 2.3). Returns the blocks taken, at most `most`.
static int run_energy(const EnergyArgs& a, int most, cudaStream_t st)
{
    const int64_t nn = (int64_t)(a.nz + 1) * a.nx, n = a.n[0] > a.n[1] ? a.n[0] : a.n[1];
    const int64_t want = ((n > nn ? n : nn) + kEBlock - 1) / kEBlock;
    const int nb = want < most ? (int)want : most;
    if (a.pot_mode == 0) k_energy<true><<<nb, kEBlock, 0, st>>>(a);
    else k_energy<false><<<nb, kEBlock, 0, st>>>(a);
    return nb;
}

int energy_blocks(const Ctx& c) { return c.nsm * 4; }

void launch_energy(Ctx& c, cudaStream_t st, double* host_out5)
{
    EnergyArgs a;
    a.nx = c.nx;
    a.nz = c.nz;
    magic_div(c.nx, a.nx_magic, a.nx_shift);
    a.nsp = c.nsp;
    for (int s = 0; s < 2; s++) {
        a.sp[s] = c.sp[s].a;
        a.n[s] = c.sp[s].n;
    }
    for (int q = 0; q < 6; q++) a.F[q] = c.F[q];
    a.rho = c.rho[c.cur];
    a.rho_s = (float)c.rho_scale;
    a.h_coef = (float)(c.r0 / (6.0 * c.cfg.dx));
    a.c_att = pot_param(c.cfg);
    a.s_rep = (float)c.cfg.s_rep;
    a.pot_mode = pot_code(c.cfg);
    a.eam = eam_params(c.cfg);
    a.partials = c.partials;
    const int nb = run_energy(a, energy_blocks(c), st);
    k_energy_final<<<1, 32 * kSlots, 0, st>>>(c.partials, nb, c.red_out);
    double raw[kSlots];
    cudaMemcpyAsync(raw, c.red_out, sizeof(raw), cudaMemcpyDeviceToHost, st);
    cudaStreamSynchronize(st);
    const double vol = c.cfg.dx * c.cfg.dx;
    const double mu0 = 1.0 / (kEps0 * kC * kC);
    host_out5[0] = raw[0] * c.w * c.sp[0].mass * kC * kC;
    host_out5[1] = c.nsp > 1 ? raw[1] * c.w * c.sp[1].mass * kC * kC : 0.0;
    host_out5[2] = 0.5 * kEps0 * raw[2] * vol;
    host_out5[3] = 0.5 / mu0 * raw[3] * vol;
    host_out5[4] = 0.5 * c.D * raw[4] * c.w;
}

}  // namespace gbpic

// ---------------------------------------------------------------------------------------------
// Workspace-free variant of the energy reduction (pic_energy_noalloc in include/pic.h).
//
// Some callers cannot allocate device memory at all: a host that hands this library buffers it
// owns but forbids further cudaMalloc (a caller-managed memory pool, or code that must not
// allocate while a CUDA graph is being recorded by someone else). For them the reduction's
// scratch -- one partial-sum record per block -- lives in a fixed array in this translation unit,
// reserved on every GPU that loads the library until the process exits.
// ---------------------------------------------------------------------------------------------

namespace gbpic {

constexpr int kStaticBlocks = 1024;                     // partial records the fixed scratch holds
static __device__ __align__(256) double g_noalloc_scratch[kStaticBlocks * kSlots];

// Final pass of the workspace-free variant: adds the block partials in block order (the same
// fixed-shape tree as k_energy_final) and writes the five energies in J per metre of y.
__global__ void __launch_bounds__(32 * kSlots)
    k_energy_final_scaled(const double* __restrict__ partials, int nb, double s0, double s1, double s2, double s3,
                          double s4, double* out)
{
    const int s = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const double r = sum_slot(partials, nb, s, lane);
    if (lane == 0) out[s] = r * (s == 0 ? s0 : s == 1 ? s1 : s == 2 ? s2 : s == 3 ? s3 : s4);
}

}  // namespace gbpic

#include <mutex>

namespace {

constexpr int kMaxDevices = 64;
std::mutex g_noalloc_mutex;
double* g_noalloc_ptr[kMaxDevices] = {};

// Device address of the fixed scratch on the current device. The symbol name is only a host-side
// handle: its device address comes from cudaGetSymbolAddress, taken once per device with that
// device current, on the first call.
int noalloc_scratch(double** out)
{
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return PIC_ECUDA;
    std::lock_guard<std::mutex> lock(g_noalloc_mutex);
    if (!g_noalloc_ptr[dev]) {
        void* p = nullptr;
        if (cudaGetSymbolAddress(&p, gbpic::g_noalloc_scratch) != cudaSuccess || !p) return PIC_ECUDA;
        g_noalloc_ptr[dev] = static_cast<double*>(p);
    }
    *out = g_noalloc_ptr[dev];
    return PIC_OK;
}

}  // namespace

extern "C" int pic_energy_noalloc(const pic_config* cfg, const pic_state_view* in, double* dev_out5, void* stream)
{
    using namespace gbpic;
    if (!cfg || !in || !dev_out5) return PIC_EINVAL;
    if (cfg->dims != 0 && cfg->dims != 2) return PIC_EINVAL;     // 2D states only
    if (cfg->nx < 3 || cfg->nz < 4 || cfg->nx >= 32768 || cfg->nz >= 32768) return PIC_EINVAL;
    if (cfg->mode != PIC_MODE_FULL && cfg->mode != PIC_MODE_TRANSPORT) return PIC_EINVAL;
    if (!(cfg->dx > 0) || !(cfg->n_atoms > 0) || !(cfg->ion_mass_amu > 0) || cfg->ppc_ion <= 0) return PIC_EINVAL;
    if (cfg->pot_mode < 0 || cfg->pot_mode > 3) return PIC_EINVAL;
    if (cfg->pot_mode == 2 && !(cfg->morse_a > 0 && cfg->morse_a < 1e3)) return PIC_EINVAL;
    if (cfg->lattice != PIC_LATTICE_CUBIC && cfg->lattice != PIC_LATTICE_HCP) return PIC_EINVAL;
    if (!eam_config_ok(*cfg)) return PIC_EINVAL;
    const int nsp = cfg->mode == PIC_MODE_FULL ? 2 : 1;
    for (int s = 0; s < nsp; s++) {
        // sizes beyond what the kernels index with 32-bit cells are refused
        if (in->n[s] < 0 || in->n[s] > (int64_t)INT32_MAX) return PIC_EINVAL;
        if (in->n[s] > 0 && (!in->cell[s] || !in->fx[s] || !in->fz[s] || !in->ux[s] || !in->uy[s] || !in->uz[s]))
            return PIC_EINVAL;
    }
    for (int q = 0; q < 6; q++)
        if (!in->F[q]) return PIC_EINVAL;
    if (!in->rho) return PIC_EINVAL;

    double* scratch = nullptr;
    int r = noalloc_scratch(&scratch);
    if (r) return r;
    int dev = 0, nsm = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        return PIC_ECUDA;
    const int most = nsm * 4 < kStaticBlocks ? nsm * 4 : kStaticBlocks;

    // derived constants, as pic_init derives them
    const double w = cfg->n_atoms * cfg->dx * cfg->dx / (double)cfg->ppc_ion;
    const double r0 = cfg->r0 > 0 ? cfg->r0 : pow(cfg->n_atoms, -1.0 / 3.0);
    const double D = cfg->D_eV * kQe;
    const double rho_scale = w / (4294967296.0 * cfg->dx * cfg->dx) * r0 * r0 * r0;
    const double mi = cfg->ion_mass_amu * kAmu;

    EnergyArgs a;
    a.nx = cfg->nx;
    a.nz = cfg->nz;
    magic_div(cfg->nx, a.nx_magic, a.nx_shift);
    a.nsp = nsp;
    for (int s = 0; s < 2; s++) {
        const bool on = s < nsp;
        a.sp[s].cell = on ? const_cast<int32_t*>(in->cell[s]) : nullptr;
        a.sp[s].fx = on ? const_cast<float*>(in->fx[s]) : nullptr;
        a.sp[s].fz = on ? const_cast<float*>(in->fz[s]) : nullptr;
        a.sp[s].ux = on ? const_cast<float*>(in->ux[s]) : nullptr;
        a.sp[s].uy = on ? const_cast<float*>(in->uy[s]) : nullptr;
        a.sp[s].uz = on ? const_cast<float*>(in->uz[s]) : nullptr;
        a.n[s] = on ? in->n[s] : 0;
    }
    for (int q = 0; q < 6; q++) a.F[q] = in->F[q];
    a.rho = reinterpret_cast<const u64*>(in->rho);
    a.rho_s = (float)rho_scale;
    a.h_coef = (float)(r0 / (6.0 * cfg->dx));
    a.c_att = pot_param(*cfg);
    a.s_rep = (float)cfg->s_rep;
    a.pot_mode = pot_code(*cfg);
    a.eam = eam_params(*cfg);
    a.partials = scratch;    // every block overwrites its own record: nothing to clear
    const cudaStream_t st = (cudaStream_t)stream;
    const double vol = cfg->dx * cfg->dx;
    const double mu0 = 1.0 / (kEps0 * kC * kC);
    const int nb = run_energy(a, most, st);
    k_energy_final_scaled<<<1, 32 * kSlots, 0, st>>>(scratch, nb, w * mi * kC * kC, nsp > 1 ? w * kMe * kC * kC : 0.0,
                                                  0.5 * kEps0 * vol, 0.5 / mu0 * vol, 0.5 * D * w, dev_out5);
    return cudaGetLastError() == cudaSuccess ? PIC_OK : PIC_ECUDA;
}
