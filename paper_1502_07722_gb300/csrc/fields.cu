// Maxwell update of the PIC cycle (paper: PIC integrates the Maxwell and Lorentz equations),
// 2D3V Yee scheme with d/dy = 0: B advanced by half a step, E by a full step with the current
// of the particle kernel (int64 fixed point -> A/m^2) and the laser antenna, B by the second
// half step. x is periodic; the tangential E components on the wall rows z = 0 and z = nz take
// the first-order Mur absorbing condition.
//
// The whole update is one kernel. It reads one set of the six field grids and writes the other (the
// context swaps them), so a warp may recompute its neighbours' intermediate values from the old
// ones; the same pass clears the current grids the next step deposits into (the other set) and
// starts the next node density from the current one.
//
// What bounds it: memory traffic on the large grids, the launch on the small ones. Against three
// in-place passes (B half, E, B half) with a copy/clear kernel and a one-thread antenna kernel, a
// node moves 112 bytes instead of 172 and a step has two launches instead of six. (The largest states have no room
// for a second set and keep the three passes: k_half_B, k_E.)
#include "pic_device.cuh"
#include "pic_internal.cuh"

namespace gbpic {

// A warp owns kCols columns (plus one to the left and two to the right that it recomputes) and walks
// up a segment of rows with the last rows' values in registers: the x neighbours come by shuffle, the
// z neighbours from the row before, and no barrier or shared memory is needed. The next row's loads
// are issued one row ahead.
constexpr int kCols = 29, kFieldThreads = 128;

__device__ __forceinline__ int wrap_col(int i, int nx)
{
    if (i < 0) i += nx;
    while (i >= nx) i -= nx;       // a warp wider than the grid wraps more than once
    return i;
}

struct V3 {
    float x, y, z;
};
struct J3 {
    u64 x, y, z;
};
__device__ __forceinline__ V3 load3(const float* const F[3], size_t c, bool in)
{
    return in ? V3{__ldg(F[0] + c), __ldg(F[1] + c), __ldg(F[2] + c)} : V3{0.0f, 0.0f, 0.0f};
}
__device__ __forceinline__ J3 load3(const u64* const J[3], size_t c, bool in)
{
    return in ? J3{__ldg(J[0] + c), __ldg(J[1] + c), __ldg(J[2] + c)} : J3{0, 0, 0};
}
__device__ __forceinline__ float right(float v) { return __shfl_down_sync(0xffffffffu, v, 1); }
__device__ __forceinline__ float left(float v) { return __shfl_up_sync(0xffffffffu, v, 1); }

// The update of rows k0 .. k1 - 1 of the columns i0 .. i0 + kCols - 1 by one warp. Lane l holds column
// i0 + l - 1; lanes 1 .. kCols write. At row r the warp knows E(r), E(r + 1) (old), takes B(r) to the
// half step, E(r) to the new step, and finishes row r - 1 (its second half step of B needs the new
// E(r)). Rows 0 and nz of the new tangential E follow from the new row beside them (Mur).
__device__ __forceinline__ void field_rows(const FieldArgs& f, int i0, int k0, int k1, float a0, float a1)
{
    const int nx = f.nx, nz = f.nz, lane = threadIdx.x & 31;
    const int gi = wrap_col(i0 + lane - 1, nx);
    const bool own = lane >= 1 && lane <= kCols && i0 + lane - 1 < nx;
    const float* const Ep[3] = {f.F[0], f.F[1], f.F[2]};
    const float* const Bp[3] = {f.F[3], f.F[4], f.F[5]};
    const float antc = f.antc[gi], ants = f.ants[gi];
    const int r0 = k0 > 0 ? k0 - 1 : 0;
    size_t c = (size_t)r0 * nx + gi;
    V3 e = load3(Ep, c, true), en = load3(Ep, c + nx, true);      // old E of rows r, r + 1
    V3 bl = load3(Bp, c, true);
    J3 jl = load3(f.J, c, true);
    V3 ep = {0, 0, 0}, bp = {0, 0, 0}, np = {0, 0, 0};           // row r - 1: old E, half-step B, new E
    for (int r = r0; r <= k1; r++, c += nx) {
        if (r > nz) {
            // the wall row nz (the last segment): its B is finished below from np alone
            break;
        }
        // one row ahead
        const V3 e2 = load3(Ep, c + 2 * (size_t)nx, r + 2 <= nz && r < k1);
        const V3 b2 = load3(Bp, c + nx, r + 1 <= nz && r < k1);
        const J3 j2 = load3(f.J, c + nx, r + 1 <= nz && r < k1);
        // B(r) to the half step (Bx, By have nz rows)
        V3 b = bl;
        const float eyr = right(e.y), ezr = right(e.z);
        if (r < nz) {
            b.x += f.h_b * (en.y - e.y);
            b.y += f.h_b * ((ezr - e.z) - (en.x - e.x));
        }
        b.z -= f.h_b * (eyr - e.y);
        // E(r) to the new step
        const float byl = left(b.y), bzl = left(b.z);
        V3 n = e;
        if (r > 0 && r < nz) {
            float v = e.x - f.h_e * (b.y - bp.y) - f.cj * (float)(long long)jl.x;
            if (r == f.k_ant) v += antc * a0 + ants * a1;
            n.x = v;
            n.y = e.y + f.h_e * ((b.x - bp.x) - (b.z - bzl)) - f.cjy * (float)(long long)jl.y;
        }
        if (r < nz) n.z += f.h_e * (b.y - byl) - f.cj * (float)(long long)jl.z;
        if (r == 1) {
            np.x = e.x + f.mur * (n.x - ep.x);
            np.y = e.y + f.mur * (n.y - ep.y);
        } else if (r == nz) {
            n.x = ep.x + f.mur * (np.x - e.x);
            n.y = ep.y + f.mur * (np.y - e.y);
        }
        if (r == f.k_flux && r >= k0 && r < k1) {            // uniform over the warp
            // (Ex By - Ey Bx) at the half step
            float s = own ? 0.25f * ((e.x + n.x) * (bp.y + b.y) - (e.y + n.y) * (bp.x + b.x)) : 0.0f;
            for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
            if (lane == 0 && s != 0.0f) atomicAdd(f.flux, (double)s);
        }
        // finish row r - 1
        const float npyr = right(np.y), npzr = right(np.z);
        if (r > k0 && own) {
            const size_t q = c - nx;
            f.G[0][q] = np.x;
            f.G[1][q] = np.y;
            f.G[2][q] = np.z;
            f.G[3][q] = bp.x + f.h_b * (n.y - np.y);
            f.G[4][q] = bp.y + f.h_b * ((npzr - np.z) - (n.x - np.x));
            f.G[5][q] = bp.z - f.h_b * (npyr - np.y);
        }
        // the next step's currents and node density
        if (r >= k0 && r < k1 && own) {
            f.Z[0][c] = 0;
            f.Z[1][c] = 0;
            f.Z[2][c] = 0;
            f.rho_next[c] = f.rho[c];
        }
        ep = e;
        bp = b;
        np = n;
        e = en;
        en = e2;
        bl = b2;
        jl = j2;
    }
    if (k1 == nz + 1) {
        const float npyr = right(np.y);
        if (own) {
            const size_t q = (size_t)nz * nx + gi;
            f.G[0][q] = np.x;
            f.G[1][q] = np.y;
            f.G[2][q] = np.z;
            f.G[3][q] = bp.x;
            f.G[4][q] = bp.y;
            f.G[5][q] = bp.z - f.h_b * (npyr - np.y);
        }
    }
}

// Rows per segment. A warp's walk is serial (each row waits for its loads, ~0.7 us), while the row and
// a half that every segment repeats comes from L2: short segments win on every grid (2048^2: 97 us
// at 4 rows, 101 at 8, 99 at 16, 102 at 64; 403 x 311: 10.3, 12.3, 22, 82; with the events' ~3 us), and two
// rows where the grid gives under four warps per SM (64^2: 21.4 -> 19.4 us per step). The last segment takes the remainder (at
// least seg rows: the wall row needs the row beside it).
static int field_segment(const Ctx& c)
{
    return (int64_t)((c.nx + kCols - 1) / kCols) * ((c.nz + 1) / 4) < 4 * (int64_t)c.nsm ? 2 : 4;
}
__host__ __device__ inline int field_segments(int nz, int seg) { return (nz + 1) / seg; }     // nz >= 4

__device__ __forceinline__ void field_item(const FieldArgs& f, int item, float a0, float a1)
{
    const int nseg = field_segments(f.nz, f.seg), col = item / nseg, s = item - col * nseg;
    if (col * kCols >= f.nx) return;
    field_rows(f, col * kCols, s * f.seg, s + 1 == nseg ? f.nz + 1 : (s + 1) * f.seg, a0, a1);
}
static int field_blocks(const FieldArgs& f)
{
    const int items = (f.nx + kCols - 1) / kCols * field_segments(f.nz, f.seg), w = kFieldThreads / 32;
    return (items + w - 1) / w;
}

// The first block evaluates the antenna scalars of the next step (it starts first: on the smallest grids the other
// blocks take as long).
__global__ void __launch_bounds__(kFieldThreads, 8)
    k_fields(const __grid_constant__ FieldArgs f, const __grid_constant__ AntennaParams ap, long long next, float* ant_next)
{
    if (blockIdx.x == 0) {
        if (threadIdx.x == 0) antenna_scalars(ap, next, ant_next);
        return;
    }
    field_item(f, (int)((blockIdx.x - 1) * (kFieldThreads / 32) + threadIdx.x / 32), f.ant[0], f.ant[1]);
}

// All slabs of a batch: blockIdx.x runs over every slab's blocks, slab s owning blocks rb[s] ..
// rb[s + 1] - 1; every slab's arguments travel in the launch's parameter block. The antenna scalars
// of this step were written by the previous one (or with the prepare kernel): the last block evaluates
// the next step's into the other half of the array and advances the step counters.
__global__ void __launch_bounds__(kFieldThreads, 8)
    k_fields_batch(const __grid_constant__ FieldBatch P, const AntennaParams* ap, long long* step, float* ant_next)
{
    const int g = (int)blockIdx.x;
    if (g == P.rb[P.n]) {
        const int s = threadIdx.x;
        if (s < P.n) {
            const long long n = step[s] + 1;
            step[s] = n;
            antenna_scalars(ap[s], n, ant_next + 2 * s);
        }
        return;
    }
    int s = 0;
    while (s + 1 < P.n && P.rb[s + 1] <= g) s++;
    const FieldArgs& f = P.f[s];
    field_item(f, (g - P.rb[s]) * (kFieldThreads / 32) + (int)threadIdx.x / 32, f.ant[0], f.ant[1]);
}

// antenna scalars of the step a simulation, or each slab of a batch, is at
__global__ void k_antenna(const __grid_constant__ AntennaParams p, long long step, float* ant)
{
    antenna_scalars(p, step, ant);
}
__global__ void k_antenna_batch(const AntennaParams* p, const long long* step, float* ant, int nslab)
{
    const int s = threadIdx.x;
    if (s < nslab) antenna_scalars(p[s], step[s], ant + 2 * s);
}

// ---- one set of grids ---------------------------------------------------------------------
// States that leave no room for the second set (kTwinBytes) take the update in place, in three passes over the nodes: B
// half, E with the current and the antenna, B half. The first one keeps the tangential E of the rows beside the walls for
// the absorbing condition. 172 bytes per node with the copy and clear in front, and the same bits.
__global__ void k_half_B(const __grid_constant__ FieldArgs f, int save)
{
    const int nx = f.nx, nz = f.nz, i = blockIdx.x * blockDim.x + threadIdx.x, k = blockIdx.y;
    if (i >= nx) return;
    const int ip = i + 1 == nx ? 1 - nx : 1;
    const size_t c = (size_t)k * nx + i;
    const float *Ex = f.G[0], *Ey = f.G[1], *Ez = f.G[2];
    const float ey = Ey[c];
    if (k < nz) {
        const size_t u = c + nx;
        f.G[3][c] += f.h_b * (Ey[u] - ey);
        f.G[4][c] += f.h_b * ((Ez[c + ip] - Ez[c]) - (Ex[u] - Ex[c]));
    }
    f.G[5][c] -= f.h_b * (Ey[c + ip] - ey);
    const int slot = k == 0 ? 0 : k == 1 ? 1 : k == nz - 1 ? 2 : k == nz ? 3 : -1;
    if (save && slot >= 0) {
        f.save[slot * nx + i] = Ex[c];
        f.save[(4 + slot) * nx + i] = ey;
    }
}

// new Ex / Ey of an interior node from its old value
__device__ __forceinline__ float ex_new(const FieldArgs& f, size_t c, int i, int k, float old)
{
    float v = old - f.h_e * (f.G[4][c] - f.G[4][c - f.nx]) - f.cj * (float)(long long)f.J[0][c];
    if (k == f.k_ant) v += f.antc[i] * f.ant[0] + f.ants[i] * f.ant[1];
    return v;
}
__device__ __forceinline__ float ey_new(const FieldArgs& f, size_t c, int i, float old)
{
    const int im = i == 0 ? f.nx - 1 : -1;
    return old + f.h_e * ((f.G[3][c] - f.G[3][c - f.nx]) - (f.G[5][c] - f.G[5][c + im])) - f.cjy * (float)(long long)f.J[1][c];
}

__global__ void k_E(const __grid_constant__ FieldArgs f)
{
    const int nx = f.nx, nz = f.nz, i = blockIdx.x * blockDim.x + threadIdx.x, k = blockIdx.y;
    float s = 0.0f;              // on the flux row: (Ex By - Ey Bx) at the half step
    if (i < nx) {
        const size_t c = (size_t)k * nx + i;
        if (k > 0 && k < nz) {
            const float ex0 = f.G[0][c], ey0 = f.G[1][c];
            const float ex1 = ex_new(f, c, i, k, ex0), ey1 = ey_new(f, c, i, ey0);
            f.G[0][c] = ex1;
            f.G[1][c] = ey1;
            if (k == f.k_flux)
                s = 0.25f * ((ex0 + ex1) * (f.G[4][c - nx] + f.G[4][c]) - (ey0 + ey1) * (f.G[3][c - nx] + f.G[3][c]));
        } else {
            // a wall row (Mur): its old value, and the row beside it before and after this step
            const int w = k == 0 ? 0 : 3, b = k == 0 ? 1 : 2, kb = k == 0 ? 1 : nz - 1;
            const size_t cb = (size_t)kb * nx + i;
            const float x0 = f.save[w * nx + i], x1 = f.save[b * nx + i];
            const float y0 = f.save[(4 + w) * nx + i], y1 = f.save[(4 + b) * nx + i];
            f.G[0][c] = x1 + f.mur * (ex_new(f, cb, i, kb, x1) - x0);
            f.G[1][c] = y1 + f.mur * (ey_new(f, cb, i, y1) - y0);
        }
        if (k < nz) {
            const int im = i == 0 ? nx - 1 : -1;
            f.G[2][c] += f.h_e * (f.G[4][c] - f.G[4][c + im]) - f.cj * (float)(long long)f.J[2][c];
        }
    }
    if (k != f.k_flux) return;
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if ((threadIdx.x & 31) == 0 && s != 0.0f) atomicAdd(f.flux, (double)s);
}

void launch_fields_one_set(const FieldArgs& f, cudaStream_t st)
{
    const dim3 block(256), grid((f.nx + 255) / 256, f.nz + 1);
    k_half_B<<<grid, block, 0, st>>>(f, 1);
    k_E<<<grid, block, 0, st>>>(f);
    k_half_B<<<grid, block, 0, st>>>(f, 0);
}

__global__ void k_step_done(long long* step, int n)
{
    if ((int)threadIdx.x < n) step[threadIdx.x]++;
}

void launch_step_done(long long* step_dev, int n, cudaStream_t st) { k_step_done<<<1, 64, 0, st>>>(step_dev, n); }

// each slab's first block (rb[n] = the total)
void field_row_blocks(FieldBatch& P)
{
    P.rb[0] = 0;
    for (int s = 0; s < P.n; s++) P.rb[s + 1] = P.rb[s] + field_blocks(P.f[s]);
}

AntennaParams make_antenna_params(const Ctx& c)
{
    AntennaParams p;
    p.on = c.cfg.laser_profile != PIC_LASER_NONE;
    p.dt = c.dt;
    p.t_ant = c.t_ant;
    p.tau_fwhm = c.cfg.tau_fwhm > 0 ? c.cfg.tau_fwhm : 1.0;
    p.omega = c.omega;
    p.coef = 2.0 * (kC * c.dt / c.cfg.dx) * c.E0;
    return p;
}

// The arguments of the field update that follows the particle kernel: density rho[cur] and currents J
// just deposited, fields F read and Fn written, Jn cleared for the next step.
FieldArgs make_field_args(const Ctx& c)
{
    FieldArgs f;
    f.nx = c.nx;
    f.nz = c.nz;
    f.k_ant = c.k_ant;
    f.seg = field_segment(c);
    f.h_b = (float)(0.5 * c.dt / c.cfg.dx);
    f.h_e = (float)(kC * kC * c.dt / c.cfg.dx);
    f.cj = (float)(kQe * c.w / (8589934592.0 * c.cfg.dx * kEps0));
    f.cjy = (float)(kQe * c.w * kC * c.dt / (6.0 * ldexp(1.0, 32 + c.jy_bits) * c.cfg.dx * c.cfg.dx * kEps0));
    const double cdt = kC * c.dt;
    f.mur = (float)((cdt - c.cfg.dx) / (cdt + c.cfg.dx));
    for (int q = 0; q < 6; q++) f.F[q] = c.F[q];
    for (int q = 0; q < 6; q++) f.G[q] = c.Fn[q] ? c.Fn[q] : c.F[q];
    f.save = c.mur_save;
    for (int q = 0; q < 3; q++) f.J[q] = c.J[q];
    for (int q = 0; q < 3; q++) f.Z[q] = c.Jn[q];
    f.rho = c.rho[c.cur];
    f.rho_next = c.rho[1 - c.cur];
    f.antc = c.ant_c;
    f.ants = c.ant_s;
    f.ant = c.ant + 2 * (c.step & 1);
    f.k_flux = c.k_ant - 1 >= 1 ? c.k_ant - 1 : -1;
    f.flux = c.red_out + 5;
    return f;
}

void launch_fields(Ctx& c, cudaStream_t st, int64_t step, int64_t* launches)
{
    const FieldArgs f = make_field_args(c);
    if (!c.Fn[0]) {
        launch_fields_one_set(f, st);
        if (launches) *launches += 3;
        return;
    }
    k_fields<<<1 + field_blocks(f), kFieldThreads, 0, st>>>(f, make_antenna_params(c), (long long)step + 1,
                                                            c.ant + 2 * ((step + 1) & 1));
    swap_fields(c);
    if (launches) *launches += 1;
}

void launch_antenna(const Ctx& c, cudaStream_t st, int64_t step)
{
    k_antenna<<<1, 1, 0, st>>>(make_antenna_params(c), (long long)step, c.ant + 2 * (step & 1));
}

void launch_antenna_batch(const AntennaParams* ap_dev, const long long* step_dev, float* ant, int n, cudaStream_t st)
{
    k_antenna_batch<<<1, 64, 0, st>>>(ap_dev, step_dev, ant, n);
}

void launch_fields_batch(const FieldBatch& P, const AntennaParams* ap_dev, long long* step_dev, float* ant_next,
                         cudaStream_t st)
{
    k_fields_batch<<<P.rb[P.n] + 1, kFieldThreads, 0, st>>>(P, ap_dev, step_dev, ant_next);
}

}  // namespace gbpic
