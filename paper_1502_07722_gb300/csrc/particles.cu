// The particle kernel of one PIC step (paper, the PIC-cycle paragraph and Fig. 1B):
// for every macroparticle -- gather E, B (Lorentz force) and the node density with its gradient
// (pair-potential force, Eqs. 1-3) -> relativistic Boris push -> move -> charge-conserving
// current deposition (Esirkepov, fixed point) -> node density at the new position.
//
// Work decomposition (GB300):
//  * one CTA takes one work item at a time: a tile of T x T cells (particles are sorted into tiles), or
//    a part of a tile when tiles are few; the items are listed after each sort (k_work_items);
//  * the CTA stages a window of (T + 2M + 3)^2 nodes in shared memory: the six field
//    components and the pair density n / n0 in FP32, components of one Yee stagger side by side
//    (one 64-bit load per corner fetches two of them);
//  * thread t of the CTA (128 threads) takes the item's records t, t + 128, ... straight from global
//    memory (coalesced loads and stores, no block barrier), in warps aligned to 32 records; the
//    position of its next record is loaded one iteration ahead. The cell sort stores each block of a
//    tile's cell-ordered particles as a 32-row matrix, column by column, so the lanes of a warp hold
//    particles of neighbouring cells, whose deposits go to distinct nodes that share cache sectors;
//  * deposits (current, node-density change) are exact 64-bit integer reductions straight into
//    global memory: fire-and-forget on the SM, native in L2. Measured against exact sums in the
//    shared-memory window (32-bit (lo, hi) pairs whose low-word atomic must return the old value
//    for the carry) they are slightly faster and free 17 KB of shared memory per CTA;
//  * the node density is updated incrementally: the next density starts as a copy of the
//    current one and each pair particle adds S(new) - S(old) only when its fixed-point position
//    changed. Ions move ~1e-7 cells per step against a quantum of 1.5e-5 cells, so most of them
//    deposit nothing; the integer result equals a full re-deposit bit for bit;
//  * a particle that stays in its cell (almost all of them) deposits on the four corners of the
//    cell (an electron without per-term zero tests: its terms are almost never zero); a particle
//    that crossed a cell edge uses the 3 x 3 Esirkepov stencil (rare); a particle that drifted
//    beyond the margin since the last sort gathers from global memory (rare);
//  * the code is specialised per species kind (ion, electron, neutral atom) and per potential
//    and lattice, so no per-particle branch tests a species or potential property; Eq. (3) as
//    printed evaluates both in-plane axes at once with packed FP32x2 arithmetic.
// Integer sums make every result independent of the order of the additions.
#include <atomic>

#include "pic_device.cuh"

namespace gbpic {

constexpr int kMargin = 2;              // cells a particle may drift out of its tile between sorts
constexpr int kBlock = 128;             // threads per CTA
// Resident CTAs: with fields 9 (56 registers; 8 at 64: 1.74 against 1.70 ms per launch on the 2048^2
// slab), the transport stage 8 (9: 0.129 against 0.116 ms on the crater slab). The Morse, altered, HCP and embedded-atom
// instances spill up to 24 bytes (embedded atom 72) at 56 registers and still take 14 to 19 % less per step than the 64
// registers and 8 CTAs of the kernel before (33.5 M particles, ms a step: Morse 0.634 -> 0.533, altered 0.589 -> 0.497, HCP 0.610 ->
// 0.536, embedded atom 0.936 -> 0.805; tiles of 20 cells 0.648 -> 0.559, 0.611 -> 0.524, 0.649 -> 0.563, 1.026 -> 0.784).
constexpr int kCtasPerSm = 9;
constexpr int kCtasPerSmAtoms = 8;
constexpr int kMinChunk = 512;
constexpr int kWin = 16 + 2 * kMargin + 3;  // window edge of the 16-cell tile (compiled-in instances)
// The batched kernel reads each slab's arguments from a constant-memory table with a run-time index:
// every use is an indexed constant load into a register, so it needs more registers than the single
// kernel for the same code: 8 CTAs (64 registers) on the 16-slab sweep 1.37 ms per launch, 7 CTAs (72) 1.42,
// 9 CTAs (56) 1.73.
constexpr int kCtasPerSmBatch = 8;


__device__ __forceinline__ int wrap_any(int i, int nx)
{
    int r = i % nx;
    return r < 0 ? r + nx : r;
}

// The tile's window in shared memory. Field instances keep the components that share a Yee
// stagger side by side, so one 64-bit load fetches both at a corner: (Ex, Bz) at (i + 1/2, k),
// (Ez, Bx) at (i, k + 1/2), (Ey, n / n0) at (i, k), By at (i + 1/2, k + 1/2). Transport
// instances keep n / n0 alone.
struct Window {
    float2* exbz;
    float2* ezbx;
    float2* eyn;
    float* by;
    float* nh;
    int ox1, oz, W;           // grid column of the window's second column, grid row of its first row
};

// bilinear sum of the corners (c00, c10, c01, c11) of a stagger pair, both components at once
__device__ __forceinline__ float2 bilerp2(float2 c00, float2 c10, float2 c01, float2 c11, float2 gx, float2 wx,
                                          float2 gz, float2 wz)
{
    const float2 b0 = __ffma2_rn(wx, c10, __fmul2_rn(gx, c00));
    const float2 b1 = __ffma2_rn(wx, c11, __fmul2_rn(gx, c01));
    return __ffma2_rn(wz, b1, __fmul2_rn(gz, b0));
}

__device__ __forceinline__ float bilerp1(float c00, float c10, float c01, float c11, float gx, float wx, float gz,
                                         float wz)
{
    const float b0 = __fmaf_rn(wx, c10, __fmul_rn(gx, c00));
    const float b1 = __fmaf_rn(wx, c11, __fmul_rn(gx, c01));
    return __fmaf_rn(wz, b1, __fmul_rn(gz, b0));
}

__device__ __forceinline__ void red64g(u64* p, long long v)
{
    if (v != 0) atomicAdd(p, (u64)v);
}


// exact cell -> (i, k) (magic_div; a multiply-high by floor(2^32 / nx) needs a correction)
__device__ __forceinline__ void split_cell(int cell, const StepArgs& a, int& i, int& k)
{
    k = (int)(__umulhi((unsigned)cell, a.nx_magic) >> a.nx_shift);
    i = cell - k * a.nx;
}

// Rare path: fields and node density straight from global memory (particle outside the window).
__device__ __noinline__ void gather_global(const float* F0, const float* F1, const float* F2, const float* F3,
                                           const float* F4, const float* F5, const u64* rho, int nx, int nz,
                                           float rho_s, int full, int pair, int i, int k, float fx, float fz,
                                           float* g)
{
    if (full) {
        g[0] = gather_field(F0, nx, nz, i, k, fx, fz, 1, 0);
        g[1] = gather_field(F1, nx, nz, i, k, fx, fz, 0, 0);
        g[2] = gather_field(F2, nx, nz, i, k, fx, fz, 0, 1);
        g[3] = gather_field(F3, nx, nz, i, k, fx, fz, 0, 1);
        g[4] = gather_field(F4, nx, nz, i, k, fx, fz, 1, 1);
        g[5] = gather_field(F5, nx, nz, i, k, fx, fz, 1, 0);
    }
    if (pair) gather_density(rho, nx, nz, rho_s, i, k, fx, fz, g[6], g[7], g[8]);
}

// Rare path: 3 x 3 Esirkepov stencil and new node density with global atomics. (X, Z) are
// global fixed-point coordinates; X1 may lie outside [0, nx 2^16) (periodic x).
__device__ __noinline__ void deposit_global(u64* rho_next, u64* Jx, u64* Jy, u64* Jz, int nx, int X0, int Z0,
                                            int X1, int Z1, int jsign, int V, int pair)
// pair != 0: the node density changes by S(X1, Z1) - S(X0, Z0)
{
    const int bx = min(X0, X1) >> kQBits, bz = min(Z0, Z1) >> kQBits;
    int S0x[3], S1x[3], S0z[3], S1z[3];
    hat3(X0 - bx * kQOne, S0x[0], S0x[1], S0x[2]);
    hat3(X1 - bx * kQOne, S1x[0], S1x[1], S1x[2]);
    hat3(Z0 - bz * kQOne, S0z[0], S0z[1], S0z[2]);
    hat3(Z1 - bz * kQOne, S1z[0], S1z[1], S1z[2]);
    const long long sg = jsign;
    for (int b = 0; b < 3; b++) {
        const size_t row = (size_t)(bz + b) * nx;
        if (jsign != 0) {
            const long long wz = (long long)(S0z[b] + S1z[b]);
            long long acc = 0;
            for (int c = 0; c < 2; c++) {
                acc -= (long long)(S1x[c] - S0x[c]) * wz;
                if (acc != 0) atomicAdd(Jx + row + wrap_any(bx + c, nx), (u64)(sg * acc));
            }
        }
        for (int c = 0; c < 3; c++) {
            const size_t g = row + wrap_any(bx + c, nx);
            if (jsign != 0 && V != 0) {
                const long long w6 = 2LL * S0x[c] * S0z[b] + (long long)S1x[c] * S0z[b] + (long long)S0x[c] * S1z[b] +
                                     2LL * S1x[c] * S1z[b];
                if (w6 != 0) atomicAdd(Jy + g, (u64)(sg * V * w6));
            }
            if (pair) {
                const long long r = (long long)S1x[c] * S1z[b] - (long long)S0x[c] * S0z[b];
                if (r != 0) atomicAdd(rho_next + g, (u64)r);
            }
        }
    }
    if (jsign != 0) {
        for (int c = 0; c < 3; c++) {
            const long long wx = (long long)(S0x[c] + S1x[c]);
            long long acc = 0;
            for (int b = 0; b < 2; b++) {
                acc -= (long long)(S1z[b] - S0z[b]) * wx;
                if (acc != 0) atomicAdd(Jz + (size_t)(bz + b) * nx + wrap_any(bx + c, nx), (u64)(sg * acc));
            }
        }
    }
}

// Species kinds the particle code is specialised for.
enum Kind { kIon = 0, kElectron = 1, kAtom = 2 };

// Fixed-point offset as the bit pattern of rint(f 2^16) + 1.5 2^23: one FMA rounds to the integer (half
// to even, as the conversion would) and the integer sits in the low bits. Differences of two patterns
// are differences of the offsets.
constexpr int kQBias = 0x4B400000;
__device__ __forceinline__ int qbits(float f) { return __float_as_int(__fmaf_rn(f, 65536.0f, 12582912.0f)); }

// One particle of record p (position already loaded): its momenta are read, the record advanced one
// step and written back before its deposits, so that little state is live during them.
//   kIon:      Lorentz force + pair force, current (charge +e), node density
//   kElectron: Lorentz force, current (charge -e)
//   kAtom:     pair force, node density (neutral atoms of the transport stage)
// WC: the window edge when it is compiled in (0: the run-time W).
// The kernel is bound by instruction issue, so a particle that stays in its cell (almost every one)
// takes the short way: no floor, no wall test, no new cell index, and its cell is not written (44
// instead of 48 bytes move per particle). With the window edge compiled in and the one-instruction
// fixed-point rounding: 424 -> 355 M warp instructions per launch on the 1024^2 slab of 33.5 M
// particles; 1.90 -> 1.72 ms on the 2048^2 slab, 1.92 -> 1.62 ms on the 16-slab sweep, 0.122 -> 0.114
// ms on the crater slab, 0.235 -> 0.195 ms with the embedded-atom form on 7.7 M atoms.
template <int KIND, int POT, int WC>
__device__ __forceinline__ void process_particle(const StepArgs& a, const Species& S, const Window& w, int p,
                                                 const int cell0, const float fx, const float fz)
{
    constexpr bool kFields = KIND != kAtom;
    constexpr bool kPair = KIND != kElectron;
    constexpr bool kCurrent = KIND != kAtom;
    constexpr int kSign = KIND == kElectron ? -1 : 1;
    const int nx = a.nx, nz = a.nz, W = WC ? WC : w.W;
    float ux = S.a.ux[p], uy = S.a.uy[p], uz = S.a.uz[p];
    int i, k;
    split_cell(cell0, a, i, k);

    // window coordinates (w.ox1 lies in [0, nx): a column left of it is one period further on). A particle is
    // inside from the window's second column on, so the period is taken there: on a grid narrower than the window
    // its first column is the same as a later one.
    unsigned lx1 = (unsigned)(i - w.ox1);
    lx1 = min(lx1, lx1 + (unsigned)nx);
    const int lz = k - w.oz;
    const bool inwin = lx1 < (unsigned)(W - 3) && (unsigned)(lz - 1) < (unsigned)(W - 3);

    float kx = 0.f, ky = 0.f, kz = 0.f, bx = 0.f, by = 0.f, bz = 0.f;
    float n = 0.f, dnx = 0.f, dnz = 0.f;
    if (inwin) {
        const int base = lz * W + (int)lx1 + 1;
        const float gx = 1.0f - fx, gz = 1.0f - fz;
        if (kFields) {
            // four stagger patterns: (0,0) Ey, n; (1/2,0) Ex, Bz; (0,1/2) Ez, Bx; (1/2,1/2) By
            const bool ux_ = fx >= 0.5f, uz_ = fz >= 0.5f;
            const int ox_ = ux_ ? 0 : -1, oz_ = uz_ ? 0 : -W;
            const float hx = ux_ ? fx - 0.5f : fx + 0.5f, hz = uz_ ? fz - 0.5f : fz + 0.5f;
            const float ghx = 1.0f - hx, ghz = 1.0f - hz;
            // the two components of a stagger pair share their weights: one packed FP32x2 bilinear
            // sum interpolates both. Every operation here is an explicit intrinsic (no contraction
            // left to the compiler), so the single and the batched kernel round alike.
            const float2 gx2 = make_float2(gx, gx), fx2 = make_float2(fx, fx);
            const float2 gz2 = make_float2(gz, gz), fz2 = make_float2(fz, fz);
            {
                const float2* q = w.eyn + base;
                const float2 c00 = q[0], c10 = q[1], c01 = q[W], c11 = q[W + 1];
                if (kPair) {
                    const float2 r = bilerp2(c00, c10, c01, c11, gx2, fx2, gz2, fz2);
                    ky = __fmul_rn(S.e_kick, r.x);
                    n = r.y;
                    dnx = __fmaf_rn(fz, __fsub_rn(c11.y, c01.y), __fmul_rn(gz, __fsub_rn(c10.y, c00.y)));
                    dnz = __fmaf_rn(fx, __fsub_rn(c11.y, c10.y), __fmul_rn(gx, __fsub_rn(c01.y, c00.y)));
                } else {
                    ky = __fmul_rn(S.e_kick, bilerp1(c00.x, c10.x, c01.x, c11.x, gx, fx, gz, fz));
                }
            }
            {
                const float2* q = w.exbz + base + ox_;
                const float2 r = bilerp2(q[0], q[1], q[W], q[W + 1], make_float2(ghx, ghx), make_float2(hx, hx), gz2, fz2);
                kx = __fmul_rn(S.e_kick, r.x);
                bz = r.y;
            }
            {
                const float2* q = w.ezbx + base + oz_;
                const float2 r = bilerp2(q[0], q[1], q[W], q[W + 1], gx2, fx2, make_float2(ghz, ghz), make_float2(hz, hz));
                kz = __fmul_rn(S.e_kick, r.x);
                bx = r.y;
            }
            {
                const float* q = w.by + base + ox_ + oz_;
                by = bilerp1(q[0], q[1], q[W], q[W + 1], ghx, hx, ghz, hz);
            }
        } else if (kPair) {
            const float* q = w.nh + base;
            const float n00 = q[0], n10 = q[1], n01 = q[W], n11 = q[W + 1];
            n = gz * (gx * n00 + fx * n10) + fz * (gx * n01 + fx * n11);
            dnx = gz * (n10 - n00) + fz * (n11 - n01);
            dnz = gx * (n01 - n00) + fx * (n11 - n10);
        }
    } else {
        float g[9];
        gather_global(a.F[0], a.F[1], a.F[2], a.F[3], a.F[4], a.F[5], a.rho_cur, nx, nz, a.rho_s, kFields ? 1 : 0,
                      kPair ? 1 : 0, i, k, fx, fz, g);
        if (kFields) {
            kx = S.e_kick * g[0]; ky = S.e_kick * g[1]; kz = S.e_kick * g[2];
            bx = g[3]; by = g[4]; bz = g[5];
        }
        if (kPair) { n = g[6]; dnx = g[7]; dnz = g[8]; }
    }
    if (kPair) {
        float pfx, pfz;
        if (POT == kPotLJ) lj_pair_xz2(n, dnx, dnz, a.h_coef, pfx, pfz);
        else pair_force_xz<false, POT>(n, dnx, dnz, a.h_coef, a.pot_mode, a.c_att, a.s_rep, pfx, pfz, a.eam);
        kx += S.p_kick * pfx;
        kz += S.p_kick * pfz;
    }
    // relativistic Boris: half kick, rotation, half kick
    ux += kx; uy += ky; uz += kz;
    if (kFields) {
        const float rot = S.b_rot * rsqrtf(1.0f + ux * ux + uy * uy + uz * uz);
        const float tx = rot * bx, ty = rot * by, tz = rot * bz;
        const float s = 2.0f * fast_rcp(1.0f + tx * tx + ty * ty + tz * tz);
        const float px = ux + (uy * tz - uz * ty);
        const float py = uy + (uz * tx - ux * tz);
        const float pz = uz + (ux * ty - uy * tx);
        ux += s * (py * tz - pz * ty);
        uy += s * (pz * tx - px * tz);
        uz += s * (px * ty - py * tx);
    }
    ux += kx; uy += ky; uz += kz;

    // move (in-plane), cells per step = u c dt / (gamma dx)
    const float step = a.cdt_dx * rsqrtf(1.0f + ux * ux + uy * uy + uz * uz);
    const float dxi = __fmul_rn(ux, step), dze = __fmul_rn(uz, step);
    float nfx = __fadd_rn(fx, dxi), nfz = __fadd_rn(fz, dze);
    if (!(nfx >= 0.0f && nfx < 1.0f && nfz >= 0.0f && nfz < 1.0f && fabsf(dze) < 1.0f)) {
        // leaves its cell, reflects off a wall, or moved too far (or is not finite)
        if (!(fabsf(dxi) < 1.0f && fabsf(dze) < 1.0f)) {
            // refused: the particle keeps its record (what it deposits is that of a particle at rest
            // in the plane with its old momenta)
            atomicOr(a.status, (isfinite(ux) && isfinite(uy) && isfinite(uz)) ? kErrMove : kErrNan);
            ux = S.a.ux[p];
            uy = S.a.uy[p];
            uz = S.a.uz[p];
            nfx = fx;
            nfz = fz;
        }
        int di = (int)floorf(nfx);
        nfx -= (float)di;
        if (nfx >= 1.0f) { nfx = 0.0f; di += 1; }
        int dk = 0;
        if (k == 0 && nfz < 0.0f) {                   // reflect off the wall z = 0
            nfz = -nfz; uz = -uz;
        } else if (k == nz - 1 && nfz >= 1.0f) {      // reflect off the wall z = nz
            nfz = 2.0f - nfz; uz = -uz;
        } else {
            dk = (int)floorf(nfz);
            nfz -= (float)dk;
            if (nfz >= 1.0f) { nfz = 0.0f; dk += 1; }
        }
        S.a.cell[p] = (k + dk) * nx + wrap_x(i + di, nx);
        S.a.fx[p] = nfx;
        S.a.fz[p] = nfz;
        S.a.ux[p] = ux;
        S.a.uy[p] = uy;
        S.a.uz[p] = uz;
        const int V = (kCurrent && fabsf(uy) >= a.jy_zero) ? jy_code(ux, uy, uz, a.jy_scale) : 0;
        deposit_global(a.rho_next, a.J[0], a.J[1], a.J[2], nx, i * kQOne + qoff(fx), k * kQOne + qoff(fz),
                       (i + di) * kQOne + qoff(nfx), (k + dk) * kQOne + qoff(nfz), kCurrent ? kSign : 0, V,
                       kPair ? 1 : 0);
        return;
    }
    S.a.fx[p] = nfx;
    S.a.fz[p] = nfz;
    S.a.ux[p] = ux;
    S.a.uy[p] = uy;
    S.a.uz[p] = uz;

    // stays in its cell: stencil = the four corners of the cell (global reductions)
    const int bx0 = qbits(fx), bx1 = qbits(nfx), bz0 = qbits(fz), bz1 = qbits(nfz);
    // |u_y| < 2^-(b+1) gives |beta_y| 2^b < 1/2, i.e. V = 0 without evaluating the code
    const int V = (kCurrent && fabsf(uy) >= a.jy_zero) ? kSign * jy_code(ux, uy, uz, a.jy_scale) : 0;
    const bool moved = bx1 != bx0 || bz1 != bz0;
    // nothing to deposit (most ions); an electron always moves in fixed point and almost always has
    // V != 0, so its reductions are issued without per-term tests (a zero term adds nothing)
    if (KIND != kElectron && !moved && V == 0) return;
    const int x0 = bx0 - kQBias, x1 = bx1 - kQBias, z0 = bz0 - kQBias, z1 = bz1 - kQBias;
    const int d1 = i + 1 == nx ? 1 - nx : 1;
    if (kCurrent) {
        const int dX = kSign * (bx1 - bx0), dZ = kSign * (bz1 - bz0);
        u64* jx = a.J[0] + cell0;
        u64* jy = a.J[1] + cell0;
        u64* jz = a.J[2] + cell0;
        // The out-of-plane weights are 6 W = A0 U0 + A1 U1 with A = 2^16 - x and U0 = 2 C0 + C1,
        // U1 = C0 + 2 C1 (C = 2^16 - z) on the lower-left corner, and likewise with x for A and z for
        // C on the others: two widening 32 x 32-bit products per corner.
        if (KIND == kElectron || dX != 0) {
            atomicAdd(jx, (u64)((long long)dX * (2 * kQOne - z0 - z1)));
            atomicAdd(jx + nx, (u64)((long long)dX * (z0 + z1)));
        }
        if (KIND == kElectron || dZ != 0) {
            atomicAdd(jz, (u64)((long long)dZ * (2 * kQOne - x0 - x1)));
            atomicAdd(jz + d1, (u64)((long long)dZ * (x0 + x1)));
        }
        if (KIND == kElectron || V != 0) {
            const int A0 = kQOne - x0, A1 = kQOne - x1, C0 = kQOne - z0, C1 = kQOne - z1;
            const int U0 = 2 * C0 + C1, U1 = C0 + 2 * C1, Z0 = 2 * z0 + z1, Z1 = z0 + 2 * z1;
            atomicAdd(jy, (u64)(V * ((long long)A0 * U0 + (long long)A1 * U1)));
            atomicAdd(jy + d1, (u64)(V * ((long long)x0 * U0 + (long long)x1 * U1)));
            atomicAdd(jy + nx, (u64)(V * ((long long)A0 * Z0 + (long long)A1 * Z1)));
            atomicAdd(jy + nx + d1, (u64)(V * ((long long)x0 * Z0 + (long long)x1 * Z1)));
        }
    }
    if (kPair && moved) {
        // weights are at most 2^16: each product is one 32 x 32 -> 64-bit multiply
        const int a0 = kQOne - x0, a1 = kQOne - x1, c0 = kQOne - z0, c1 = kQOne - z1;
        u64* r = a.rho_next + cell0;
        red64g(r, (long long)a1 * c1 - (long long)a0 * c0);
        red64g(r + d1, (long long)x1 * c1 - (long long)x0 * c0);
        red64g(r + nx, (long long)a1 * z1 - (long long)a0 * z0);
        red64g(r + nx + d1, (long long)x1 * z1 - (long long)x0 * z0);
    }
}

// start of part `sub` of `nsub` of the records p0 .. p1 - 1; inner boundaries lie on multiples of 32
__device__ __forceinline__ int part_start(int p0, int p1, int sub, int nsub)
{
    const int p = p0 + (int)(((long long)(p1 - p0) * sub) / nsub);
    return sub == 0 ? p0 : (sub == nsub ? p1 : max(p0, p & ~31));
}

// One work item: stage the tile's window, then advance the item's records of each species in storage
// order.
template <bool FULL, int POT, int WC>
__device__ __forceinline__ void run_item(const StepArgs& a, const WorkItem& item)
{
    extern __shared__ unsigned smem[];
    const int W = WC ? WC : a.W, WW = W * W;
    Window w;
    w.W = W;
    float* fbase = reinterpret_cast<float*>(smem);
    w.exbz = reinterpret_cast<float2*>(fbase);
    w.ezbx = reinterpret_cast<float2*>(fbase + 2 * WW);
    w.eyn = reinterpret_cast<float2*>(fbase + 4 * WW);
    w.by = fbase + 6 * WW;
    w.nh = fbase;

    const int t = item.tile, tx = t % a.ntx, tz = t / a.ntx;
    const int q0[2] = {item.p0[0], item.p0[1]}, q1[2] = {item.p1[0], item.p1[1]};
    const int ox = wrap_any(tx * a.T - kMargin - 1, a.nx);
    w.ox1 = ox + 1 == a.nx ? 0 : ox + 1;
    w.oz = tz * a.T - kMargin - 1;
    // stage the window: fields, pair density (wall rows doubled)
#pragma unroll
    for (int j = threadIdx.x; j < WW; j += kBlock) {
        const int b = j / W, c = j - b * W;
        int gx = ox + c;
        while (gx >= a.nx) gx -= a.nx;
        const int gz = w.oz + b;
        const int gn = min(max(gz, 0), a.nz);          // node rows 0..nz
        const int gh = min(max(gz, 0), a.nz - 1);      // half rows 0..nz-1 (edge rows repeat)
        const size_t in = (size_t)gn * a.nx + gx, ih = (size_t)gh * a.nx + gx;
        const long long r = (long long)__ldg(a.rho_cur + in);
        const float nh = a.rho_s * (float)((gn == 0 || gn == a.nz) ? 2 * r : r);
        if (FULL) {
            w.exbz[j] = make_float2(__ldg(a.F[0] + in), __ldg(a.F[5] + in));
            w.ezbx[j] = make_float2(__ldg(a.F[2] + ih), __ldg(a.F[3] + ih));
            w.eyn[j] = make_float2(__ldg(a.F[1] + in), nh);
            w.by[j] = __ldg(a.F[4] + ih);
        } else {
            w.nh[j] = nh;
        }
    }
    __syncthreads();
#pragma unroll
    for (int s = 0; s < 2; s++) {
        if (s >= (FULL ? 2 : 1)) break;
        const Species& S = a.sp[s];
        const int p0 = q0[s], p1 = q1[s];
        // the next record's position is loaded one iteration ahead (its first use is at the top
        // of the iteration); the momenta, first used after the gathers, are loaded in the iteration
        // Warps take aligned groups of 32 records: every access of a warp is one full 128-byte line. After
        // the first re-sort a tile starts anywhere: over steps 330-350 on the 2048^2 slab 1.919 -> 1.769 ms
        // per launch, 1.538 -> 1.468 in the sweep (aligned tiles, before it: 1.674 -> 1.696, the test).
        int ncell = 0;
        float nfx = 0.0f, nfz = 0.0f;
        const int first = (p0 & ~31) + (int)threadIdx.x;
        if (first < p1) {
            ncell = S.a.cell[first];
            nfx = S.a.fx[first];
            nfz = S.a.fz[first];
        }
        for (int p = first; p < p1; p += kBlock) {
            const int cell = ncell;
            const float fx = nfx, fz = nfz;
            if (p + kBlock < p1) {
                ncell = S.a.cell[p + kBlock];
                nfx = S.a.fx[p + kBlock];
                nfz = S.a.fz[p + kBlock];
            }
            if (p < p0) continue;
            if (s == 0) process_particle<FULL ? kIon : kAtom, POT, WC>(a, S, w, p, cell, fx, fz);
            else process_particle<kElectron, POT, WC>(a, S, w, p, cell, fx, fz);
        }
    }
    __syncthreads();
}

// The CTA's work items: the first is its block index, the others come from a ticket counter in the
// status words (dynamic assignment: the items take uneven times). atomicInc wraps the counter to 0
// after n draws, i.e. exactly when every CTA has drawn its last (failing) ticket, so every launch finds
// it at 0; with no more items than CTAs nothing is drawn.
__device__ __forceinline__ int next_item(const WorkItem* __restrict__ items, int n, unsigned* ticket, int first,
                                         WorkItem* buf, int* slot)
{
    if (threadIdx.x < 32) {
        int g = first;
        if (first < 0) {
            g = n;
            if (n > (int)gridDim.x) {
                if (threadIdx.x == 0) g = (int)(atomicInc(ticket, (unsigned)(n - 1)) + gridDim.x);
                g = __shfl_sync(0xffffffffu, g, 0);
            }
        }
        if (g < n && threadIdx.x < sizeof(WorkItem) / 4)
            reinterpret_cast<int*>(buf)[threadIdx.x] = reinterpret_cast<const int*>(items + g)[threadIdx.x];
        if (threadIdx.x == 0) *slot = g;
    }
    __syncthreads();
    return *slot;
}

template <bool FULL, int POT, int WC>
__global__ void __launch_bounds__(kBlock, FULL ? kCtasPerSm : kCtasPerSmAtoms)
    k_particles(const StepArgs a, const WorkItem* __restrict__ items, const int* __restrict__ nitems)
{
    __shared__ WorkItem item;
    __shared__ int slot;
    const int n = *nitems;
    for (int g = next_item(items, n, a.status + 2, (int)blockIdx.x, &item, &slot); g < n;
         g = next_item(items, n, a.status + 2, -1, &item, &slot))
        run_item<FULL, POT, WC>(a, item);
}

// Arguments of the simulations of a batch for the current step, in constant memory: the slab
// index is uniform across a CTA, so the kernel reads them as constant-bank operands like the
// single-simulation kernel reads its parameters. Uploaded (device to device) in front of each
// batched launch; two batches stepping at the same time on different streams would race on it.
constexpr int kMaxBatchSlabs = 48;
__constant__ StepArgs c_batch_args[kMaxBatchSlabs];

// All simulations of a batch in one persistent launch over one list of work items.
template <bool FULL, int POT, int WC>
__global__ void __launch_bounds__(kBlock, kCtasPerSmBatch)
    k_particles_batch(const WorkItem* __restrict__ items, const int* __restrict__ nitems)
{
    // one ticket counter for the whole batch: the first simulation's
    __shared__ WorkItem item;
    __shared__ int slot;
    const int n = *nitems;
    unsigned* ticket = c_batch_args[0].status + 2;
    for (int g = next_item(items, n, ticket, (int)blockIdx.x, &item, &slot); g < n;
         g = next_item(items, n, ticket, -1, &item, &slot))
        run_item<FULL, POT, WC>(c_batch_args[item.slab], item);
}

// Work items from the tiles' particle counts (rebuilt after a sort), appended to the list in tile order
// (neighbouring tiles run at about the same time and share lines of the grids in L2: a scrambled order
// took 1.735 instead of 1.695 ms on the 2048^2 slab). A tile of cnt particles is cut into
// round(cnt / chunk) parts, at least one, each with its share of both species; tiles without particles
// give none. One block: a scan over the tiles.
constexpr int kItemThreads = 1024;
__global__ void __launch_bounds__(kItemThreads) k_work_items(const int32_t* __restrict__ start0,
                                                            const int32_t* __restrict__ start1, int ntiles, int slab,
                                                            int chunk, WorkItem* items, int* nitems, int cap)
{
    __shared__ int sums[kItemThreads / 32], first[kItemThreads];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int base = *nitems;
    for (int t0 = 0; t0 < ntiles; t0 += kItemThreads) {
        const int t = t0 + (int)threadIdx.x;
        int parts = 0;
        if (t < ntiles) {
            const long long cnt = (long long)(start0[t + 1] - start0[t]) + (start1 ? start1[t + 1] - start1[t] : 0);
            if (cnt > 0) parts = max(1, (int)((cnt + chunk / 2) / chunk));
        }
        int scan = parts;
        for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(0xffffffffu, scan, o);
            if (lane >= o) scan += v;
        }
        if (lane == 31) sums[warp] = scan;
        __syncthreads();
        int before = 0, total = 0;
        for (int q = 0; q < kItemThreads / 32; q++) {
            if (q < warp) before += sums[q];
            total += sums[q];
        }
        // the items of these tiles, one per thread: its tile is the last one that starts at or before it
        first[threadIdx.x] = before + scan - parts;
        __syncthreads();
        for (int q = threadIdx.x; q < total && base + q < cap; q += kItemThreads) {     // always below cap
            int lo = 0, hi = kItemThreads - 1;
            while (lo < hi) {
                const int mid = (lo + hi + 1) >> 1;
                if (first[mid] <= q) lo = mid;
                else hi = mid - 1;
            }
            const int u = t0 + lo, sub = q - first[lo], n = (lo + 1 < kItemThreads ? first[lo + 1] : total) - first[lo];
            WorkItem w;
            w.tile = u;
            w.slab = slab;
            w.p0[0] = part_start(start0[u], start0[u + 1], sub, n);
            w.p1[0] = part_start(start0[u], start0[u + 1], sub + 1, n);
            w.p0[1] = start1 ? part_start(start1[u], start1[u + 1], sub, n) : 0;
            w.p1[1] = start1 ? part_start(start1[u], start1[u + 1], sub + 1, n) : 0;
            w.pad[0] = w.pad[1] = 0;
            items[base + q] = w;
        }
        base += total;
        __syncthreads();
    }
    if (threadIdx.x == 0) *nitems = base;
}

// Particles per work item: about four items per resident CTA (counted as if nine fitted, tiles of 64 cells had items of a
// ninth of the size and staged nine times as much: 0.73 -> 1.25 ms a step for 8.4 M particles), at least 512 particles (an item costs its
// window's staging: 403 x 311 cells of 13 + 13 particles 0.041 ms per launch at 512, 0.048 at 300). With
// fewer than 512 particles per CTA the launch is one chain of latencies and takes one round of the CTA's
// threads per species (64^2 cells of 8 + 8: 14.1 us at 512, 12.6 at 256).
int item_chunk(int64_t n, int slots)
{
    if (n < (int64_t)slots * kMinChunk) return 2 * kBlock;
    const int64_t c = n / ((int64_t)slots * 4);
    return (int)(c < kMinChunk ? kMinChunk : (c > (1 << 30) ? (1 << 30) : c));
}

// Entries of a list for n particles on ntiles tiles: a tile with particles has at most cnt / chunk + 1.
int64_t work_item_cap(int64_t n, int64_t ntiles) { return n / (2 * kBlock) + ntiles; }

void launch_work_items(const Ctx& c, int slab, int chunk, WorkItem* items, int* nitems, int cap, cudaStream_t st)
{
    k_work_items<<<1, kItemThreads, 0, st>>>(c.sp[0].tile_start, c.nsp > 1 ? c.sp[1].tile_start : nullptr, c.ntiles, slab,
                                             chunk, items, nitems, cap);
}

size_t particle_smem_bytes(int W) { return sizeof(unsigned) * (size_t)7 * W * W; }

// Resident CTAs of the particle kernel: the registers' limit, or that of the windows in an SM's shared memory (228
// KB, 1 KB of it per CTA the system's) for tiles above 22 cells.
int particle_slots(int nsm, int full, int batch, int W)
{
    const int regs = batch ? kCtasPerSmBatch : (full ? kCtasPerSm : kCtasPerSmAtoms);
    const int smem = (int)(228 * 1024 / (particle_smem_bytes(W) + 1024 + sizeof(WorkItem) + sizeof(int)));
    return nsm * (smem < 1 ? 1 : (smem < regs ? smem : regs));
}


// The kernel instances: Eq. (3), the altered potential and the Morse form, on the cubic and the
// HCP lattice, and the embedded-atom form on the cubic lattice (potential code in bits 0-1,
// kLatHcp in bit 2), with and without fields.
#define GBPIC_FOR_EACH_POT(X) X(kPotLJ) X(kPotAlt) X(kPotMorse) X(kPotEam) X(kPotLJ | kLatHcp) X(kPotAlt | kLatHcp) \
    X(kPotMorse | kLatHcp)

static void set_smem(const void* k, size_t shmem)
{
    cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)shmem);
    // the largest carve-out, so that several CTAs fit on one SM
    cudaFuncSetAttribute(k, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
}

void launch_particle_step(Ctx& c, const StepArgs& a, cudaStream_t st)
{
    const size_t shmem = particle_smem_bytes(a.W);
    // the attributes are per device: remember what each device has been given
    static std::atomic<size_t> configured[kMaxDevices];
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) dev = 0;
    if (shmem > configured[dev].load()) {
#define GBPIC_ATTR(P)                                                                                       \
    set_smem((const void*)k_particles<true, (P), 0>, shmem);                                               \
    set_smem((const void*)k_particles<false, (P), 0>, shmem);                                              \
    set_smem((const void*)k_particles<true, (P), kWin>, shmem);                                            \
    set_smem((const void*)k_particles<false, (P), kWin>, shmem);
        GBPIC_FOR_EACH_POT(GBPIC_ATTR)
#undef GBPIC_ATTR
        configured[dev].store(shmem);
    }
    const int grid = particle_slots(c.nsm, a.full, 0, a.W);
    if (!c.items_ok) {
        const int64_t n = c.sp[0].n + (c.nsp > 1 ? c.sp[1].n : 0);
        cudaMemsetAsync(c.nitems, 0, sizeof(int), st);
        launch_work_items(c, 0, item_chunk(n, grid), c.items, c.nitems, c.items_cap, st);
        c.items_ok = 1;
    }
    // the instance with the potential and the lattice compiled in, and the window edge when it is
    // the 16-cell tile's
    switch ((a.pot_mode & 7) | (a.full ? 8 : 0) | (a.W == kWin ? 16 : 0)) {
#define GBPIC_CASE(P)                                                                                 \
    case 24 | (P): k_particles<true, (P), kWin><<<grid, kBlock, shmem, st>>>(a, c.items, c.nitems); break;         \
    case 16 | (P): k_particles<false, (P), kWin><<<grid, kBlock, shmem, st>>>(a, c.items, c.nitems); break;        \
    case 8 | (P): k_particles<true, (P), 0><<<grid, kBlock, shmem, st>>>(a, c.items, c.nitems); break;             \
    case (P): k_particles<false, (P), 0><<<grid, kBlock, shmem, st>>>(a, c.items, c.nitems); break;
        GBPIC_FOR_EACH_POT(GBPIC_CASE)
#undef GBPIC_CASE
    }
}

int max_batch_slabs() { return kMaxBatchSlabs; }

void launch_particle_step_batch(const StepArgs* args_dev, int nslab, const WorkItem* items, const int* nitems, int full,
                                int pot, int minW, int maxW, int nsm, cudaStream_t st)
{
    cudaMemcpyToSymbolAsync(c_batch_args, args_dev, sizeof(StepArgs) * nslab, 0, cudaMemcpyDeviceToDevice, st);
    const size_t shmem = particle_smem_bytes(maxW);
    // the attributes are per device: remember what each device has been given
    static std::atomic<size_t> configured[kMaxDevices];
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) dev = 0;
    if (shmem > configured[dev].load()) {
#define GBPIC_ATTR(P)                                                                                       \
    set_smem((const void*)k_particles_batch<true, (P), 0>, shmem);                                         \
    set_smem((const void*)k_particles_batch<false, (P), 0>, shmem);                                        \
    set_smem((const void*)k_particles_batch<true, (P), kWin>, shmem);                                      \
    set_smem((const void*)k_particles_batch<false, (P), kWin>, shmem);
        GBPIC_FOR_EACH_POT(GBPIC_ATTR)
#undef GBPIC_ATTR
        configured[dev].store(shmem);
    }
    const int grid = particle_slots(nsm, full, 1, maxW);
    // pot: the instance code shared by every slab (potential and lattice); the compiled-in window
    // edge when every slab has it
    switch ((pot & 7) | (full ? 8 : 0) | (minW == kWin && maxW == kWin ? 16 : 0)) {
#define GBPIC_CASE(P)                                                                                              \
    case 24 | (P): k_particles_batch<true, (P), kWin><<<grid, kBlock, shmem, st>>>(items, nitems); break; \
    case 16 | (P): k_particles_batch<false, (P), kWin><<<grid, kBlock, shmem, st>>>(items, nitems); break; \
    case 8 | (P): k_particles_batch<true, (P), 0><<<grid, kBlock, shmem, st>>>(items, nitems); break;    \
    case (P): k_particles_batch<false, (P), 0><<<grid, kBlock, shmem, st>>>(items, nitems); break;
        GBPIC_FOR_EACH_POT(GBPIC_CASE)
#undef GBPIC_CASE
    }
}

int tile_window(int T) { return T + 2 * kMargin + 3; }

}  // namespace gbpic
