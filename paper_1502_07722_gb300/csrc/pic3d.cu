// The PIC cycle with the pair-potential force in three dimensions (3D3V): the same method as the
// 2D kernels with Eqs. (1)-(3) along x, y and z (the cubic lattice's six neighbours), trilinear
// weights, Esirkepov's 3D current and the 3D Yee scheme. x and y are periodic, z has walls.
// Fixed point: 2^14 per axis (a particle's weight product is at most 2^42). Grids are
// (nz+1) x ny x nx, index (k*ny + j)*nx + i. Yee positions: Ex (i+1/2,j,k), Ey (i,j+1/2,k),
// Ez (i,j,k+1/2), Bx (i,j+1/2,k+1/2), By (i+1/2,j,k+1/2), Bz (i+1/2,j+1/2,k).
//
// The particle kernel stages each tile's fields and node density in shared memory and streams the
// tile's particles straight from their records in coalesced order (the next record's position is
// loaded one iteration ahead); the cell sort stores each block of a tile's cell-ordered particles (256 to 4096,
// 32 x the particles per cell) column by column as a 32-row matrix, so the lanes of a warp hold
// particles of neighbouring cells. CTAs draw tiles, or parts of them, from a ticket counter (dynamic
// assignment: 10.46 -> 8.79 ms per launch on the 384^2 x 256 slab against a static round robin).
// Deposits use global 64-bit reductions, which are native in L2.
#include <atomic>

#include "pic_device.cuh"

namespace gbpic {

// The kernel instances: Eq. (3), the altered potential and the Morse form, on the cubic and the
// HCP lattice, and the embedded-atom form on the cubic lattice (potential code in bits 0-1,
// kLatHcp in bit 2).
#define GBPIC_FOR_EACH_POT3(X) X(kPotLJ) X(kPotAlt) X(kPotMorse) X(kPotEam) X(kPotLJ | kLatHcp) \
    X(kPotAlt | kLatHcp) X(kPotMorse | kLatHcp)

constexpr int kQ3Bits = 14;
constexpr int kQ3 = 1 << kQ3Bits;
constexpr int kBlock3 = 256;
// Resident CTAs: 3 with fields (80 registers), 4 without (64). All potentials gain from the fourth, also the embedded
// atom and HCP Morse, which spill 12 to 28 bytes at 64 registers (1.5 M cells of 16 atoms, ms a step before and after: Eq. (3)
// 0.577 -> 0.520, Morse 0.681 -> 0.587, HCP Morse 1.136 -> 1.010, embedded atom 1.035 -> 0.941).
constexpr int kCtas3 = 3, kCtas3Atoms = 4;
// Parts per tile (a power of two up to 16) until there are kFill3 items per resident CTA: a grid of few
// tiles left most of the chip idle. Every item stages its tile's window, seven arrays with fields and the
// density alone without. ms per launch, whole tiles -> parts: 37 x 27 x 32 cells of 16 + 16 particles 0.176 ->
// 0.041, 90 x 80 x 60 of 8 + 8 0.205 -> 0.118 (at 2 per CTA 0.126), 88 x 246 x 28 of 9 atoms 0.143 -> 0.083
// (at 2 per CTA 0.087). Past one item per CTA a part keeps at least kMinPart3
// particles on average, a round of the CTA's threads (96 x 64 x 64 cells of 1 atom 43 -> 41 us a step; a bound on the
// first parts too took 25 instead of 21 us on 24^3 cells of 4 atoms).
constexpr int kMaxLog2Sub3 = 4, kFill3 = 1, kFill3Atoms = 4, kMinPart3 = 256;

__device__ __forceinline__ int wrapn(int i, int n) { return i < 0 ? i + n : (i >= n ? i - n : i); }
__device__ __forceinline__ int qoff3(float f) { return __float2int_rn(f * 16384.0f); }

__device__ __forceinline__ void hat3q(int d, int& s0, int& s1, int& s2)
{
    s0 = max(0, kQ3 - d);
    s1 = kQ3 - abs(d - kQ3);
    s2 = max(0, d - kQ3);
}

struct Geo3 {
    int nx, ny, nz;
    unsigned mag_x, mag_y;     // exact division by nx and ny: q = umulhi(v, mag) >> shift for v < 2^31
    int sh_x, sh_y;            // 2^shift < n <= 2^(shift + 1), mag = ceil(2^(32 + shift) / n)
};

__device__ __forceinline__ void split3(int cell, const Geo3& g, int& i, int& j, int& k)
{
    const int q = (int)(__umulhi((unsigned)cell, g.mag_x) >> g.sh_x);
    i = cell - q * g.nx;
    k = (int)(__umulhi((unsigned)q, g.mag_y) >> g.sh_y);
    j = q - k * g.ny;
}

__device__ __forceinline__ size_t idx3(const Geo3& g, int i, int j, int k)
{
    return ((size_t)k * g.ny + j) * g.nx + i;
}

// staggered trilinear gather; (hx, hy, hz) = 1 where the component sits half a cell up
__device__ __forceinline__ float gather3(const float* __restrict__ A, const Geo3& g, int i, int j, int k, float fx,
                                         float fy, float fz, int hx, int hy, int hz)
{
    int i0 = i, j0 = j, r0 = k, r1 = k + 1;
    float wx = fx, wy = fy, wz = fz;
    if (hx) {
        if (fx >= 0.5f) wx = fx - 0.5f;
        else { i0 = wrapn(i - 1, g.nx); wx = fx + 0.5f; }
    }
    if (hy) {
        if (fy >= 0.5f) wy = fy - 0.5f;
        else { j0 = wrapn(j - 1, g.ny); wy = fy + 0.5f; }
    }
    if (hz) {
        if (fz >= 0.5f) {
            wz = fz - 0.5f;
            if (k >= g.nz - 1) { r0 = g.nz - 2; r1 = g.nz - 1; wz = 1.0f; }
        } else if (k >= 1) {
            r0 = k - 1; r1 = k; wz = fz + 0.5f;
        } else {
            r0 = 0; r1 = 1; wz = 0.0f;
        }
    }
    const int i1 = wrapn(i0 + 1, g.nx), j1 = wrapn(j0 + 1, g.ny);
    const float a000 = __ldg(A + idx3(g, i0, j0, r0)), a100 = __ldg(A + idx3(g, i1, j0, r0));
    const float a010 = __ldg(A + idx3(g, i0, j1, r0)), a110 = __ldg(A + idx3(g, i1, j1, r0));
    const float a001 = __ldg(A + idx3(g, i0, j0, r1)), a101 = __ldg(A + idx3(g, i1, j0, r1));
    const float a011 = __ldg(A + idx3(g, i0, j1, r1)), a111 = __ldg(A + idx3(g, i1, j1, r1));
    const float b00 = a000 + wx * (a100 - a000), b10 = a010 + wx * (a110 - a010);
    const float b01 = a001 + wx * (a101 - a001), b11 = a011 + wx * (a111 - a011);
    const float c0 = b00 + wy * (b10 - b00), c1 = b01 + wy * (b11 - b01);
    return c0 + wz * (c1 - c0);
}

// trilinear node density (units n0) and its exact gradient (units n0 per cell); wall rows doubled
__device__ __forceinline__ void density3(const u64* __restrict__ rho, const Geo3& g, float rho_s, int i, int j, int k,
                                         float fx, float fy, float fz, float& n, float* grad)
{
    const int i1 = wrapn(i + 1, g.nx), j1 = wrapn(j + 1, g.ny);
    float v[8];
#pragma unroll
    for (int c = 0; c < 2; c++)
#pragma unroll
        for (int b = 0; b < 2; b++)
#pragma unroll
            for (int a = 0; a < 2; a++) {
                long long r = (long long)__ldg(rho + idx3(g, a ? i1 : i, b ? j1 : j, k + c));
                if (k + c == 0 || k + c == g.nz) r *= 2;
                v[c * 4 + b * 2 + a] = rho_s * (float)r;
            }
    const float gx = 1.0f - fx, gy = 1.0f - fy, gz = 1.0f - fz;
    // along x: differences of the x-pairs weighted in y and z
    const float dx00 = v[1] - v[0], dx10 = v[3] - v[2], dx01 = v[5] - v[4], dx11 = v[7] - v[6];
    grad[0] = gz * (gy * dx00 + fy * dx10) + fz * (gy * dx01 + fy * dx11);
    const float dy00 = v[2] - v[0], dy10 = v[3] - v[1], dy01 = v[6] - v[4], dy11 = v[7] - v[5];
    grad[1] = gz * (gx * dy00 + fx * dy10) + fz * (gx * dy01 + fx * dy11);
    const float dz00 = v[4] - v[0], dz10 = v[5] - v[1], dz01 = v[6] - v[2], dz11 = v[7] - v[3];
    grad[2] = gy * (gx * dz00 + fx * dz10) + fy * (gx * dz01 + fx * dz11);
    n = gz * (gy * (gx * v[0] + fx * v[1]) + fy * (gx * v[2] + fx * v[3])) +
        fz * (gy * (gx * v[4] + fx * v[5]) + fy * (gx * v[6] + fx * v[7]));
}

struct Species3 {
    int32_t* cell;
    float *fx, *fy, *fz, *ux, *uy, *uz;
    const int32_t* tile_start;
    float e_kick, b_rot, p_kick;
    int jsign, pair;
};

struct Args3 {
    Geo3 g;
    int ntiles, nsp, full, pot_mode;
    int log2sub;            // parts per tile
    int T, ntx, nty, W;     // tile edge, tiles along x and y, staged window edge (0: no window)
    float cdt_dx, rho_s, h_coef, c_att, s_rep;
    EamP eam;
    const float* F[6];
    const u64* rho_cur;
    u64* rho_next;
    u64* J[3];
    unsigned* status;
    Species3 sp[2];
};


__device__ __forceinline__ void red64(u64* p, long long v)
{
    if (v != 0) atomicAdd(p, (u64)v);
}

// General 3 x 3 x 3 Esirkepov stencil and node-density change with global reductions.
// (X, Y, Z) global fixed-point coordinates; X1, Y1 may lie outside the periodic range.
__device__ __noinline__ void deposit3_general(Geo3 g, u64* J0, u64* J1, u64* J2, u64* rho_next, int X0, int Y0,
                                              int Z0, int X1, int Y1, int Z1, int jsign, int pair)
{
    const int bx = min(X0, X1) >> kQ3Bits, by = min(Y0, Y1) >> kQ3Bits, bz = min(Z0, Z1) >> kQ3Bits;
    int S0x[3], S1x[3], S0y[3], S1y[3], S0z[3], S1z[3];
    hat3q(X0 - bx * kQ3, S0x[0], S0x[1], S0x[2]);
    hat3q(X1 - bx * kQ3, S1x[0], S1x[1], S1x[2]);
    hat3q(Y0 - by * kQ3, S0y[0], S0y[1], S0y[2]);
    hat3q(Y1 - by * kQ3, S1y[0], S1y[1], S1y[2]);
    hat3q(Z0 - bz * kQ3, S0z[0], S0z[1], S0z[2]);
    hat3q(Z1 - bz * kQ3, S1z[0], S1z[1], S1z[2]);
    // edge sums and weight products in 32-bit (at most 6 * 2^28), widened once per term
    const int sg = jsign;
    for (int c = 0; c < 3; c++)
        for (int b = 0; b < 3; b++) {
            const int jj = wrapn(by + b, g.ny);
            if (jsign) {
                const int P = 2 * S0y[b] * S0z[c] + S1y[b] * S0z[c] + S0y[b] * S1z[c] + 2 * S1y[b] * S1z[c];
                long long acc = 0;
                for (int q = 0; q < 2; q++) {
                    acc -= (long long)(sg * (S1x[q] - S0x[q])) * P;
                    red64(J0 + idx3(g, wrapn(bx + q, g.nx), jj, bz + c), acc);
                }
            }
            if (pair)
                for (int q = 0; q < 3; q++)
                    red64(rho_next + idx3(g, wrapn(bx + q, g.nx), jj, bz + c),
                          (long long)(S1x[q] * S1y[b]) * S1z[c] - (long long)(S0x[q] * S0y[b]) * S0z[c]);
        }
    if (!jsign) return;
    for (int c = 0; c < 3; c++)
        for (int q = 0; q < 3; q++) {
            const int P = 2 * S0x[q] * S0z[c] + S1x[q] * S0z[c] + S0x[q] * S1z[c] + 2 * S1x[q] * S1z[c];
            long long acc = 0;
            for (int b = 0; b < 2; b++) {
                acc -= (long long)(sg * (S1y[b] - S0y[b])) * P;
                red64(J1 + idx3(g, wrapn(bx + q, g.nx), wrapn(by + b, g.ny), bz + c), acc);
            }
        }
    for (int b = 0; b < 3; b++)
        for (int q = 0; q < 3; q++) {
            const int P = 2 * S0x[q] * S0y[b] + S1x[q] * S0y[b] + S0x[q] * S1y[b] + 2 * S1x[q] * S1y[b];
            long long acc = 0;
            for (int c = 0; c < 2; c++) {
                acc -= (long long)(sg * (S1z[c] - S0z[c])) * P;
                red64(J2 + idx3(g, wrapn(bx + q, g.nx), wrapn(by + b, g.ny), bz + c), acc);
            }
        }
}

// A tile's staged window: the six field components and the pair density (units n0, wall rows
// doubled) on W^3 nodes from (ox, oy, oz); x and y wrap, z rows outside 0..nz repeat the edge row
// (the same values the global gathers clamp to).
struct Win3 {
    const float* f;         // fields and density, laid out as Lay3 says
    int ox1, oy1, oz, W;    // grid column and row of the window's second ones, grid plane of its first
};

// Window gathers. Every component of a particle reads the corners of one cell of the window: the
// particle's node cell for an integer-node axis, or that cell shifted one node down along a
// half-node axis when the particle sits in the lower half of its cell (offset o = 0 or -stride,
// weight f -+ 1/2). One base index serves all seven components; with the window edge WC known
// at compile time the corner and component offsets are immediates.
constexpr int kWin3 = 13;               // window edge of the 10-cell tile (compiled-in instances)

// The window's layout in shared memory. The run-time window is seven dense W^3 arrays, x fastest. The
// compiled-in one stores three components side by side in each x row, 42 floats from row to row (42 = 10
// mod 32) and 576 from plane to plane (0 mod 32): the 32 lanes of a warp sit in 32 consecutive cells of
// the tile's cell order (rows of 10), so lane l reads bank l + const at every corner, and the lanes that a
// half-node axis sends one node down meet either the same word or a free bank. (Dense rows of 13 gave
// two wavefronts per load.) The density stays dense behind them.
template <int WC>
struct Lay3 {
    int W;
    __device__ __forceinline__ int sy() const { return WC ? 42 : W; }
    __device__ __forceinline__ int sz() const { return WC ? 576 : W * W; }
    // component q (Ex, Ey, Ez, Bx, By, Bz)
    __device__ __forceinline__ int comp(int q) const { return WC ? (q / 3) * (576 * WC) + (q % 3) * 14 : q * W * W * W; }
    template <bool FULL>
    __device__ __forceinline__ int density() const
    {
        return !FULL ? 0 : (WC ? 2 * 576 * WC : 6 * W * W * W);
    }
};
static size_t window3_floats(int W, int full)
{
    const size_t n = (size_t)W * W * W;
    return !full ? n : (W == kWin3 ? 2 * 576 * (size_t)kWin3 + n : 7 * n);
}

struct Axis3 {
    float g, w;       // weights of the lower and upper node (1 - w, w)
};

// trilinear interpolation of the corners of the cell at p (strides sy, sz of the window's layout) on z-pairs of
// corners: each packed FP32x2 operation interpolates the lower and the upper face at once
// (measured on the 384^2 x 256 slab with the deposit below inlined: 7.73 -> 7.44 ms per launch)
__device__ __forceinline__ float trilerp3(const float* p, int sy, int sz, Axis3 x, Axis3 y, Axis3 z)
{
    const float2 gx2 = make_float2(x.g, x.g), wx2 = make_float2(x.w, x.w);
    const float2 Q0 = __ffma2_rn(wx2, make_float2(p[1], p[sz + 1]), __fmul2_rn(gx2, make_float2(p[0], p[sz])));
    const float2 Q1 = __ffma2_rn(wx2, make_float2(p[sy + 1], p[sz + sy + 1]),
                                 __fmul2_rn(gx2, make_float2(p[sy], p[sz + sy])));
    const float2 R = __ffma2_rn(make_float2(y.w, y.w), Q1, __fmul2_rn(make_float2(y.g, y.g), Q0));
    return z.g * R.x + z.w * R.y;
}

// E and B at the particle from the window (out: Ex, Ey, Ez, Bx, By, Bz); base = index of the
// particle's cell in the fields' layout
template <int WC>
__device__ __forceinline__ void wfields3(const float* f, int Wr, int base, float fx, float fy, float fz, float* out)
{
    const Lay3<WC> L{Wr};
    const int W = L.sy(), WW = L.sz();
    const bool ux = fx >= 0.5f, uy = fy >= 0.5f, uz = fz >= 0.5f;
    const int ox = ux ? 0 : -1, oy = uy ? 0 : -W, oz = uz ? 0 : -WW;
    const Axis3 X{1.0f - fx, fx}, Y{1.0f - fy, fy}, Z{1.0f - fz, fz};
    const float hx = ux ? fx - 0.5f : fx + 0.5f, hy = uy ? fy - 0.5f : fy + 0.5f, hz = uz ? fz - 0.5f : fz + 0.5f;
    const Axis3 HX{1.0f - hx, hx}, HY{1.0f - hy, hy}, HZ{1.0f - hz, hz};
    out[0] = trilerp3(f + L.comp(0) + base + ox, W, WW, HX, Y, Z);                       // Ex (i+1/2, j, k)
    out[1] = trilerp3(f + L.comp(1) + base + oy, W, WW, X, HY, Z);                 // Ey (i, j+1/2, k)
    out[2] = trilerp3(f + L.comp(2) + base + oz, W, WW, X, Y, HZ);             // Ez (i, j, k+1/2)
    out[3] = trilerp3(f + L.comp(3) + base + oy + oz, W, WW, X, HY, HZ);       // Bx (i, j+1/2, k+1/2)
    out[4] = trilerp3(f + L.comp(4) + base + ox + oz, W, WW, HX, Y, HZ);       // By (i+1/2, j, k+1/2)
    out[5] = trilerp3(f + L.comp(5) + base + ox + oy, W, WW, HX, HY, Z);       // Bz (i+1/2, j+1/2, k)
}

// trilinear density and exact gradient from the window (the arithmetic of density3)
template <int WC>
__device__ __forceinline__ void wdensity3(const float* nh, int Wr, int base, float fx, float fy, float fz, float& n,
                                          float* grad)
{
    const int W = WC ? WC : Wr, sy = W, sz = W * W;
    const float* p = nh + base;
    const float v0 = p[0], v1 = p[1], v2 = p[sy], v3 = p[sy + 1];
    const float v4 = p[sz], v5 = p[sz + 1], v6 = p[sz + sy], v7 = p[sz + sy + 1];
    const float gx = 1.0f - fx, gy = 1.0f - fy, gz = 1.0f - fz;
    const float dz00 = v4 - v0, dz10 = v5 - v1, dz01 = v6 - v2, dz11 = v7 - v3;
    grad[2] = gy * (gx * dz00 + fx * dz10) + fy * (gx * dz01 + fx * dz11);
    // z-pairs (v0, v4), (v1, v5), (v2, v6), (v3, v7); a difference b - a is fma(-1, a, b), exact
    const float2 P0 = make_float2(v0, v4), P1 = make_float2(v1, v5), P2 = make_float2(v2, v6),
                 P3 = make_float2(v3, v7), m1 = make_float2(-1.0f, -1.0f);
    const float2 gx2 = make_float2(gx, gx), fx2 = make_float2(fx, fx), gy2 = make_float2(gy, gy),
                 fy2 = make_float2(fy, fy);
    const float2 Gx = __ffma2_rn(fy2, __ffma2_rn(m1, P2, P3), __fmul2_rn(gy2, __ffma2_rn(m1, P0, P1)));
    grad[0] = gz * Gx.x + fz * Gx.y;
    const float2 Gy = __ffma2_rn(fx2, __ffma2_rn(m1, P1, P3), __fmul2_rn(gx2, __ffma2_rn(m1, P0, P2)));
    grad[1] = gz * Gy.x + fz * Gy.y;
    const float2 R = __ffma2_rn(fy2, __ffma2_rn(fx2, P3, __fmul2_rn(gx2, P2)),
                                __fmul2_rn(gy2, __ffma2_rn(fx2, P1, __fmul2_rn(gx2, P0))));
    n = gz * R.x + fz * R.y;
}

// rare path (a particle outside its tile's window): everything from global memory.
// out: E x3, B x3, n, grad x3
__device__ __noinline__ void gather_global3(const float* F0, const float* F1, const float* F2, const float* F3,
                                            const float* F4, const float* F5, const u64* rho, Geo3 g, float rho_s,
                                            int fields, int pair, int i, int j, int k, float fx, float fy, float fz,
                                            float* out)
{
    if (fields) {
        out[0] = gather3(F0, g, i, j, k, fx, fy, fz, 1, 0, 0);
        out[1] = gather3(F1, g, i, j, k, fx, fy, fz, 0, 1, 0);
        out[2] = gather3(F2, g, i, j, k, fx, fy, fz, 0, 0, 1);
        out[3] = gather3(F3, g, i, j, k, fx, fy, fz, 0, 1, 1);
        out[4] = gather3(F4, g, i, j, k, fx, fy, fz, 1, 0, 1);
        out[5] = gather3(F5, g, i, j, k, fx, fy, fz, 1, 1, 0);
    }
    if (pair) density3(rho, g, rho_s, i, j, k, fx, fy, fz, out[6], out + 7);
}

// A particle that stays in its cell: currents on the cell's edges, node density changes on its corners, as
// global 64-bit reductions.
// The edge sums 2 S0 S0' + S1 S0' + S0 S1' + 2 S1 S1' are formed as S0 (2 S0' + S1') + S1 (S0' + 2 S1')
// from the second axis' two combinations (each product at most 3 * 2^28, the sum at most
// 6 * 2^28 < 2^31: exact in 32-bit); one widening multiply per term. Every reduction is issued
// without a zero test: a particle that moved along an axis almost never has a zero term, and a zero
// adds nothing. Inlined: the currents' base pointers stay kernel parameters (against an
// out-of-line call: 7.68 -> 7.44 ms per launch on the 384^2 x 256 slab).
// The offsets to the cell's other corners (x, y periodic) fit 32 bits: a grid has fewer than 2^31 nodes.
__device__ __forceinline__ void deposit3_cell(Geo3 g, u64* J0, u64* J1, u64* J2, u64* rho_next, int base, int i,
                                              int j, int x0, int y0, int z0, int x1, int y1, int z1, int jsign,
                                              int pair)
{
    const int ox = i + 1 == g.nx ? 1 - g.nx : 1, oy = j + 1 == g.ny ? (1 - g.ny) * g.nx : g.nx, oz = g.nx * g.ny;
    const int ax0 = kQ3 - x0, ax1 = kQ3 - x1, ay0 = kQ3 - y0, ay1 = kQ3 - y1, az0 = kQ3 - z0, az1 = kQ3 - z1;
    if (jsign) {
        const int dX = jsign * (x1 - x0), dY = jsign * (y1 - y0), dZ = jsign * (z1 - z0);
        // (2 S0' + S1', S0' + 2 S1') of the lower (L) and upper (H) node of y and z
        const int Ly0 = 2 * ay0 + ay1, Ly1 = ay0 + 2 * ay1, Hy0 = 2 * y0 + y1, Hy1 = y0 + 2 * y1;
        const int Lz0 = 2 * az0 + az1, Lz1 = az0 + 2 * az1, Hz0 = 2 * z0 + z1, Hz1 = z0 + 2 * z1;
        if (dX) {
            // J6x(i+1/2, j+b, k+c) = dX (2 S0y S0z + S1y S0z + S0y S1z + 2 S1y S1z)
            atomicAdd(J0 + base, (u64)((long long)dX * (ay0 * Lz0 + ay1 * Lz1)));
            atomicAdd(J0 + base + oy, (u64)((long long)dX * (y0 * Lz0 + y1 * Lz1)));
            atomicAdd(J0 + base + oz, (u64)((long long)dX * (ay0 * Hz0 + ay1 * Hz1)));
            atomicAdd(J0 + base + oy + oz, (u64)((long long)dX * (y0 * Hz0 + y1 * Hz1)));
        }
        if (dY) {
            atomicAdd(J1 + base, (u64)((long long)dY * (ax0 * Lz0 + ax1 * Lz1)));
            atomicAdd(J1 + base + ox, (u64)((long long)dY * (x0 * Lz0 + x1 * Lz1)));
            atomicAdd(J1 + base + oz, (u64)((long long)dY * (ax0 * Hz0 + ax1 * Hz1)));
            atomicAdd(J1 + base + ox + oz, (u64)((long long)dY * (x0 * Hz0 + x1 * Hz1)));
        }
        if (dZ) {
            atomicAdd(J2 + base, (u64)((long long)dZ * (ax0 * Ly0 + ax1 * Ly1)));
            atomicAdd(J2 + base + ox, (u64)((long long)dZ * (x0 * Ly0 + x1 * Ly1)));
            atomicAdd(J2 + base + oy, (u64)((long long)dZ * (ax0 * Hy0 + ax1 * Hy1)));
            atomicAdd(J2 + base + ox + oy, (u64)((long long)dZ * (x0 * Hy0 + x1 * Hy1)));
        }
    }
    if (pair) {
        // the density changes by S(new) - S(old) on each corner; x-y products exact in 32-bit
        const int sx0[2] = {ax0, x0}, sx1[2] = {ax1, x1};
        const int sy0[2] = {ay0, y0}, sy1[2] = {ay1, y1};
        const int sz0[2] = {az0, z0}, sz1[2] = {az1, z1};
#pragma unroll
        for (int c = 0; c < 2; c++)
#pragma unroll
            for (int b = 0; b < 2; b++)
#pragma unroll
                for (int q = 0; q < 2; q++)
                    atomicAdd(rho_next + base + (q ? ox : 0) + (b ? oy : 0) + (c ? oz : 0),
                              (u64)((long long)(sx1[q] * sy1[b]) * sz1[c] - (long long)(sx0[q] * sy0[b]) * sz0[c]));
    }
}

// Fixed-point offset as the bit pattern of rint(f 2^14) + 1.5 2^23: one FMA rounds to the integer (half
// to even, as the conversion would); differences of two patterns are differences of the offsets.
constexpr int kQ3Bias = 0x4B400000;
__device__ __forceinline__ int qbits3(float f) { return __float_as_int(__fmaf_rn(f, 16384.0f, 12582912.0f)); }

// Particle p of species S (position (cell, fx, fy, fz) loaded by the caller): its momenta are read,
// the record advanced one step and written back before its deposits, so that little state is live
// during them. PAIR is a run-time flag (the pair species): one instance of this code serves both
// species, which keeps the kernel inside the instruction cache. WC is the window edge when it is
// compiled in (0: the run-time a.W).
// As in 2D, a particle that stays in its cell (almost every one) takes the short way: no floor, no
// wall test, no new cell index, and its cell is not written (52 instead of 56 bytes move per particle):
// 602 -> 526 warp instructions per 32 particles, 7.39 -> 7.01 ms per launch on the 384^2 x 256 slab, 2.89
// -> 2.79 ms on the 144 M atoms of the 3D crater slab.
template <bool FULL, int POT, int WC>
__device__ __forceinline__ void process3(const Args3& a, const Species3& S, const Win3& w, const bool PAIR, int p,
                                         const int cell, const float fx, const float fy, const float fz)
{
    const Geo3& g = a.g;
    float ux = S.ux[p], uy = S.uy[p], uz = S.uz[p];
    int i, j, k;
    split3(cell, g, i, j, k);
    // window coordinates from its second column and row on, as in 2D (w.ox1, w.oy1 lie in [0, n): a node before
    // them is one period further on)
    const int W = WC ? WC : w.W;
    unsigned lx1 = (unsigned)(i - w.ox1), ly1 = (unsigned)(j - w.oy1);
    lx1 = min(lx1, lx1 + (unsigned)g.nx);
    ly1 = min(ly1, ly1 + (unsigned)g.ny);
    const int lz = k - w.oz;
    const bool inwin = W > 0 && lx1 < (unsigned)(W - 3) && ly1 < (unsigned)(W - 3) && (unsigned)(lz - 1) < (unsigned)(W - 3);
    float kx = 0.f, ky = 0.f, kz = 0.f, bx = 0.f, by = 0.f, bz = 0.f;
    float n = 0.f, gr[3] = {0.f, 0.f, 0.f};
    if (inwin) {
        const Lay3<WC> L{W};
        if (FULL) {
            float o[6];
            wfields3<WC>(w.f, W, lz * L.sz() + ((int)ly1 + 1) * L.sy() + (int)lx1 + 1, fx, fy, fz, o);
            kx = S.e_kick * o[0]; ky = S.e_kick * o[1]; kz = S.e_kick * o[2];
            bx = o[3]; by = o[4]; bz = o[5];
        }
        if (PAIR)
            wdensity3<WC>(w.f + L.template density<FULL>(), W, (lz * W + (int)ly1 + 1) * W + (int)lx1 + 1, fx, fy, fz, n,
                          gr);
    } else {
        float o[10];
        gather_global3(a.F[0], a.F[1], a.F[2], a.F[3], a.F[4], a.F[5], a.rho_cur, g, a.rho_s, FULL ? 1 : 0,
                       PAIR ? 1 : 0, i, j, k, fx, fy, fz, o);
        if (FULL) {
            kx = S.e_kick * o[0]; ky = S.e_kick * o[1]; kz = S.e_kick * o[2];
            bx = o[3]; by = o[4]; bz = o[5];
        }
        if (PAIR) { n = o[6]; gr[0] = o[7]; gr[1] = o[8]; gr[2] = o[9]; }
    }
    if (PAIR) {
        if (n > 0.0f) {
            const float c = fast_cbrt(n);
            const float inv43 = fast_rcp(n * c);
            float pf[3];
            pair_force3<POT>(n, c, inv43, gr, a.h_coef, a.pot_mode, a.c_att, a.s_rep, pf, a.eam);
            kx += S.p_kick * pf[0];
            ky += S.p_kick * pf[1];
            kz += S.p_kick * pf[2];
        }
    }
    ux += kx; uy += ky; uz += kz;
    if (FULL) {
        const float ig = rsqrtf(1.0f + ux * ux + uy * uy + uz * uz);
        const float tx = S.b_rot * ig * bx, ty = S.b_rot * ig * by, tz = S.b_rot * ig * bz;
        const float s = 2.0f * fast_rcp(1.0f + tx * tx + ty * ty + tz * tz);
        const float px = ux + (uy * tz - uz * ty);
        const float py = uy + (uz * tx - ux * tz);
        const float pz = uz + (ux * ty - uy * tx);
        ux += s * (py * tz - pz * ty);
        uy += s * (pz * tx - px * tz);
        uz += s * (px * ty - py * tx);
    }
    ux += kx; uy += ky; uz += kz;
    const float ig = rsqrtf(1.0f + ux * ux + uy * uy + uz * uz);
    const float dxi = __fmul_rn(__fmul_rn(ux, a.cdt_dx), ig), dyi = __fmul_rn(__fmul_rn(uy, a.cdt_dx), ig),
                dze = __fmul_rn(__fmul_rn(uz, a.cdt_dx), ig);
    float nfx = __fadd_rn(fx, dxi), nfy = __fadd_rn(fy, dyi), nfz = __fadd_rn(fz, dze);
    if (!(nfx >= 0.0f && nfx < 1.0f && nfy >= 0.0f && nfy < 1.0f && nfz >= 0.0f && nfz < 1.0f && fabsf(dze) < 1.0f)) {
        // leaves its cell, reflects off a wall, or moved too far (or is not finite)
        if (!(fabsf(dxi) < 1.0f && fabsf(dyi) < 1.0f && fabsf(dze) < 1.0f)) {
            // refused: the particle keeps its record
            atomicOr(a.status, (isfinite(ux) && isfinite(uy) && isfinite(uz)) ? kErrMove : kErrNan);
            ux = S.ux[p];
            uy = S.uy[p];
            uz = S.uz[p];
            nfx = fx;
            nfy = fy;
            nfz = fz;
        }
        int di = (int)floorf(nfx);
        nfx -= (float)di;
        if (nfx >= 1.0f) { nfx = 0.0f; di += 1; }
        int dj = (int)floorf(nfy);
        nfy -= (float)dj;
        if (nfy >= 1.0f) { nfy = 0.0f; dj += 1; }
        int dk = 0;
        if (k == 0 && nfz < 0.0f) {
            nfz = -nfz; uz = -uz;
        } else if (k == g.nz - 1 && nfz >= 1.0f) {
            nfz = 2.0f - nfz; uz = -uz;
        } else {
            dk = (int)floorf(nfz);
            nfz -= (float)dk;
            if (nfz >= 1.0f) { nfz = 0.0f; dk += 1; }
        }
        S.cell[p] = (int)idx3(g, wrapn(i + di, g.nx), wrapn(j + dj, g.ny), k + dk);
        S.fx[p] = nfx;
        S.fy[p] = nfy;
        S.fz[p] = nfz;
        S.ux[p] = ux;
        S.uy[p] = uy;
        S.uz[p] = uz;
        deposit3_general(g, a.J[0], a.J[1], a.J[2], a.rho_next, i * kQ3 + qoff3(fx), j * kQ3 + qoff3(fy),
                         k * kQ3 + qoff3(fz), (i + di) * kQ3 + qoff3(nfx), (j + dj) * kQ3 + qoff3(nfy),
                         (k + dk) * kQ3 + qoff3(nfz), S.jsign, PAIR ? 1 : 0);
        return;
    }
    S.fx[p] = nfx;
    S.fy[p] = nfy;
    S.fz[p] = nfz;
    S.ux[p] = ux;
    S.uy[p] = uy;
    S.uz[p] = uz;

    const int x0 = qbits3(fx), x1 = qbits3(nfx), y0 = qbits3(fy), y1 = qbits3(nfy), z0 = qbits3(fz), z1 = qbits3(nfz);
    if (x1 == x0 && y1 == y0 && z1 == z0) return;
    deposit3_cell(g, a.J[0], a.J[1], a.J[2], a.rho_next, cell, i, j, x0 - kQ3Bias, y0 - kQ3Bias, z0 - kQ3Bias,
                  x1 - kQ3Bias, y1 - kQ3Bias, z1 - kQ3Bias, S.jsign, PAIR ? 1 : 0);
}

// start of part `sub` of 2^log2sub of the records q0 .. q1 - 1; inner boundaries lie on multiples of 32
__device__ __forceinline__ int part3(int q0, int q1, int sub, int log2sub)
{
    if (sub == 0) return q0;
    if (sub >> log2sub) return q1;
    return max(q0, (q0 + (int)((u64)(unsigned)(q1 - q0) * (unsigned)sub >> log2sub)) & ~31);
}

template <bool FULL, int POT, int WC>
__global__ void __launch_bounds__(kBlock3, FULL ? kCtas3 : kCtas3Atoms) k_particles3(const __grid_constant__ Args3 a)
{
    extern __shared__ unsigned smem3[];
    const int W = WC ? WC : a.W, WW = W * W, WWW = WW * W;
    Win3 w;
    w.W = W;
    float* wf = reinterpret_cast<float*>(smem3);
    w.f = wf;
    const Lay3<WC> L{W};
    const Geo3& g = a.g;
    // tiles are handed out dynamically from the ticket counter in the status words (atomicInc wraps
    // it back to 0 once every CTA has drawn its last, failing, ticket)
    __shared__ int slot;
    for (;;) {
        if (threadIdx.x == 0) slot = (int)atomicInc(a.status + 2, (unsigned)((a.ntiles << a.log2sub) + gridDim.x - 1));
        __syncthreads();
        const int t = slot >> a.log2sub, sub = slot & ((1 << a.log2sub) - 1);
        __syncthreads();
        if (t >= a.ntiles) break;
        int cnt = 0;
        for (int s = 0; s < a.nsp; s++) cnt += a.sp[s].tile_start[t + 1] - a.sp[s].tile_start[t];
        if (cnt == 0) continue;
        const int tx = t % a.ntx, ty = (t / a.ntx) % a.nty, tz = t / (a.ntx * a.nty);
        const int ox = wrapn(tx * a.T - 1, g.nx), oy = wrapn(ty * a.T - 1, g.ny);
        w.ox1 = tx * a.T;
        w.oy1 = ty * a.T;
        w.oz = tz * a.T - 1;
        if (W > 0) {
            __syncthreads();                       // the previous tile is done with the window
            // (the density alone: three nodes' loads in flight, as 64 registers would leave one; a step of 0.2 M atoms at one
            // per cell 40.9 -> 37.5 us)
            constexpr int kStage = FULL ? 1 : 3;
#pragma unroll kStage
            for (int q = threadIdx.x; q < WWW; q += kBlock3) {
                const int c = q / WW, r = q - c * WW, b = r / W, e = r - b * W;
                int gx = ox + e, gy = oy + b;
                while (gx >= g.nx) gx -= g.nx;
                while (gy >= g.ny) gy -= g.ny;
                const int gz = w.oz + c;
                const int gn = min(max(gz, 0), g.nz), gh = min(max(gz, 0), g.nz - 1);
                const size_t in = idx3(g, gx, gy, gn), ih = idx3(g, gx, gy, gh);
                if (FULL) {
                    float* d = wf + c * L.sz() + b * L.sy() + e;
                    d[L.comp(0)] = __ldg(a.F[0] + in);
                    d[L.comp(1)] = __ldg(a.F[1] + in);
                    d[L.comp(2)] = __ldg(a.F[2] + ih);
                    d[L.comp(3)] = __ldg(a.F[3] + ih);
                    d[L.comp(4)] = __ldg(a.F[4] + ih);
                    d[L.comp(5)] = __ldg(a.F[5] + in);
                }
                const long long r0 = (long long)__ldg(a.rho_cur + in);
                wf[L.template density<FULL>() + q] = a.rho_s * (float)((gn == 0 || gn == g.nz) ? 2 * r0 : r0);
            }
            __syncthreads();
        }
#pragma unroll 1
        for (int s = 0; s < 2; s++) {
            if (s >= a.nsp) break;
            const Species3& S = a.sp[s];
            const int p0 = part3(S.tile_start[t], S.tile_start[t + 1], sub, a.log2sub),
                      p1 = part3(S.tile_start[t], S.tile_start[t + 1], sub + 1, a.log2sub);
            // consecutive threads take consecutive records (coalesced); the cell sort's block
            // layout gives a warp's lanes neighbouring cells
            // the next record's position is loaded one iteration ahead (its first use is at the top
            // of the iteration); the momenta, first used after the gathers, are loaded in the iteration
            // warps take aligned groups of 32 records: every access of a warp is one full 128-byte line,
            // also after a re-sort, when tiles start anywhere (3D crater slab, steps 45-55: 3.04 -> 2.82 ms)
            int ncell = 0;
            float nfx = 0.0f, nfy = 0.0f, nfz = 0.0f;
            const int first = (p0 & ~31) + (int)threadIdx.x;
            if (first < p1) {
                ncell = S.cell[first]; nfx = S.fx[first]; nfy = S.fy[first]; nfz = S.fz[first];
            }
            for (int p = first; p < p1; p += kBlock3) {
                const int cell = ncell;
                const float fx = nfx, fy = nfy, fz = nfz;
                if (p + kBlock3 < p1) {
                    const int q = p + kBlock3;
                    ncell = S.cell[q]; nfx = S.fx[q]; nfy = S.fy[q]; nfz = S.fz[q];
                }
                if (p >= p0) process3<FULL, POT, WC>(a, S, w, S.pair != 0, p, cell, fx, fy, fz);
            }
        }
    }
}

static Geo3 geo_of(const Ctx& c)
{
    Geo3 g;
    g.nx = c.nx;
    g.ny = c.ny;
    g.nz = c.nz;
    magic_div(c.nx, g.mag_x, g.sh_x);
    magic_div(c.ny, g.mag_y, g.sh_y);
    return g;
}

void launch_particle_step3(Ctx& c, cudaStream_t st)
{
    Args3 a;
    memset(&a, 0, sizeof(a));
    a.g = geo_of(c);
    a.ntiles = c.ntiles;
    a.nsp = c.nsp;
    a.full = c.cfg.mode == PIC_MODE_FULL;
    a.pot_mode = pot_code(c.cfg);
    a.cdt_dx = (float)(kC * c.dt / c.cfg.dx);
    a.rho_s = (float)c.rho_scale;
    a.h_coef = (float)(c.r0 / (6.0 * c.cfg.dx));
    a.c_att = pot_param(c.cfg);
    a.s_rep = (float)c.cfg.s_rep;
    a.eam = eam_params(c.cfg);
    for (int q = 0; q < 6; q++) a.F[q] = c.F[q];
    a.rho_cur = c.rho[c.cur];
    a.rho_next = c.rho[1 - c.cur];
    for (int q = 0; q < 3; q++) a.J[q] = c.J[q];
    a.status = c.status;
    for (int s = 0; s < 2; s++) {
        const Species& S = c.sp[s];
        Species3& d = a.sp[s];
        d.cell = S.a.cell; d.fx = S.a.fx; d.fy = S.a.fy; d.fz = S.a.fz;
        d.ux = S.a.ux; d.uy = S.a.uy; d.uz = S.a.uz;
        d.tile_start = S.tile_start;
        d.e_kick = S.e_kick; d.b_rot = S.b_rot; d.p_kick = S.p_kick;
        d.jsign = S.jsign; d.pair = S.pair;
    }
    a.T = c.T;
    a.ntx = c.ntx;
    a.nty = c.nty;
    // window of the tile plus one node below and two above on each axis; staged when three CTAs
    // still fit on one SM
    const int W = c.T + 3;
    a.W = (size_t)7 * W * W * W * 4 <= 72 * 1024 ? W : 0;
    const size_t shmem = sizeof(float) * window3_floats(a.W, a.full);
    // the attributes are per device: remember what each device has been given
    static std::atomic<size_t> configured[kMaxDevices];
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) dev = 0;
    if (shmem > configured[dev].load()) {
#define GBPIC_ATTR(P)                                                                                   \
        for (const void* k : {(const void*)k_particles3<true, (P), 0>, (const void*)k_particles3<false, (P), 0>, \
                              (const void*)k_particles3<true, (P), kWin3>,                                   \
                              (const void*)k_particles3<false, (P), kWin3>}) {                               \
            cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)shmem);           \
            cudaFuncSetAttribute(k, cudaFuncAttributePreferredSharedMemoryCarveout, 100);                \
        }
        GBPIC_FOR_EACH_POT3(GBPIC_ATTR)
#undef GBPIC_ATTR
        configured[dev].store(shmem);
    }
    const int slots = c.nsm * (a.full ? kCtas3 : kCtas3Atoms);
    const int64_t n = c.sp[0].n + (c.nsp > 1 ? c.sp[1].n : 0);
    for (a.log2sub = 0; a.log2sub < kMaxLog2Sub3; a.log2sub++) {
        const int64_t items = (int64_t)c.ntiles << a.log2sub;
        if (items >= (int64_t)slots * (a.full ? kFill3 : kFill3Atoms)) break;
        if (items >= slots && n >> (a.log2sub + 1) < (int64_t)kMinPart3 * c.ntiles) break;
    }
    const int64_t items = (int64_t)c.ntiles << a.log2sub;
    int grid = items < slots ? (int)items : slots;
    if (grid < 1) grid = 1;
    // the instance with the potential and the lattice compiled in, and the window edge when it is
    // the 10-cell tile's
    const bool wc = a.W == kWin3;
    switch ((a.pot_mode & 7) | (a.full ? 8 : 0)) {
#define GBPIC_CASE(P)                                                                                         \
    case 8 | (P):                                                                                             \
        if (wc) k_particles3<true, (P), kWin3><<<grid, kBlock3, shmem, st>>>(a);                              \
        else k_particles3<true, (P), 0><<<grid, kBlock3, shmem, st>>>(a);                                     \
        break;                                                                                                \
    case (P):                                                                                                 \
        if (wc) k_particles3<false, (P), kWin3><<<grid, kBlock3, shmem, st>>>(a);                             \
        else k_particles3<false, (P), 0><<<grid, kBlock3, shmem, st>>>(a);                                    \
        break;
        GBPIC_FOR_EACH_POT3(GBPIC_CASE)
#undef GBPIC_CASE
    }
}

// ---- stand-alone node density and pair force ------------------------------------------------

// as k_deposit_density (deposit.cu): a lane walks runs of particles of one cell and issues the eight corner
// reductions once per run
__global__ void __launch_bounds__(256) k_deposit_density3(const int32_t* __restrict__ cell, const float* __restrict__ fx,
                                                          const float* __restrict__ fy, const float* __restrict__ fz,
                                                          int64_t n, Geo3 g, int cols, u64* out)
{
    const int lane = threadIdx.x & 31;
    const int64_t warp = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5, nwarp = ((int64_t)gridDim.x * blockDim.x) >> 5;
    const int64_t chunk = 32 * (int64_t)cols;
    for (int64_t base = warp * chunk; base < n; base += nwarp * chunk) {
        int at = -1;
        u64 s[8] = {0, 0, 0, 0, 0, 0, 0, 0};
        auto flush = [&]() {
            int i, j, k;
            split3(at, g, i, j, k);
            const int i1 = wrapn(i + 1, g.nx), j1 = wrapn(j + 1, g.ny);
#pragma unroll
            for (int c = 0; c < 8; c++) {
                if (s[c]) atomicAdd(out + idx3(g, c & 1 ? i1 : i, c & 2 ? j1 : j, k + (c >> 2)), s[c]);
                s[c] = 0;
            }
        };
        for (int q0 = 0; q0 < cols; q0 += kRunBatch) {
            int c[kRunBatch];
            float ox[kRunBatch], oy[kRunBatch], oz[kRunBatch];
#pragma unroll
            for (int q = 0; q < kRunBatch; q++) {
                const int64_t p = base + 32 * (int64_t)(q0 + q) + lane;
                const bool in = q0 + q < cols && p < n;
                c[q] = in ? cell[p] : -1;
                ox[q] = in ? fx[p] : 0.0f;
                oy[q] = in ? fy[p] : 0.0f;
                oz[q] = in ? fz[p] : 0.0f;
            }
#pragma unroll
            for (int q = 0; q < kRunBatch; q++) {
                if (c[q] < 0) continue;
                if (c[q] != at) {
                    if (at >= 0) flush();
                    at = c[q];
                }
                const unsigned x = (unsigned)qoff3(ox[q]), y = (unsigned)qoff3(oy[q]), z = (unsigned)qoff3(oz[q]);
                const unsigned ax = kQ3 - x, ay = kQ3 - y, az = kQ3 - z;
                const unsigned w00 = ax * ay, w10 = x * ay, w01 = ax * y, w11 = x * y;       // at most 2^28
                s[0] += (u64)w00 * az;
                s[1] += (u64)w10 * az;
                s[2] += (u64)w01 * az;
                s[3] += (u64)w11 * az;
                s[4] += (u64)w00 * z;
                s[5] += (u64)w10 * z;
                s[6] += (u64)w01 * z;
                s[7] += (u64)w11 * z;
            }
        }
        if (at >= 0) flush();
    }
}

__global__ void k_pair_force3(const int32_t* __restrict__ cell, const float* __restrict__ fx,
                              const float* __restrict__ fy, const float* __restrict__ fz, int64_t n, Geo3 g,
                              const u64* __restrict__ rho, float rho_s, float h_coef, int pot_mode, float c_att,
                              float s_rep, float f_unit, EamP eam, float* __restrict__ out)
{
    for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < n; p += (int64_t)gridDim.x * blockDim.x) {
        int i, j, k;
        split3(cell[p], g, i, j, k);
        float dens, gr[3];
        density3(rho, g, rho_s, i, j, k, fx[p], fy[p], fz[p], dens, gr);
        float F[3] = {0.f, 0.f, 0.f};
        if (dens > 0.0f) {
            const float cr = fast_cbrt(dens);
            const float inv43 = fast_rcp(dens * cr);
            pair_force3(dens, cr, inv43, gr, h_coef, pot_mode, c_att, s_rep, F, eam);
            for (int d = 0; d < 3; d++) F[d] *= f_unit;
        }
        out[3 * p] = F[0];
        out[3 * p + 1] = F[1];
        out[3 * p + 2] = F[2];
    }
}

static int grid3(const Ctx& c, int64_t n)
{
    int64_t g = (n + 255) / 256;
    if (g > (int64_t)c.nsm * 8) g = (int64_t)c.nsm * 8;
    return g < 1 ? 1 : (int)g;
}

void launch_deposit_density3(Ctx& c, u64* out, cudaStream_t st)
{
    cudaMemsetAsync(out, 0, sizeof(u64) * c.nn, st);
    const Species& S = c.sp[0];
    if (S.n == 0) return;
    const int cols = run_columns(c, S);
    k_deposit_density3<<<run_grid(c, S.n, cols), 256, 0, st>>>(S.a.cell, S.a.fx, S.a.fy, S.a.fz, S.n, geo_of(c), cols,
                                                               out);
}

void launch_pair_force3(Ctx& c, float* out, cudaStream_t st)
{
    const Species& S = c.sp[0];
    if (S.n == 0) return;
    k_pair_force3<<<grid3(c, S.n), 256, 0, st>>>(S.a.cell, S.a.fx, S.a.fy, S.a.fz, S.n, geo_of(c), c.rho[c.cur],
                                                  (float)c.rho_scale, (float)(c.r0 / (6.0 * c.cfg.dx)),
                                                  pot_code(c.cfg), pot_param(c.cfg), (float)c.cfg.s_rep,
                                                  (float)(c.D / c.r0), eam_params(c.cfg), out);
}

// ---- 3D Yee --------------------------------------------------------------------------------

struct Field3 {
    Geo3 g;
    int k_ant;
    int seg;              // planes per block
    int bx, by, bz;       // blocks along x, y and z
    float h_b, h_e, cj, mur;
    const float* ant;     // 2: this step's antenna scalars
    AntennaParams ap;     // for the next step's, into ant_next
    long long next;
    float* ant_next;
    const float* F[6];    // read
    float* G[6];          // written (the same grids with one set)
    float* save;          // one set: 8 planes of nx ny
    const u64* J[3];      // this step's currents
    u64* Z[3];            // cleared for the next step
    const u64* rho;       // node density after this step's moves
    u64* rho_next;        // starts as its copy
    const float* antc;    // nx*ny
    const float* ants;
    int k_flux;           // node plane below the antenna (Poynting flux of the injected energy)
    double* flux;
};

// The whole update as one out-of-place kernel, as in 2D (fields.cu): B half step, E step with current,
// antenna and Mur planes, B half step, the clear of the next step's currents and the start of its density.
// A block walks up a segment of planes with a patch of kRows3 + 3 rows (one per warp) of 32 columns:
// x neighbours come by shuffle, y neighbours through shared memory, z neighbours from the plane before
// in registers. The patch recomputes one row and column below and two above what it writes (13 x 29).
// It is bound by memory traffic: 112 bytes per node and step instead of 172 in three in-place passes and
// a copy/clear kernel. 384^2 x 256 cells: 0.92 ms against 1.06 plus 0.3 of the copy (segments of 8 planes
// 0.97, 32 planes 0.91; 192^2 x 128: 0.130, 0.137, 0.153); one block per SM 1.44.
constexpr int kCols3 = 29, kRows3 = 13, kWarps3 = kRows3 + 3;

struct F3 {
    float x, y, z;
};

__global__ void __launch_bounds__(32 * kWarps3, 2) k_fields3(const __grid_constant__ Field3 f)
{
    __shared__ float sex[kWarps3][32], sez[kWarps3][32], sbx[kWarps3][32], sbz[kWarps3][32], snx[kWarps3][32],
        snz[kWarps3][32];
    const Geo3& g = f.g;
    // the first block evaluates the next step's antenna scalars
    if (blockIdx.x == 0) {
        if (threadIdx.x == 0) antenna_scalars(f.ap, f.next, f.ant_next);
        return;
    }
    const int nz = g.nz, lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int blk = (int)blockIdx.x - 1, bxy = blk / f.bx, bz = bxy / f.by;
    const int i = (blk - bxy * f.bx) * kCols3 + lane - 1, j = (bxy - bz * f.by) * kRows3 + w - 1;
    int gi = i < 0 ? i + g.nx : i, gj = j < 0 ? j + g.ny : j;
    while (gi >= g.nx) gi -= g.nx;
    while (gj >= g.ny) gj -= g.ny;
    const bool own = lane >= 1 && lane <= kCols3 && i < g.nx && w >= 1 && w <= kRows3 && j < g.ny;
    const int wm = w > 0 ? w - 1 : 0, wp = w + 1 < kWarps3 ? w + 1 : w;     // the patch's outer rows are not written
    // planes k0 .. k1 - 1; the last segment takes the remainder
    const int k0 = bz * f.seg, k1 = bz + 1 == f.bz ? nz + 1 : k0 + f.seg;
    const size_t plane = (size_t)g.nx * g.ny;
    const size_t col = (size_t)gj * g.nx + gi;
    const float antc = f.antc[col], ants = f.ants[col], ant0 = f.ant[0], ant1 = f.ant[1];
    const int r0 = k0 > 0 ? k0 - 1 : 0;
    size_t c = (size_t)r0 * plane + col;
    F3 e = {__ldg(f.F[0] + c), __ldg(f.F[1] + c), __ldg(f.F[2] + c)};                     // old E of plane r
    F3 en = {__ldg(f.F[0] + c + plane), __ldg(f.F[1] + c + plane), __ldg(f.F[2] + c + plane)};   // and r + 1
    F3 b = {__ldg(f.F[3] + c), __ldg(f.F[4] + c), __ldg(f.F[5] + c)};
    u64 jx = __ldg(f.J[0] + c), jy = __ldg(f.J[1] + c), jz = __ldg(f.J[2] + c);
    F3 ep = {0, 0, 0}, bp = {0, 0, 0}, np = {0, 0, 0};       // plane r - 1: old E, half-step B, new E
    sex[w][lane] = e.x;
    sez[w][lane] = e.z;
    __syncthreads();
    for (int r = r0; r <= k1 && r <= nz; r++, c += plane) {
        // one plane ahead
        F3 e2 = {0, 0, 0}, b2 = {0, 0, 0};
        u64 jx2 = 0, jy2 = 0, jz2 = 0;
        if (r < k1 && r + 1 <= nz) {
            const size_t u = c + plane;
            b2 = F3{__ldg(f.F[3] + u), __ldg(f.F[4] + u), __ldg(f.F[5] + u)};
            jx2 = __ldg(f.J[0] + u);
            jy2 = __ldg(f.J[1] + u);
            jz2 = __ldg(f.J[2] + u);
            if (r + 2 <= nz) e2 = F3{__ldg(f.F[0] + u + plane), __ldg(f.F[1] + u + plane), __ldg(f.F[2] + u + plane)};
        }
        // B(r) to the half step (Bx, By have nz planes)
        const float exj = sex[wp][lane], ezj = sez[wp][lane];
        const float eyi = __shfl_down_sync(0xffffffffu, e.y, 1), ezi = __shfl_down_sync(0xffffffffu, e.z, 1);
        if (r < nz) {
            b.x += f.h_b * ((en.y - e.y) - (ezj - e.z));
            b.y += f.h_b * ((ezi - e.z) - (en.x - e.x));
        }
        b.z += f.h_b * ((exj - e.x) - (eyi - e.y));
        sbx[w][lane] = b.x;
        sbz[w][lane] = b.z;
        __syncthreads();
        // E(r) to the new step
        const float bxj = sbx[wm][lane], bzj = sbz[wm][lane];
        const float byi = __shfl_up_sync(0xffffffffu, b.y, 1), bzi = __shfl_up_sync(0xffffffffu, b.z, 1);
        F3 n = e;
        if (r > 0 && r < nz) {
            float v = e.x + f.h_e * ((b.z - bzj) - (b.y - bp.y)) - f.cj * (float)(long long)jx;
            if (r == f.k_ant) v += antc * ant0 + ants * ant1;
            n.x = v;
            n.y = e.y + f.h_e * ((b.x - bp.x) - (b.z - bzi)) - f.cj * (float)(long long)jy;
        }
        if (r < nz) n.z += f.h_e * ((b.y - byi) - (b.x - bxj)) - f.cj * (float)(long long)jz;
        if (r == 1) {                      // Mur: the wall planes from the new plane beside them
            np.x = e.x + f.mur * (n.x - ep.x);
            np.y = e.y + f.mur * (n.y - ep.y);
        } else if (r == nz) {
            n.x = ep.x + f.mur * (np.x - e.x);
            n.y = ep.y + f.mur * (np.y - e.y);
        }
        if (r == f.k_flux && r >= k0 && r < k1) {             // uniform over the block
            // (Ex By - Ey Bx) at the half step
            float s = own ? 0.25f * ((e.x + n.x) * (bp.y + b.y) - (e.y + n.y) * (bp.x + b.x)) : 0.0f;
            for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
            if (lane == 0 && s != 0.0f) atomicAdd(f.flux, (double)s);
        }
        // the new E of plane r - 1 for the rows below, the old E of plane r + 1 for the next turn
        snx[w][lane] = np.x;
        snz[w][lane] = np.z;
        sex[w][lane] = en.x;
        sez[w][lane] = en.z;
        __syncthreads();
        // finish plane r - 1
        const float npyi = __shfl_down_sync(0xffffffffu, np.y, 1), npzi = __shfl_down_sync(0xffffffffu, np.z, 1);
        if (r > k0 && own) {
            const size_t q = c - plane;
            const float npxj = snx[wp][lane], npzj = snz[wp][lane];
            f.G[0][q] = np.x;
            f.G[1][q] = np.y;
            f.G[2][q] = np.z;
            f.G[3][q] = bp.x + f.h_b * ((n.y - np.y) - (npzj - np.z));
            f.G[4][q] = bp.y + f.h_b * ((npzi - np.z) - (n.x - np.x));
            f.G[5][q] = bp.z + f.h_b * ((npxj - np.x) - (npyi - np.y));
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
        b = b2;
        jx = jx2;
        jy = jy2;
        jz = jz2;
    }
    if (k1 == nz + 1) {                    // the wall plane nz: only its Bz is updated
        __syncthreads();                   // the rows below have read plane nz - 1
        snx[w][lane] = np.x;
        __syncthreads();
        const float npyi = __shfl_down_sync(0xffffffffu, np.y, 1);
        if (own) {
            const size_t q = (size_t)nz * plane + col;
            f.G[0][q] = np.x;
            f.G[1][q] = np.y;
            f.G[2][q] = np.z;
            f.G[3][q] = bp.x;
            f.G[4][q] = bp.y;
            f.G[5][q] = bp.z + f.h_b * ((snx[wp][lane] - np.x) - (npyi - np.y));
        }
    }
}

// ---- one set of grids: in place, in three passes, as in 2D ----------------------------------
__global__ void k_half_B3(const __grid_constant__ Field3 f, int save)
{
    const Geo3& g = f.g;
    const int i = blockIdx.x * blockDim.x + threadIdx.x, j = blockIdx.y, k = blockIdx.z;
    if (i >= g.nx) return;
    const int ip = i + 1 == g.nx ? 0 : i + 1, jp = j + 1 == g.ny ? 0 : j + 1;
    const size_t c = idx3(g, i, j, k), plane = (size_t)g.nx * g.ny;
    const float *Ex = f.G[0], *Ey = f.G[1], *Ez = f.G[2];
    const float ex = Ex[c], ey = Ey[c];
    if (k < g.nz) {
        const float ez = Ez[c];
        f.G[3][c] += f.h_b * ((Ey[c + plane] - ey) - (Ez[idx3(g, i, jp, k)] - ez));
        f.G[4][c] += f.h_b * ((Ez[idx3(g, ip, j, k)] - ez) - (Ex[c + plane] - ex));
    }
    f.G[5][c] += f.h_b * ((Ex[idx3(g, i, jp, k)] - ex) - (Ey[idx3(g, ip, j, k)] - ey));
    const int slot = k == 0 ? 0 : k == 1 ? 1 : k == g.nz - 1 ? 2 : k == g.nz ? 3 : -1;
    if (save && slot >= 0) {
        const size_t q = (size_t)j * g.nx + i;
        f.save[slot * plane + q] = ex;
        f.save[(4 + slot) * plane + q] = ey;
    }
}

__device__ __forceinline__ float ex3_new(const Field3& f, int i, int j, int k, float old)
{
    const Geo3& g = f.g;
    const size_t c = idx3(g, i, j, k);
    const int jm = j == 0 ? g.ny - 1 : j - 1;
    float v = old + f.h_e * ((f.G[5][c] - f.G[5][idx3(g, i, jm, k)]) - (f.G[4][c] - f.G[4][idx3(g, i, j, k - 1)])) -
              f.cj * (float)(long long)f.J[0][c];
    if (k == f.k_ant) {
        const size_t q = (size_t)j * g.nx + i;
        v += f.antc[q] * f.ant[0] + f.ants[q] * f.ant[1];
    }
    return v;
}
__device__ __forceinline__ float ey3_new(const Field3& f, int i, int j, int k, float old)
{
    const Geo3& g = f.g;
    const size_t c = idx3(g, i, j, k);
    const int im = i == 0 ? g.nx - 1 : i - 1;
    return old + f.h_e * ((f.G[3][c] - f.G[3][idx3(g, i, j, k - 1)]) - (f.G[5][c] - f.G[5][idx3(g, im, j, k)])) -
           f.cj * (float)(long long)f.J[1][c];
}

__global__ void k_E3(const __grid_constant__ Field3 f)
{
    const Geo3& g = f.g;
    const int i = blockIdx.x * blockDim.x + threadIdx.x, j = blockIdx.y, k = blockIdx.z;
    float s = 0.0f;
    if (i < g.nx) {
        const size_t c = idx3(g, i, j, k), plane = (size_t)g.nx * g.ny, q = (size_t)j * g.nx + i;
        if (k > 0 && k < g.nz) {
            const float ex0 = f.G[0][c], ey0 = f.G[1][c];
            const float ex1 = ex3_new(f, i, j, k, ex0), ey1 = ey3_new(f, i, j, k, ey0);
            f.G[0][c] = ex1;
            f.G[1][c] = ey1;
            if (k == f.k_flux)
                s = 0.25f * ((ex0 + ex1) * (f.G[4][c - plane] + f.G[4][c]) - (ey0 + ey1) * (f.G[3][c - plane] + f.G[3][c]));
        } else {
            const int w = k == 0 ? 0 : 3, b = k == 0 ? 1 : 2, kb = k == 0 ? 1 : g.nz - 1;
            const float x0 = f.save[w * plane + q], x1 = f.save[b * plane + q];
            const float y0 = f.save[(4 + w) * plane + q], y1 = f.save[(4 + b) * plane + q];
            f.G[0][c] = x1 + f.mur * (ex3_new(f, i, j, kb, x1) - x0);
            f.G[1][c] = y1 + f.mur * (ey3_new(f, i, j, kb, y1) - y0);
        }
        if (k < g.nz) {
            const int im = i == 0 ? g.nx - 1 : i - 1, jm = j == 0 ? g.ny - 1 : j - 1;
            f.G[2][c] += f.h_e * ((f.G[4][c] - f.G[4][idx3(g, im, j, k)]) - (f.G[3][c] - f.G[3][idx3(g, i, jm, k)])) -
                         f.cj * (float)(long long)f.J[2][c];
        }
    }
    if (k != f.k_flux) return;
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if ((threadIdx.x & 31) == 0 && s != 0.0f) atomicAdd(f.flux, (double)s);
}

void launch_fields3(Ctx& c, cudaStream_t st, int64_t step, int64_t* launches)
{
    Field3 f;
    f.g = geo_of(c);
    f.k_ant = c.k_ant;
    f.h_b = (float)(0.5 * c.dt / c.cfg.dx);
    f.h_e = (float)(kC * kC * c.dt / c.cfg.dx);
    f.cj = (float)(kQe * c.w / (6.0 * 4398046511104.0 * c.cfg.dx * c.cfg.dx * kEps0));
    const double cdt = kC * c.dt;
    f.mur = (float)((cdt - c.cfg.dx) / (cdt + c.cfg.dx));
    f.ant = c.ant + 2 * (step & 1);
    f.ap = make_antenna_params(c);
    f.next = (long long)step + 1;
    f.ant_next = c.ant + 2 * ((step + 1) & 1);
    for (int q = 0; q < 6; q++) f.F[q] = c.F[q];
    for (int q = 0; q < 6; q++) f.G[q] = c.Fn[q] ? c.Fn[q] : c.F[q];
    f.save = c.mur_save;
    for (int q = 0; q < 3; q++) f.J[q] = c.J[q];
    for (int q = 0; q < 3; q++) f.Z[q] = c.Jn[q];
    f.rho = c.rho[c.cur];
    f.rho_next = c.rho[1 - c.cur];
    f.antc = c.ant_c;
    f.ants = c.ant_s;
    f.k_flux = c.k_ant - 1 >= 1 ? c.k_ant - 1 : -1;
    f.flux = c.red_out + 5;
    if (!c.Fn[0]) {
        const dim3 block(256), grid((c.nx + 255) / 256, c.ny, c.nz + 1);
        k_half_B3<<<grid, block, 0, st>>>(f, 1);
        k_E3<<<grid, block, 0, st>>>(f);
        k_half_B3<<<grid, block, 0, st>>>(f, 0);
        if (launches) *launches += 3;
        return;
    }
    // 16 planes per block (every segment repeats about two), fewer where that leaves under four blocks per SM
    // (90 x 80 x 60 cells: 56 us at 16 planes, 29 at 4; 37 x 27 x 32: 29, 15, 11 at 2); the last segment takes the remainder, at least `seg` planes
    f.bx = (c.nx + kCols3 - 1) / kCols3;
    f.by = (c.ny + kRows3 - 1) / kRows3;
    f.seg = 16;
    while (f.seg > 2 && (int64_t)f.bx * f.by * ((c.nz + 1) / f.seg) < 4 * (int64_t)c.nsm) f.seg >>= 1;
    f.bz = (c.nz + 1) / f.seg > 1 ? (c.nz + 1) / f.seg : 1;
    k_fields3<<<1 + f.bx * f.by * f.bz, 32 * kWarps3, 0, st>>>(f);
    swap_fields(c);
    if (launches) *launches += 1;
}

// ---- energies ------------------------------------------------------------------------------

// lanes of a warp, a fixed-shape tree (the result in lane 0)
__device__ __forceinline__ double warp_sum3(double v)
{
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    return v;
}

// Four blocks per SM, all that are launched, so that they run at once: without the bound the kernel takes 76 registers
// and three fit (37.7 M particles 694 us with one particle at a time and FP64 sums, 1048 with three blocks and the density
// conversions by i64_f32, 659 with four, 535 with plain conversions).
__global__ void __launch_bounds__(256, 4) k_energy3(const Species3 s0, const Species3 s1, int64_t n0, int64_t n1, int nsp, Geo3 g,
                                                 const float* F0, const float* F1, const float* F2, const float* F3,
                                                 const float* F4, const float* F5, const u64* rho, float rho_s,
                                                 float h_coef, int pot_mode, float c_att, float s_rep, EamP eam,
                                                 double* partials)
{
    __shared__ double sh[5][256];
    const int64_t tid = blockIdx.x * (int64_t)256 + threadIdx.x, stride = (int64_t)gridDim.x * 256;
    LongSum ke[2], pe;
    double fe = 0.0, fb = 0.0;
    for (int s = 0; s < nsp; s++) {
        const Species3& S = s == 0 ? s0 : s1;
        const int64_t ns = s == 0 ? n0 : n1;
        int terms = 0;
        for (int64_t p0 = tid; p0 < ns; p0 += 2 * stride) {
            // two particles' loads in flight together
            float ux[2], uy[2], uz[2], fx[2], fy[2], fz[2];
            int cell[2];
#pragma unroll
            for (int q = 0; q < 2; q++) {
                const int64_t p = p0 + q * stride;
                const bool in = p < ns;
                ux[q] = in ? S.ux[p] : 0.0f;
                uy[q] = in ? S.uy[p] : 0.0f;
                uz[q] = in ? S.uz[p] : 0.0f;
                if (s == 0) {
                    cell[q] = in ? S.cell[p] : 0;
                    fx[q] = in ? S.fx[p] : 0.0f;
                    fy[q] = in ? S.fy[p] : 0.0f;
                    fz[q] = in ? S.fz[p] : 0.0f;
                }
            }
            float dens[2], gr[2][3];
            if (s == 0) {
#pragma unroll
                for (int q = 0; q < 2; q++) {
                    int i, j, k;
                    split3(cell[q], g, i, j, k);
                    density3(rho, g, rho_s, i, j, k, fx[q], fy[q], fz[q], dens[q], gr[q]);
                }
            }
#pragma unroll
            for (int q = 0; q < 2; q++) {
                if (p0 + q * stride >= ns) continue;
                const float u2 = ux[q] * ux[q] + uy[q] * uy[q] + uz[q] * uz[q];
                const float t = u2 / (sqrtf(1.0f + u2) + 1.0f);
                if (s == 0) ke[0].add(t);
                else ke[1].add(t);
                if (s == 0 && dens[q] > 0.0f) {
                    const float cr = fast_cbrt(dens[q]), inv43 = fast_rcp(dens[q] * cr);
                    pe.add(pair_energy3(cr, inv43, gr[q], h_coef, pot_mode, c_att, s_rep, eam));
                }
            }
            if ((terms += 2) == kFold) {
                terms = 0;
                if (s == 0) ke[0].fold();
                else ke[1].fold();
                if (s == 0) pe.fold();
            }
        }
    }
    const int64_t nn = (int64_t)(g.nz + 1) * g.ny * g.nx, plane = (int64_t)g.ny * g.nx;
    for (int64_t c = tid; c < nn; c += stride) {
        const int k = (int)(c / plane);
        const double wn = (k == 0 || k == g.nz) ? 0.5 : 1.0;
        const double ex = F0[c], ey = F1[c], bz = F5[c];
        fe += wn * (ex * ex + ey * ey);
        fb += wn * bz * bz;
        if (k < g.nz) {
            const double ez = F2[c], bx = F3[c], by = F4[c];
            fe += ez * ez;
            fb += bx * bx + by * by;
        }
    }
    // warp q adds up slot q (13 FP64 instructions per slot and block)
    sh[0][threadIdx.x] = ke[0].value();
    sh[1][threadIdx.x] = ke[1].value();
    sh[2][threadIdx.x] = fe;
    sh[3][threadIdx.x] = fb;
    sh[4][threadIdx.x] = pe.value();
    __syncthreads();
    const int q = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (q < 5) {
        double v = sh[q][lane];
        for (int w = 1; w < 8; w++) v += sh[q][lane + 32 * w];
        v = warp_sum3(v);
        if (lane == 0) partials[(size_t)blockIdx.x * 5 + q] = v;
    }
}

// one warp per slot, blocks assigned to lanes in a fixed way
__global__ void __launch_bounds__(160) k_energy3_final(const double* __restrict__ partials, int nb, double* out)
{
    const int q = threadIdx.x >> 5, lane = threadIdx.x & 31;
    double v = 0.0;
    for (int b = lane; b < nb; b += 32) v += partials[(size_t)b * 5 + q];
    v = warp_sum3(v);
    if (lane == 0) out[q] = v;
}

void launch_energy3(Ctx& c, cudaStream_t st, double* host_out5)
{
    Species3 sp[2];
    memset(sp, 0, sizeof(sp));
    for (int s = 0; s < 2; s++) {
        const Species& S = c.sp[s];
        sp[s].cell = S.a.cell; sp[s].fx = S.a.fx; sp[s].fy = S.a.fy; sp[s].fz = S.a.fz;
        sp[s].ux = S.a.ux; sp[s].uy = S.a.uy; sp[s].uz = S.a.uz;
    }
    // small states take as many blocks as give every thread a particle or a node
    const int64_t n1 = c.nsp > 1 ? c.sp[1].n : 0, n = c.sp[0].n > n1 ? c.sp[0].n : n1;
    const int64_t want = ((n > (int64_t)c.nn ? n : (int64_t)c.nn) + 255) / 256;
    const int nb = want < c.nsm * 4 ? (int)want : c.nsm * 4;
    k_energy3<<<nb, 256, 0, st>>>(sp[0], sp[1], c.sp[0].n, n1, c.nsp, geo_of(c), c.F[0], c.F[1],
                                  c.F[2], c.F[3], c.F[4], c.F[5], c.rho[c.cur], (float)c.rho_scale,
                                  (float)(c.r0 / (6.0 * c.cfg.dx)), pot_code(c.cfg), pot_param(c.cfg),
                                  (float)c.cfg.s_rep, eam_params(c.cfg), c.partials);
    k_energy3_final<<<1, 160, 0, st>>>(c.partials, nb, c.red_out);
    double raw[5];
    cudaMemcpyAsync(raw, c.red_out, sizeof(raw), cudaMemcpyDeviceToHost, st);
    cudaStreamSynchronize(st);
    const double vol = c.cfg.dx * c.cfg.dx * c.cfg.dx, mu0 = 1.0 / (kEps0 * kC * kC);
    host_out5[0] = raw[0] * c.w * c.sp[0].mass * kC * kC;
    host_out5[1] = c.nsp > 1 ? raw[1] * c.w * c.sp[1].mass * kC * kC : 0.0;
    host_out5[2] = 0.5 * kEps0 * raw[2] * vol;
    host_out5[3] = 0.5 / mu0 * raw[3] * vol;
    host_out5[4] = 0.5 * c.D * raw[4] * c.w;
}

}  // namespace gbpic
