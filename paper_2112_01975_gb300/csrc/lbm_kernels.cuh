// Device code of the two-phase lattice Boltzmann step (arXiv 2112.01975).
//
// Storage: populations SoA f[i * N + n] (FP64), entry n = x + px (y + ny z);
// side fields written once per step by k_macro and read by the collision:
//   rp[n] = (rho, s psi)   double2; s = +1 where P > P0, else -1 (Sec. 2.3.4)
//   u[a * N + n]           bare velocity sum c f / rho (Sec. 2.3.3)
//   g[a * N + n]           rho u_a^3, the flux differenced by Phi (Eq. correction)
// Solid nodes hold the virtual density rho_w, u = g = 0 (written at init).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "lbm_pdl.cuh"

namespace lbmk {

// A lattice of M = nx ny nz nodes. The library's own fields have rows of px >=
// nx entries (px = nx except in D3Q27 reduced storage, whose rows start on 16
// bytes): node (x, y, z) is entry x + px (y + ny z) of a field of N = px ny nz
// entries. The caller's fields have no padding: see flat().
struct Geo {
    int nx, ny, nz;
    unsigned N;
    int px;
    unsigned M;
};

__host__ __device__ __forceinline__ Geo flat(Geo g)
{
    g.px = g.nx;
    g.N = g.M;
    return g;
}

__device__ __forceinline__ unsigned entry(const Geo &g, int x, int y, int z)
{
    return (unsigned)x + (unsigned)g.px * ((unsigned)y + (unsigned)g.ny * (unsigned)z);
}

struct Phys {
    int eos;
    double a, b, RT, alpha;   // EOS constants at the run's temperature (R = 1)
    double aalpha;            // a alpha
    double kappa;             // capillary coefficient kappa~
    double omega;             // 1 / tau
    double phi_pref;          // -(1 - omega/2), or 0 with the correction off
    double rho_w;             // virtual solid density
    double g[3];              // body acceleration; rho g joins the force (Sec. 4.1)
    int body;                 // g is not zero
    double kr;                // -kappa / 36 (D3Q27) or -kappa / 6 (D2Q9), see force_of_sums
    // density-dependent relaxation (var_visc): nu linear in rho from nu_l at
    // visc_rl to nu_v at visc_rv, constant beyond; phi_sign = -1, or 0 with
    // the correction off
    int var_visc;
    double nu_l, nu_v, visc_rv, visc_rl, phi_sign;
};

// Relaxation rate at density rho (the constant omega unless var_visc).
__device__ __forceinline__ double omega_at(const Phys &p, double rho)
{
    if (!p.var_visc) return p.omega;
    const double t = fmin(fmax((p.visc_rl - rho) / (p.visc_rl - p.visc_rv), 0.0), 1.0);
    return 1.0 / (3.0 * (p.nu_l + (p.nu_v - p.nu_l) * t) + 0.5);
}

template <int LAT> struct Lattice;
template <> struct Lattice<0> { static constexpr int D = 2, Q = 9; };
template <> struct Lattice<1> { static constexpr int D = 3, Q = 27; };

__host__ __device__ constexpr int cxi(int i) { return i % 3 - 1; }
__host__ __device__ constexpr int cyi(int i) { return (i / 3) % 3 - 1; }
__host__ __device__ constexpr int czi(int i) { return i / 9 - 1; }

// An FP64 instruction (a comparison or a conversion too) takes 64 cycles of
// one SM sub-partition and 19 of the SM's shared pipe, whatever the number of
// active lanes (measured): as long as 76 issue slots. The FP64 kernels are
// bound by how many they execute per node, so what can be shared between
// neighbours is, signs and finiteness are tested on the bit patterns, and
// one reciprocal serves the equation of state and 1/rho.

// P - rho/3 of the equations of state of Sec. 3.1 and Appendix G (gas
// constant 1) and 1/rho, from one reciprocal where the EOS has a denominator:
// P = rho n / D, 1/(rho D) gives both. (Error of P - rho/3 over the densities in
// use: 8.8e-17 of rho/3 rms, with a division in its place 7.3e-17; against 128-bit
// arithmetic the step's populations, u and U are closer than with divisions and FP64
// sums of the populations: U 1.16e-17 rms on 80x72x70, then 1.71e-17.)
__device__ __forceinline__ double excess_pressure(const Phys &p, double rho, double &inv)
{
    double n, D;   // P / rho + m = n / D
    double m = 0.0;
    switch (p.eos) {
    case 0:  // van der Waals
        n = p.RT;
        D = fma(-p.b, rho, 1.0);
        m = p.a * rho;
        break;
    case 1: {  // Peng-Robinson
        const double br = p.b * rho, d1 = 1.0 - br, d2 = fma(br, 2.0 - br, 1.0);
        n = fma(p.RT, d2, -(p.aalpha * rho) * d1);
        D = d1 * d2;
        break;
    }
    case 2: {  // Redlich-Kwong-Soave
        const double br = p.b * rho, d1 = 1.0 - br, d2 = 1.0 + br;
        n = fma(p.RT, d2, -(p.aalpha * rho) * d1);
        D = d1 * d2;
        break;
    }
    case 3: {  // Carnahan-Starling
        const double e = 0.25 * p.b * rho, om = 1.0 - e;
        n = p.RT * fma(e * e, om, 1.0 + e);
        D = om * om * om;
        m = p.a * rho;
        break;
    }
    case 4: {  // Shan-Chen, psi_SC = 1 - exp(-rho); RT holds the coupling G
        const double q = 1.0 - exp(-rho);
        inv = 1.0 / rho;
        return p.RT * (1.0 / 6.0) * q * q;
    }
    default: {  // Shan-Chen, psi_SC = exp(-1/rho)
        inv = 1.0 / rho;
        const double q = exp(-inv);
        return p.RT * (1.0 / 6.0) * q * q;
    }
    }
    const double r = 1.0 / (rho * D);
    inv = r * D;
    return rho * (fma(n, r * rho, -m) - 1.0 / 3.0);
}

// d > 0 by its bits (false for NaN, as the comparison is).
__device__ __forceinline__ bool positive(double d)
{
    const long long v = __double_as_longlong(d);
    return v > 0 && v <= 0x7ff0000000000000ll;
}

__device__ __forceinline__ bool finite_bits(double d)
{
    return (__double2hiint(d) & 0x7ff00000) != 0x7ff00000;
}

// Signed pseudo-potential s psi with psi = sqrt|P - P0|, P0 = rho/3.
__device__ __forceinline__ double signed_psi_of(double d)
{
    const double r = sqrt(fabs(d));
    return positive(d) ? r : -r;
}

// The same equations of state as pressures, for the initial state and the
// walls' virtual density (see korteweg_force).
__device__ __forceinline__ double eos_pressure(const Phys &p, double rho)
{
    switch (p.eos) {
    case 0:  // van der Waals
        return rho * p.RT / (1.0 - p.b * rho) - p.a * rho * rho;
    case 1: {  // Peng-Robinson, one division
        const double d1 = 1.0 - p.b * rho, d2 = 1.0 + 2.0 * p.b * rho - p.b * p.b * rho * rho;
        return (rho * p.RT * d2 - p.a * p.alpha * rho * rho * d1) / (d1 * d2);
    }
    case 2: {  // Redlich-Kwong-Soave, one division
        const double d1 = 1.0 - p.b * rho, d2 = 1.0 + p.b * rho;
        return (rho * p.RT * d2 - p.a * p.alpha * rho * rho * d1) / (d1 * d2);
    }
    case 3: {  // Carnahan-Starling
        const double e = 0.25 * p.b * rho;
        const double om = 1.0 - e;
        return rho * p.RT * (1.0 + e + e * e - e * e * e) / (om * om * om) - p.a * rho * rho;
    }
    case 4: {  // Shan-Chen, psi_SC = 1 - exp(-rho); RT holds the coupling G
        const double q = 1.0 - exp(-rho);
        return rho * (1.0 / 3.0) + p.RT * (1.0 / 6.0) * q * q;
    }
    default: {  // Shan-Chen, psi_SC = exp(-1/rho)
        const double q = exp(-1.0 / rho);
        return rho * (1.0 / 3.0) + p.RT * (1.0 / 6.0) * q * q;
    }
    }
}

__device__ __forceinline__ double signed_psi(const Phys &p, double rho)
{
    const double d = eos_pressure(p, rho) - rho * (1.0 / 3.0);
    return d > 0.0 ? sqrt(d) : -sqrt(-d);
}

__device__ __forceinline__ int wrapm(int v, int n) { return v < 0 ? v + n : v; }
__device__ __forceinline__ int wrapp(int v, int n) { return v >= n ? v - n : v; }

// Of shifted 16-bit storage: the weight and the node that pushed population i.
__device__ __forceinline__ double weight_d(int i, int D)
{
    const double w1[3] = {1.0 / 6.0, 2.0 / 3.0, 1.0 / 6.0};
    return w1[cxi(i) + 1] * w1[cyi(i) + 1] * (D == 3 ? w1[czi(i) + 1] : 1.0);
}

__device__ __forceinline__ unsigned source_node(const Geo &g, int D, int i, int x, int y, int z)
{
    const int sx = (x - cxi(i) + g.nx) % g.nx, sy = (y - cyi(i) + g.ny) % g.ny;
    const int sz = D == 3 ? (z - czi(i) + g.nz) % g.nz : 0;
    return entry(g, sx, sy, sz);
}

}  // namespace lbmk

#include "lbm_fixed.cuh"

namespace lbmk {

// ---- the Korteweg force of every node ---------------------------------
//   F = -2 (s psi)_c S_psi - kappa rho_c S_rho + rho_c g,
//   S_psi = sum_i (w_i/cs2) c_i [4/3 psi(r+c_i) - 1/6 psi(r+2c_i)],
//   S_rho = sum_i (w_i/cs2) c_i [2 rho(r+c_i) - rho(r+2c_i)]   (Eq. Kforce_final).
// With the 1D weights W(0) = 2/3, W(+-1) = 1/6 of Eq. wi, w_i/cs2 c_ia =
// 1/2 c_ia W(c_ib) W(c_ic): a central difference along a, then [1, 4, 1]/6
// smoothings along the other axes. Summed node by node that is 208 FP64
// operations (D3Q27; both fields, both rings), more than half of the step;
// one axis at a time, with each axis's sums shared by the nodes of a tile
// through shared memory, it is 75. The difference comes first on every axis:
// smoothed fields round at the field's size, and where it is nearly uniform
// their difference keeps that (force error of a 48^3 drop against 128-bit sums,
// rms along x, y, z: differences first 1.0, 1.0, 1.0e-17, smoothing along x
// first, 64 operations, 1.0, 5.5, 8.5e-17; node by node 1.4e-17). sum_a below
// are the sums without their common factor: ring 1 plus RING2 times ring 2,
//   S_psi = sum_psi / 54 (D2Q9: / 9),  S_rho = sum_rho / 36 (D2Q9: / 6).
constexpr double RING2_PSI = -1.0 / 8.0, RING2_RHO = -1.0 / 2.0;

template <int LAT>
__device__ __forceinline__ void force_of_sums(const Phys &p, double rho, double spsi, const double *sp,
                                              const double *sr, double *F)
{
    constexpr int D = Lattice<LAT>::D;
    const double cp = spsi * (D == 3 ? -1.0 / 27.0 : -2.0 / 9.0);
    const double cr = rho * p.kr;
#pragma unroll
    for (int a = 0; a < D; ++a) {
        F[a] = fma(cp, sp[a], cr * sr[a]);
        if (p.body) F[a] = fma(rho, p.g[a], F[a]);
    }
}

// Tiles of 32 x 8 nodes; D3Q27 marches along z through `chunk` planes. Per
// plane q of the 36 x 12 halo tile: |psi| and rho to shared memory, with the
// z-differences around plane q - 2 of the thread's own halo nodes (their last
// five planes stay in shared memory); then the x-differences and the z-
// differences smoothed along x of its 12 rows and the y-differences of its 8;
// then each node's sums of them. The z-smoothings of the x and y components build up in
// registers as the planes pass. The FP64 pipe is what is busy.
// Body: what is done with a node's sums: body(p, n, x, y, z, sp, sr).
constexpr int SWX = 32, SWY = 8;

struct SweepSmem3 {   // by field (|psi|, rho), then ring
    double raw[5][2][SWY + 4][SWX + 4];    // planes q - 4 .. q, by plane modulo 5
    double dz[2][2][SWY + 4][SWX + 4];
    double dx[2][2][SWY + 4][SWX], sz[2][2][SWY + 4][SWX];
    double dy[2][2][SWY][SWX + 4];
};

template <int ROWS> struct SweepSmem2 {
    double raw[2][ROWS + 4][SWX + 4];
    double dx[2][2][ROWS + 4][SWX];
    double dy[2][2][ROWS][SWX + 4];
};

__device__ __forceinline__ int wrap_any(int v, int n)
{
    v = v < 0 ? v + n : v;
    if (v >= n) {
        v -= n;
        if (v >= n) v %= n;
    }
    return v;
}

// [1, 4, 1] smoothing of a at distance s, `step` doubles apart.
__device__ __forceinline__ double smooth(const double *a, int s, int step)
{
    return fma(4.0, a[0], a[-s * step] + a[s * step]);
}

// x-differences of row r (of the halo tile) of both fields.
template <typename Raw, typename DX>
__device__ __forceinline__ void x_differences(const Raw &raw, DX &dx, int q, int r, int tx)
{
    const double *a = &raw[q][r][tx + 2];
#pragma unroll
    for (int s = 1; s <= 2; ++s) dx[q][s - 1][r][tx] = a[s] - a[-s];
}

// y-differences of node row r, halo column c of field q.
template <typename Raw, typename DY>
__device__ __forceinline__ void y_differences(const Raw &raw, DY &dy, int q, int r, int c)
{
#pragma unroll
    for (int s = 1; s <= 2; ++s) dy[q][s - 1][r][c] = raw[q][r + 2 + s][c] - raw[q][r + 2 - s][c];
}

template <typename Body>
__global__ void __launch_bounds__(SWX *SWY, 2)
k_force_sweep3(Geo g, Phys p, const double2 *__restrict__ rp, int chunk, Body body)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    SweepSmem3 &sm = *reinterpret_cast<SweepSmem3 *>(smem_raw);
    constexpr int NT = SWX * SWY, HX = SWX + 4, NH = HX * (SWY + 4);
    const int tid = threadIdx.x, tx = tid % SWX, ty = tid / SWX;
    const int x = blockIdx.x * SWX + tx, y = blockIdx.y * SWY + ty;
    const int z0 = blockIdx.z * chunk, z1 = min(z0 + chunk, g.nz);
    const bool inside = x < g.nx && y < g.ny;
    const unsigned plane = (unsigned)g.px * (unsigned)g.ny;
    // this thread's one or two halo nodes
    const bool two = tid + NT < NH;
    int hr[2], hc[2];
    unsigned off[2];
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        const int h = k == 0 || two ? tid + k * NT : 0;
        hr[k] = h / HX;
        hc[k] = h - hr[k] * HX;
        off[k] = (unsigned)wrap_any((int)blockIdx.x * SWX - 2 + hc[k], g.nx) +
                 (unsigned)g.px * (unsigned)wrap_any((int)blockIdx.y * SWY - 2 + hr[k], g.ny);
    }
    int zq = z0 - 2 < 0 ? z0 - 2 + g.nz : z0 - 2;
    double2 v[2];
    v[0] = rp[off[0] + plane * (unsigned)zq];
    v[1] = two ? rp[off[1] + plane * (unsigned)zq] : v[0];
    // sums under way, per field (|psi|, rho) and component x, y, after plane q:
    // n2 (ring 2 part of plane q + 2, without its factor), a1 (q + 1), a0 (q), m1 (q - 1)
    double n2[2][2] = {}, a1[2][2] = {}, a0[2][2] = {}, m1[2][2] = {};
    int w = 0;   // q's slot of sm.raw
    for (int q = z0 - 2; q < z1 + 2; ++q) {
        const bool sums = q >= z0 + 2;   // the sums of plane q - 2 are done in this iteration
        const int w1 = w == 0 ? 4 : w - 1, w3 = w < 3 ? w + 2 : w - 3, w4 = w == 4 ? 0 : w + 1;   // of q - 1, q - 3, q - 4
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            if (k == 1 && !two) break;
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const double a = e == 0 ? fabs(v[k].y) : v[k].x;
                if (sums) {
                    sm.dz[e][0][hr[k]][hc[k]] = sm.raw[w1][e][hr[k]][hc[k]] - sm.raw[w3][e][hr[k]][hc[k]];
                    sm.dz[e][1][hr[k]][hc[k]] = a - sm.raw[w4][e][hr[k]][hc[k]];
                }
                sm.raw[w][e][hr[k]][hc[k]] = a;
            }
        }
        zq = zq + 1 == g.nz ? 0 : zq + 1;
        if (q + 1 < z1 + 2) {   // the next plane, while this one is summed
            v[0] = rp[off[0] + plane * (unsigned)zq];
            if (two) v[1] = rp[off[1] + plane * (unsigned)zq];
        }
        __syncthreads();
        for (int r = ty; r < SWY + 4; r += SWY) {
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                x_differences(sm.raw[w], sm.dx, e, r, tx);
                if (sums)
#pragma unroll
                    for (int s = 1; s <= 2; ++s) sm.sz[e][s - 1][r][tx] = smooth(&sm.dz[e][s - 1][r][tx + 2], s, 1);
            }
        }
        // (by the warps that had one row)
        for (int h = tid - NT / 2; h >= 0 && h < 2 * SWY * HX; h += NT / 2)
            y_differences(sm.raw[w], sm.dy, h / (SWY * HX), h / HX % SWY, h % HX);
        __syncthreads();
        double done[2][3];
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            const double r2 = k == 0 ? RING2_PSI : RING2_RHO;
            // ring 1 and 2 sums of the plane: x and y differences, smoothed
            const double X1[2] = {smooth(&sm.dx[k][0][ty + 2][tx], 1, SWX), smooth(&sm.dy[k][0][ty][tx + 2], 1, 1)};
            const double X2[2] = {smooth(&sm.dx[k][1][ty + 2][tx], 2, SWX), smooth(&sm.dy[k][1][ty][tx + 2], 2, 1)};
#pragma unroll
            for (int a = 0; a < 2; ++a) {
                done[k][a] = fma(r2, X2[a], m1[k][a]);
                m1[k][a] = a0[k][a] + X1[a];
                a0[k][a] = fma(4.0, fma(r2, X2[a], X1[a]), a1[k][a]);
                a1[k][a] = fma(r2, n2[k][a], X1[a]);
                n2[k][a] = X2[a];
            }
            if (sums)
                done[k][2] = fma(r2, smooth(&sm.sz[k][1][ty + 2][tx], 2, SWX), smooth(&sm.sz[k][0][ty + 2][tx], 1, SWX));
        }
        if (sums && inside)
            body(g, p, entry(g, x, y, q - 2), x, y, q - 2, done[0], done[1]);
        w = w == 4 ? 0 : w + 1;
    }
}

// D3Q27 without sharing, one node per thread: each pair of opposite neighbours
// once, by weight class (208 operations). For lattices so small that the
// tiles above would be few, each summing five planes for one of its own
// (32^3: 20 us, with tiles 33; sweep_chunk has the rule).
template <typename Body>
__global__ void __launch_bounds__(128)
k_force_direct3(Geo g, Phys p, const double2 *__restrict__ rp, Body body)
{
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    if (x >= g.nx) return;
    const int y = blockIdx.y, z = blockIdx.z;
    double sum[2][3];
#pragma unroll
    for (int s = 1; s <= 2; ++s) {
        const int X[3] = {wrapm(x - s, g.nx), x, wrapp(x + s, g.nx)};
        const int Y[3] = {wrapm(y - s, g.ny), y, wrapp(y + s, g.ny)};
        const int Z[3] = {wrapm(z - s, g.nz), z, wrapp(z + s, g.nz)};
        double acc[2][3][3];   // field, component, nonzero transverse components of c
        bool set[3][3] = {};
#pragma unroll
        for (int i = 14; i < 27; ++i) {
            const int c[3] = {cxi(i), cyi(i), czi(i)};
            const double2 vp = rp[entry(g, X[c[0] + 1], Y[c[1] + 1], Z[c[2] + 1])];
            const double2 vm = rp[entry(g, X[1 - c[0]], Y[1 - c[1]], Z[1 - c[2]])];
            const double d[2] = {fabs(vp.y) - fabs(vm.y), vp.x - vm.x};
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                if (c[a] == 0) continue;
                const int k = (a != 0 && c[0] != 0) + (a != 1 && c[1] != 0) + (a != 2 && c[2] != 0);
#pragma unroll
                for (int q = 0; q < 2; ++q)
                    acc[q][a][k] = !set[a][k] ? (c[a] > 0 ? d[q] : -d[q])
                                   : c[a] > 0 ? acc[q][a][k] + d[q] : acc[q][a][k] - d[q];
                set[a][k] = true;
            }
        }
#pragma unroll
        for (int q = 0; q < 2; ++q)
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                const double v = fma(16.0, acc[q][a][0], fma(4.0, acc[q][a][1], acc[q][a][2]));
                sum[q][a] = s == 1 ? v : fma(q == 0 ? RING2_PSI : RING2_RHO, v, sum[q][a]);
            }
    }
    body(g, p, entry(g, x, y, z), x, y, z, sum[0], sum[1]);
}

// D2Q9: one tile of 32 x ROWS nodes per block, one shot; NW warps share the
// differences of the tile's rows, ROWS of them go on to the nodes. A lattice
// with too few tiles of 8 rows for the SMs takes tiles of 2 rows, 4 warps: a
// warp alone on its sub-partition is bound by its own chain of FP64
// instructions, so the tile with fewer of them per warp on more SMs wins.
template <int ROWS, int NW, typename Body>
__global__ void __launch_bounds__(32 * NW)
k_force_sweep2(Geo g, Phys p, const double2 *rp, Body body)
{
    __shared__ SweepSmem2<ROWS> sm;
    static_assert(ROWS <= NW, "a warp per row of the tile");
    constexpr int NT = 32 * NW, HX = SWX + 4, NH = HX * (ROWS + 4);
    const int tid = threadIdx.x, tx = tid % 32, w = tid / 32;
    const int x0 = blockIdx.x * SWX, y0 = blockIdx.y * ROWS;
    lbmpdl::step_trigger();
    lbmpdl::step_wait();
    for (int h = tid; h < NH; h += NT) {
        const int r = h / HX, c = h - r * HX;
        const double2 v = rp[(unsigned)wrap_any(x0 - 2 + c, g.nx) +
                             (unsigned)g.px * (unsigned)wrap_any(y0 - 2 + r, g.ny)];
        sm.raw[0][r][c] = fabs(v.y);
        sm.raw[1][r][c] = v.x;
    }
    __syncthreads();
    for (int t = w; t < 2 * (ROWS + 4); t += NW) x_differences(sm.raw, sm.dx, t & 1, t >> 1, tx);
    for (int h = tid; h < 2 * ROWS * HX; h += NT) y_differences(sm.raw, sm.dy, h / (ROWS * HX), h / HX % ROWS, h % HX);
    __syncthreads();
    const int x = x0 + tx, y = y0 + w;
    if (w >= ROWS || x >= g.nx || y >= g.ny) return;
    double sum[2][3];
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        const double r2 = k == 0 ? RING2_PSI : RING2_RHO;
        sum[k][0] = fma(r2, smooth(&sm.dx[k][1][w + 2][tx], 2, SWX), smooth(&sm.dx[k][0][w + 2][tx], 1, SWX));
        sum[k][1] = fma(r2, smooth(&sm.dy[k][1][w][tx + 2], 2, 1), smooth(&sm.dy[k][0][w][tx + 2], 1, 1));
    }
    body(g, p, entry(g, x, y, 0), x, y, 0, sum[0], sum[1]);
}

// Moments, EOS and pseudo-potential of every fluid node; flags bad densities.
// P: the populations' storage (double, float or Shifted); the moments are
// FP64 either way. FLUX: rho u_a^3 as well, which only the FP64 step reads
// (all diagnostics of 160^3 3315 -> 3217 us without it).
template <int LAT, bool FLUX, typename P>
__global__ void k_macro(Geo g, Phys p, const uint8_t *__restrict__ mask, P f, double2 *__restrict__ rp,
                        double *__restrict__ u, double *__restrict__ gflux, int *__restrict__ status)
{
    constexpr int D = Lattice<LAT>::D;
    lbmpdl::step_trigger();
    lbmpdl::step_wait();
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    if (x >= g.nx) return;
    const int y = blockIdx.y, z = blockIdx.z;
    const unsigned n = entry(g, x, y, z);
    const bool solid = mask[n];
    double rho, j[3];
    node_sums<LAT, false>(g, f, n, x, y, z, rho, j, nullptr, solid);
    if (solid) return;
    double inv;
    const double d = excess_pressure(p, rho, inv);
    bool ok = positive(rho) && finite_bits(rho);
    rp[n] = make_double2(rho, signed_psi_of(d));
#pragma unroll
    for (int a = 0; a < D; ++a) {
        const double ua = j[a] * inv;
        u[a * g.N + n] = ua;
        if (FLUX) gflux[a * g.N + n] = j[a] * ua * ua;   // rho u_a^3
        ok = ok && finite_bits(ua);
    }
    if (!ok) atomicOr(status, 1);
}

// Force, correction, product-form collision and push streaming with
// halfway bounce-back (Eqs. LBGK, LBMeq, LBMstar): the body of the force
// sweep for the FP64 step. REST: relaxation time 1, where post = f* and
// neither f nor feq is needed.
template <int LAT, bool REST>
struct CollideBody {
    const uint8_t *mask;
    const double *f;
    double *fout;
    const double2 *rp;
    const double *u, *gflux;

    __device__ __forceinline__ void operator()(const Geo &g, const Phys &p, unsigned n, int x, int y, int z,
                                               const double *sp, const double *sr) const
    {
        constexpr int D = Lattice<LAT>::D, Q = Lattice<LAT>::Q;
        const int X[3] = {wrapm(x - 1, g.nx), x, wrapp(x + 1, g.nx)};
        const int Y[3] = {wrapm(y - 1, g.ny), y, wrapp(y + 1, g.ny)};
        const int Z[3] = {D == 3 ? wrapm(z - 1, g.nz) : 0, z, D == 3 ? wrapp(z + 1, g.nz) : 0};
        const auto at = [&](int cx, int cy, int cz) {
            return entry(g, X[cx + 1], Y[cy + 1], Z[cz + 1]);
        };
        // everything read but the populations, in one round trip
        const bool solid = mask[n];
        const double2 c = rp[n];
        double un[3], dg[3];
#pragma unroll
        for (int a = 0; a < D; ++a) {
            un[a] = u[a * (size_t)g.N + n];
            dg[a] = gflux[a * (size_t)g.N + at(a == 0, a == 1, a == 2)] -
                    gflux[a * (size_t)g.N + at(-(a == 0), -(a == 1), -(a == 2))];
        }
        unsigned walls = 0;   // bit i: the destination of population i is solid
#pragma unroll
        for (int i = 0; i < Q; ++i)
            walls |= (unsigned)mask[at(cxi(i), cyi(i), D == 3 ? czi(i) : 0)] << i;
        if (solid) return;
        const double rho = c.x;
        double F[3];
        force_of_sums<LAT>(p, rho, c.y, sp, sr, F);
        // Phi_aa = -(1 - omega/2) (g_a(r + e_a) - g_a(r - e_a)) / 2, the node's omega
        const double om = REST ? 1.0 : omega_at(p, rho);
        const double pref = p.var_visc ? p.phi_sign * (1.0 - 0.5 * om) : p.phi_pref;
        // Product-form factors: equilibrium (xi = u, zeta = 1/3 + u^2) and
        // extended (xi* = u + F/rho, zeta* = 1/3 + xi*^2 + Phi/rho), as
        // (zeta -+ xi)/2 and 1 - zeta.
        const double inv = 1.0 / rho, ph = 0.25 * pref * inv;
        double E[3][3], S[3][3];
#pragma unroll
        for (int a = 0; a < D; ++a) {
            const double ua = un[a];
            if (!REST) {
                const double t = 0.5 * ua, h = fma(t, ua, 1.0 / 6.0);
                E[a][0] = h - t;
                E[a][1] = fma(-2.0, h, 1.0);
                E[a][2] = h + t;
            }
            const double xs = fma(F[a], inv, ua), t = 0.5 * xs;
            const double h = fma(ph, dg[a], fma(t, xs, 1.0 / 6.0));
            S[a][0] = h - t;
            S[a][1] = fma(-2.0, h, 1.0);
            S[a][2] = h + t;
        }
        // post = (1 - omega) f + (f* - (1 - omega) feq); feq and f* by x-y
        // partial products, the factor 1 - omega taken into feq's
        const double omw = 1.0 - om, ro = REST ? 0.0 : rho * omw;
        double Ae[3][3], As[3][3];
#pragma unroll
        for (int cx = 0; cx < 3; ++cx) {
            const double sx = rho * S[0][cx], ex = REST ? 0.0 : ro * E[0][cx];
#pragma unroll
            for (int cy = 0; cy < 3; ++cy) {
                As[cx][cy] = sx * S[1][cy];
                Ae[cx][cy] = REST ? 0.0 : ex * E[1][cy];
            }
        }
#pragma unroll
        for (int i = 0; i < Q; ++i) {
            const int cx = cxi(i), cy = cyi(i), cz = D == 3 ? czi(i) : 0;
            double post = D == 3 ? As[cx + 1][cy + 1] * S[2][cz + 1] : As[cx + 1][cy + 1];
            if (!REST) {
                post = D == 3 ? fma(-Ae[cx + 1][cy + 1], E[2][cz + 1], post) : post - Ae[cx + 1][cy + 1];
                post = fma(omw, f[(size_t)i * g.N + n], post);
            }
            if (walls >> i & 1u) fout[(size_t)(Q - 1 - i) * g.N + n] = post;
            else                 fout[(size_t)i * g.N + at(cx, cy, cz)] = post;
        }
    }
};

// Output moments: rho, bare u and U = u + F/(2 rho) (Sec. 2.3.5).
// Without U no force is needed.
template <int LAT>
__global__ void k_moments_out(Geo g, Phys p, const uint8_t *__restrict__ mask,
                              const double2 *__restrict__ rp, const double *__restrict__ u,
                              double *__restrict__ rho_out, double *__restrict__ u_out)
{
    constexpr int D = Lattice<LAT>::D;
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    if (x >= g.nx) return;
    const int y = blockIdx.y, z = blockIdx.z;
    const unsigned n = entry(g, x, y, z);
    const unsigned m = entry(flat(g), x, y, z);
    const bool solid = mask[n];
    if (rho_out) rho_out[m] = solid ? p.rho_w : rp[n].x;
#pragma unroll
    for (int a = 0; a < D; ++a)
        if (u_out) u_out[a * (size_t)g.M + m] = solid ? 0.0 : u[a * (size_t)g.N + n];
}

// The same with U: the body of the force sweep.
template <int LAT>
struct MomentsBody {
    const uint8_t *mask;
    const double2 *rp;
    const double *u;
    double *rho_out, *u_out, *U_out;

    __device__ __forceinline__ void operator()(const Geo &g, const Phys &p, unsigned n, int x, int y, int z,
                                               const double *sp, const double *sr) const
    {
        constexpr int D = Lattice<LAT>::D;
        const unsigned m = entry(flat(g), x, y, z);
        const bool solid = mask[n];
        const double2 c = solid ? make_double2(p.rho_w, 0.0) : rp[n];
        double F[3];
        force_of_sums<LAT>(p, c.x, c.y, sp, sr, F);
        const double half = 0.5 / c.x;
        if (rho_out) rho_out[m] = c.x;
#pragma unroll
        for (int a = 0; a < D; ++a) {
            const double ua = solid ? 0.0 : u[a * (size_t)g.N + n];
            if (u_out) u_out[a * (size_t)g.M + m] = ua;
            U_out[a * (size_t)g.M + m] = solid ? 0.0 : fma(F[a], half, ua);
        }
    }
};

// Interpolated (linear Bouzidi) bounce-back, after a push step with halfway
// bounce-back, one boundary node per thread. For each active link of node n
// along c_i into a solid, with the wall at the fraction q of the link
// (ib = Q-1-i; f_ib(n) holds f_i*(n), f_i(n) holds f_i*(n - c_i),
// f_ib(n - c_i) holds f_ib*(n)):
//   q < 1/2:  f_ib(n) = 2q f_i*(n) + (1 - 2q) f_i*(n - c_i)
//   q >= 1/2: f_ib(n) = f_i*(n) / (2q) + (2q - 1)/(2q) f_ib*(n)
// and the node returns the sum of its links' changes through its rest
// population (mass-conserving). Active links have n - c_i fluid, so no
// thread reads what another writes.
template <int LAT, typename T>
__global__ void k_interp_bounce_back(Geo g, const unsigned *__restrict__ bn,
                                     const unsigned *__restrict__ bmask,
                                     const double *__restrict__ bq, int nb, T *__restrict__ f)
{
    constexpr int D = Lattice<LAT>::D, Q = Lattice<LAT>::Q;
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= nb) return;
    const unsigned id = bn[b], m = bmask[b];   // id: without row padding
    const int x = id % g.nx, y = (id / g.nx) % g.ny, z = id / (g.nx * g.ny);
    const unsigned n = entry(g, x, y, z);
    T excess = T(0);
    for (int i = 0; i < Q; ++i) {
        if (!((m >> i) & 1u)) continue;
        const T q = (T)bq[(size_t)b * Q + i];
        const int ib = Q - 1 - i;
        const T a = f[(size_t)ib * g.N + n];
        T v;
        if (q < T(0.5)) {
            v = T(2) * q * a + (T(1) - T(2) * q) * f[(size_t)i * g.N + n];
        } else {
            const int xm = (x - cxi(i) + g.nx) % g.nx, ym = (y - cyi(i) + g.ny) % g.ny;
            const int zm = D == 3 ? (z - czi(i) + g.nz) % g.nz : 0;
            const unsigned nm = entry(g, xm, ym, zm);
            v = a / (T(2) * q) + (T(2) * q - T(1)) / (T(2) * q) * f[(size_t)ib * g.N + nm];
        }
        f[(size_t)ib * g.N + n] = v;
        excess += v - a;
    }
    f[(size_t)(Q / 2) * g.N + n] -= excess;
}

// Discrete pressure tensor (Appendix E) at fluid nodes: the populations'
// momentum flux sum_i c_ia c_ib f_i plus the non-local parts of the four
// ring terms of the force, with the sign of the force on the fluid:
//   s 4/3 psi S1[psi] - s/6 (psi S2[psi] + X[psi]) + kappa rho S1[rho]
//   - kappa/2 (rho S2[rho] + X[rho]),
// S_k[v] = sum_i (w_i/cs2) c_ia c_ib v(r + k c_i),
// X[v] = sum_i (w_i/cs2) c_ia c_ib v(r - c_i) v(r + c_i).
// Needs rp of the current state (k_macro). Components xx, yy[, zz],
// xy[, xz, yz] as N-planes; 0 at solid nodes.
// All terms but the populations' are linear in what a pair of opposite
// neighbours gives with the weight w_i c_ia c_ib, so each of the 13 (4)
// pairs forms its sum T of all terms once (12 FP64 operations) and the T are
// added by weight class: about 220 operations per node where term by term
// and component by component took 1200 (160^3: 11.1 ms).
template <int LAT, typename P>
__global__ void k_pressure_tensor(Geo g, Phys p, const uint8_t *__restrict__ mask, P f,
                                  const double2 *__restrict__ rp, double *__restrict__ out)
{
    constexpr int D = Lattice<LAT>::D, Q = Lattice<LAT>::Q, NA = D == 3 ? 6 : 3;
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    if (x >= g.nx) return;
    const int y = blockIdx.y, z = blockIdx.z;
    const unsigned n = entry(g, x, y, z), m = entry(flat(g), x, y, z);
    constexpr int CA[6] = {0, 1, D == 3 ? 2 : 0, 0, 0, 1};
    constexpr int CB[6] = {0, 1, D == 3 ? 2 : 1, 1, 2, 2};
    if (mask[n]) {
#pragma unroll
        for (int k = 0; k < NA; ++k) out[(size_t)k * g.M + m] = 0.0;
        return;
    }
    double rho, j[3], kin[6];
    node_sums<LAT, true>(g, f, n, x, y, z, rho, j, kin);
    const double2 c0 = rp[n];
    const double r = c0.x, sps = c0.y;   // s psi; s = +1 where P > P0, else -1
    const double s6 = positive(sps) ? -1.0 / 3.0 : 1.0 / 3.0;
    const double c1 = 4.0 / 3.0 * sps, c2 = -1.0 / 6.0 * sps;
    const double c3 = p.kappa * r, c4 = -0.5 * c3;
    int X[5], Y[5], Z[5];
#pragma unroll
    for (int k = -2; k <= 2; ++k) {
        X[k + 2] = k < 0 ? wrapm(x + k, g.nx) : wrapp(x + k, g.nx);
        Y[k + 2] = k < 0 ? wrapm(y + k, g.ny) : wrapp(y + k, g.ny);
        Z[k + 2] = D == 2 ? 0 : k < 0 ? wrapm(z + k, g.nz) : wrapp(z + k, g.nz);
    }
    // sums of T by component and weight class (nonzero components of c less one)
    double acc[6][3];
    bool set[6][3] = {};
#pragma unroll
    for (int i = Q / 2 + 1; i < Q; ++i) {
        const int c[3] = {cxi(i), cyi(i), D == 3 ? czi(i) : 0};
        const auto at = [&](int k) {
            return rp[entry(g, X[k * c[0] + 2], Y[k * c[1] + 2], Z[k * c[2] + 2])];
        };
        const double2 p1 = at(1), m1 = at(-1), p2 = at(2), m2 = at(-2);
        double T = c1 * (fabs(p1.y) + fabs(m1.y));
        T = fma(c2, fabs(p2.y) + fabs(m2.y), T);
        T = fma(s6, fabs(p1.y * m1.y), T);
        T = fma(c3, p1.x + m1.x, T);
        T = fma(c4, p2.x + m2.x, T);
        T = fma(-p.kappa, p1.x * m1.x, T);
        const int cls = (c[0] != 0) + (c[1] != 0) + (c[2] != 0) - 1;
#pragma unroll
        for (int k = 0; k < NA; ++k) {
            const int cc = c[CA[k]] * c[CB[k]];
            if (cc == 0) continue;
            acc[k][cls] = !set[k][cls] ? (cc > 0 ? T : -T) : cc > 0 ? acc[k][cls] + T : acc[k][cls] - T;
            set[k][cls] = true;
        }
    }
    // 3 w_i of the classes
    const double w[3] = {D == 3 ? 2.0 / 9.0 : 1.0 / 3.0, D == 3 ? 1.0 / 18.0 : 1.0 / 12.0, 1.0 / 72.0};
#pragma unroll
    for (int k = 0; k < NA; ++k) {
        double v = kin[k];
#pragma unroll
        for (int cls = 0; cls < D; ++cls)
            if (set[k][cls]) v = fma(w[cls], acc[k][cls], v);
        out[(size_t)k * g.M + m] = v;
    }
}

// Side field of the initial density: rp = (rho0, s psi(rho0)) at fluid nodes
// (solid nodes get theirs from k_fill_solid).
template <int LAT>
__global__ void k_init_density(Geo g, Phys p, const uint8_t *__restrict__ mask,
                               const double *__restrict__ rho0, double2 *__restrict__ rp)
{
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    if (x >= g.nx) return;
    const int y = blockIdx.y, z = blockIdx.z;
    const unsigned n = entry(g, x, y, z);
    if (mask[n]) return;
    const double rho = rho0[entry(flat(g), x, y, z)];
    rp[n] = make_double2(rho, signed_psi(p, rho));
}

// Korteweg force at one node, summed by itself: for the initial state, which is
// formed once and stays the same to the bit whatever the step's sums do (the
// last bit of an FP64 sum decides, once in a while, how a population rounds to
// 16 or 32 bits, and a density ratio of 1e4 carries that far).
//   F = -2 (s psi)_c S_psi - kappa rho_c S_rho + rho_c g,
//   S_psi = sum_i (w_i/cs2) c_i [4/3 psi(r+c_i) - 1/6 psi(r+2c_i)],
//   S_rho = sum_i (w_i/cs2) c_i [2 rho(r+c_i) - rho(r+2c_i)]   (Eq. Kforce_final).
// w_i/cs2 c_ia = 1/2 W(c_ib) W(c_ic) c_ia with the 1D weights W(0) = 2/3,
// W(+-1) = 1/6 of Eq. wi, so each ring sums neighbours by their number of
// nonzero transverse components (centre, edge, corner) before weighting.
template <int LAT>
__device__ __forceinline__ void korteweg_force(const Geo &g, const Phys &p,
                                               const double2 *__restrict__ rp, int x, int y,
                                               int z, double rho_c, double spsi_c, double *F)
{
    constexpr int D = Lattice<LAT>::D;
    double Spsi[3] = {0.0, 0.0, 0.0}, Srho[3] = {0.0, 0.0, 0.0};
#pragma unroll
    for (int s = 1; s <= 2; ++s) {
        const int xm = wrapm(x - s, g.nx), xp = wrapp(x + s, g.nx);
        const int ym = wrapm(y - s, g.ny), yp = wrapp(y + s, g.ny);
        int zm = 0, zp = 0;
        if (D == 3) { zm = wrapm(z - s, g.nz); zp = wrapp(z + s, g.nz); }
        const int X[3] = {xm, x, xp}, Y[3] = {ym, y, yp}, Z[3] = {zm, z, zp};
        double ap[3][3], ar[3][3];  // [component][0 centre, 1 edge, 2 corner]
#pragma unroll
        for (int a = 0; a < 3; ++a)
#pragma unroll
            for (int k = 0; k < 3; ++k) { ap[a][k] = 0.0; ar[a][k] = 0.0; }
        // each pair (c_i, -c_i) once: differences of the two neighbours, added
        // with the sign of c_ia to every component where c_ia != 0
#pragma unroll
        for (int i = Lattice<LAT>::Q / 2 + 1; i < Lattice<LAT>::Q; ++i) {
            const int c[3] = {cxi(i), cyi(i), D == 3 ? czi(i) : 0};
            const unsigned np_ = entry(g, X[c[0] + 1], Y[c[1] + 1], Z[c[2] + 1]);
            const unsigned nm_ = entry(g, X[1 - c[0]], Y[1 - c[1]], Z[1 - c[2]]);
            const double2 vp = rp[np_], vm = rp[nm_];
            const double dps = fabs(vp.y) - fabs(vm.y);
            const double drh = vp.x - vm.x;
#pragma unroll
            for (int a = 0; a < D; ++a) {
                if (c[a] == 0) continue;
                const int k = (a != 0 && c[0] != 0) + (a != 1 && c[1] != 0) + (a != 2 && c[2] != 0);
                if (c[a] > 0) { ap[a][k] += dps; ar[a][k] += drh; }
                else          { ap[a][k] -= dps; ar[a][k] -= drh; }
            }
        }
        const double gp = s == 1 ? 4.0 / 3.0 : -1.0 / 6.0;
        const double gr = s == 1 ? 2.0 : -1.0;
#pragma unroll
        for (int a = 0; a < D; ++a) {
            double dp, dr;
            if (D == 3) {
                dp = (2.0 / 9.0) * ap[a][0] + (1.0 / 18.0) * ap[a][1] + (1.0 / 72.0) * ap[a][2];
                dr = (2.0 / 9.0) * ar[a][0] + (1.0 / 18.0) * ar[a][1] + (1.0 / 72.0) * ar[a][2];
            } else {
                dp = (1.0 / 3.0) * ap[a][0] + (1.0 / 12.0) * ap[a][1];
                dr = (1.0 / 3.0) * ar[a][0] + (1.0 / 12.0) * ar[a][1];
            }
            Spsi[a] += gp * dp;
            Srho[a] += gr * dr;
        }
    }
#pragma unroll
    for (int a = 0; a < D; ++a) F[a] = -2.0 * spsi_c * Spsi[a] - p.kappa * rho_c * Srho[a] + rho_c * p.g[a];
}

// Initial populations at rest in the physical velocity: the equilibrium at
// the bare velocity u = U0 - F/(2 rho0), F the Korteweg force of the initial
// density (rp, filled by k_init_density and k_fill_solid), so that
// U = u + F/(2 rho) of Sec. 2.3.5 equals U0 at t = 0. Zero at solid nodes.
template <int LAT, typename T = double>
__global__ void k_init(Geo g, Phys p, const uint8_t *__restrict__ mask,
                       const double2 *__restrict__ rp, const double *__restrict__ u0,
                       T *__restrict__ f)
{
    constexpr int D = Lattice<LAT>::D, Q = Lattice<LAT>::Q;
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    if (x >= g.nx) return;
    const int y = blockIdx.y, z = blockIdx.z;
    const unsigned n = entry(g, x, y, z), m = entry(flat(g), x, y, z);
    if (mask[n]) {
#pragma unroll
        for (int i = 0; i < Q; ++i) f[(size_t)i * g.N + n] = (T)0;
        return;
    }
    const double2 c = rp[n];
    const double rho = c.x;
    double F[3] = {0.0, 0.0, 0.0};
    korteweg_force<LAT>(g, p, rp, x, y, z, rho, c.y, F);
    double E[3][3];
#pragma unroll
    for (int a = 0; a < D; ++a) {
        const double ua = (u0 ? u0[a * (size_t)g.M + m] : 0.0) - F[a] / (2.0 * rho);
        const double ze = 1.0 / 3.0 + ua * ua;
        E[a][0] = 0.5 * (ze - ua);
        E[a][1] = 1.0 - ze;
        E[a][2] = 0.5 * (ze + ua);
    }
#pragma unroll
    for (int i = 0; i < Q; ++i) {
        double eq = rho * E[0][cxi(i) + 1] * E[1][cyi(i) + 1];
        if (D == 3) eq *= E[2][czi(i) + 1];
        f[(size_t)i * g.N + n] = (T)eq;
    }
}

template <int LAT>
__global__ void k_fill_solid(Geo g, Phys p, const uint8_t *__restrict__ mask,
                             double2 *__restrict__ rp, double *__restrict__ u,
                             double *__restrict__ gflux)
{
    constexpr int D = Lattice<LAT>::D;
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    if (x >= g.nx) return;
    const int y = blockIdx.y, z = blockIdx.z;
    const unsigned n = entry(g, x, y, z);
    if (!mask[n]) return;
    rp[n] = make_double2(p.rho_w, signed_psi(p, p.rho_w));
#pragma unroll
    for (int a = 0; a < D; ++a) {
        u[a * g.N + n] = 0.0;
        if (gflux) gflux[a * g.N + n] = 0.0;
    }
}

// Wall bits of the planes near solids (GeoF::walls): bit i of node (x, y, z): its
// neighbour along c_i is solid. planes: the z of each plane.
__global__ void k_wall_bits(Geo g, const uint8_t *__restrict__ mask, const int *__restrict__ planes,
                            unsigned *__restrict__ walls)
{
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    if (x >= g.nx) return;
    const int y = blockIdx.y, z = planes[blockIdx.z];
    const int X[3] = {wrapm(x - 1, g.nx), x, wrapp(x + 1, g.nx)};
    const int Y[3] = {wrapm(y - 1, g.ny), y, wrapp(y + 1, g.ny)};
    const int Z[3] = {wrapm(z - 1, g.nz), z, wrapp(z + 1, g.nz)};
    unsigned w = 0;
#pragma unroll
    for (int i = 0; i < 27; ++i)
        w |= (unsigned)mask[entry(g, X[cxi(i) + 1], Y[cyi(i) + 1], Z[czi(i) + 1])] << i;
    walls[(size_t)g.px * g.ny * blockIdx.z + (unsigned)x + (unsigned)g.px * (unsigned)y] = w;
}

// Mass and momentum: fixed grid, fixed per-thread stride order and a fixed
// shuffle tree, so the sums are bitwise reproducible run to run.
constexpr int RED_THREADS = 256;
constexpr int RED_BLOCKS = 1024;

__device__ __forceinline__ double warp_sum(double v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

template <int LAT, typename P>
__global__ void __launch_bounds__(RED_THREADS)
k_reduce_partial(Geo g, const uint8_t *__restrict__ mask, P f, double *__restrict__ partial)
{
    constexpr int D = Lattice<LAT>::D;
    double acc[4] = {0.0, 0.0, 0.0, 0.0};
    const unsigned plane = (unsigned)g.px * (unsigned)g.ny;
    for (unsigned n = blockIdx.x * RED_THREADS + threadIdx.x; n < g.N;
         n += RED_THREADS * RED_BLOCKS) {
        if (mask[n]) continue;   // the rows' padding too: its mask is 1
        const unsigned z = n / plane, y = (n - z * plane) / g.px, x = n - z * plane - y * g.px;
        double rho, j[3];
        node_sums<LAT, false>(g, f, n, x, y, z, rho, j);
        acc[0] += rho;
#pragma unroll
        for (int a = 0; a < D; ++a) acc[1 + a] += j[a];
    }
    __shared__ double sh[4][RED_THREADS / 32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const double v = warp_sum(acc[k]);
        if (lane == 0) sh[k][w] = v;
    }
    __syncthreads();
    if (threadIdx.x < 32) {
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            double v = lane < RED_THREADS / 32 ? sh[k][lane] : 0.0;
            v = warp_sum(v);
            if (lane == 0) partial[4 * blockIdx.x + k] = v;
        }
    }
}

__global__ void __launch_bounds__(RED_BLOCKS)
k_reduce_final(const double *__restrict__ partial, double *__restrict__ out)
{
    __shared__ double sh[4][RED_BLOCKS / 32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const double v = warp_sum(partial[4 * threadIdx.x + k]);
        if (lane == 0) sh[k][w] = v;
    }
    __syncthreads();
    if (threadIdx.x < 32) {
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const double v = warp_sum(sh[k][lane]);
            if (lane == 0) out[k] = v;
        }
    }
}

// Shifted 16-bit storage (h_i = f_i / rho(src) - w_i, src = r - c_i, or r itself
// when r - c_i is solid): decode to FP64, per-node densities, encode.
template <int LAT, typename ST>
__global__ void k_decode_shifted(Geo g, const ST *__restrict__ h, const float *__restrict__ rho_src,
                                 double *__restrict__ f)
{
    constexpr int D = Lattice<LAT>::D, Q = Lattice<LAT>::Q;
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    if (x >= g.nx) return;
    const int y = blockIdx.y, z = blockIdx.z;
    const unsigned n = entry(g, x, y, z), m = entry(flat(g), x, y, z);
#pragma unroll
    for (int i = 0; i < Q; ++i) {
        // a solid source (density -1) means a population bounced by n itself
        float src = rho_src[source_node(g, D, i, x, y, z)];
        if (src < 0.0f) src = rho_src[n];
        f[(size_t)i * g.M + m] = (weight_d(i, D) + widen(lbmf::to_f(h[(size_t)i * g.N + n]))) * widen(src);
    }
}

// The source-density field of shifted storage, written to both buffers (-1 at
// solid nodes stays for good): each fluid node's density, -1 at solid nodes
// (their populations' sources are the fluid nodes that bounced them; see the
// decoders).
// gf: the layout of f (the caller's or the library's). INIT: the initial state,
// summed in FP64 one after the other.
template <int LAT, bool INIT>
__global__ void k_density(Geo g, Geo gf, const uint8_t *__restrict__ mask, const double *__restrict__ f,
                          float *__restrict__ rho0, float *__restrict__ rho1)
{
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    if (x >= g.nx) return;
    const int y = blockIdx.y, z = blockIdx.z;
    const unsigned n = entry(g, x, y, z);
    float v = -1.0f;
    if (!mask[n]) {
        double s = 0.0, j[3];
        const unsigned m = entry(gf, x, y, z);
        if constexpr (INIT) {
#pragma unroll
            for (int i = 0; i < Lattice<LAT>::Q; ++i) s += f[(size_t)i * gf.N + m];
        } else {
            node_sums<LAT, false>(gf, f, m, x, y, z, s, j);
        }
        v = (float)s;
    }
    rho0[n] = rho1[n] = v;
}

// d rounded to nearest even in FP32, as the conversion, which takes as long as
// an FP64 operation, does; results that are not normal FP32 numbers by it.
__device__ __forceinline__ float narrow(double d)
{
    const unsigned hi = (unsigned)__double2hiint(d), lo = (unsigned)__double2loint(d);
    const unsigned e = hi & 0x7ff00000u;
    if (e < 0x38200000u || e > 0x47c00000u) return (float)d;   // below 2^-125, above 2^125
    const unsigned top = (((hi & 0x7fffffffu) - 0x38000000u) << 3) | (lo >> 29), drop = lo << 3;
    return __uint_as_float((hi & 0x80000000u) | (top + (drop > 0x80000000u || (drop == 0x80000000u && (top & 1u)))));
}

// (float)(f / v - w) in 5 FP64 operations: the quotient starts from the FP32
// one and is corrected twice by its exact remainder, a fused multiply-add's
// (P. W. Markstein, IBM J. Res. Dev. 34, 1990, 111; to 2^-70, so its FP64
// rounding is the division's but for about 1 in 10^5). Encoding 128x96x112
// with its densities: 426 us, with a multiplication by 1/v first and the
// conversion instruction (7 operations) 544 us.
__device__ __forceinline__ float shifted_of(double f, float v, double w)
{
    const unsigned hi = (unsigned)__double2hiint(f), ef = (hi >> 20) & 0x7ff, ev = (__float_as_uint(v) >> 23) & 0xff;
    if (ef - 963u > 120u || ev - 67u > 120u) return (float)(f / (double)v - w);   // outside 2^-60 .. 2^60
    const float f32 = __uint_as_float((hi & 0x80000000u) | (((hi & 0x7fffffffu) - 0x38000000u) << 3));
    const float r32 = __frcp_rn(v);
    const double d = widen(v), r = widen(r32);
    double q = widen(f32 * r32);
    q = fma(fma(-d, q, f), r, q);
    q = fma(fma(-d, q, f), r, q);
    return narrow(q - w);
}

template <int LAT, typename ST>
__global__ void k_encode_shifted(Geo g, Geo gf, const double *__restrict__ f, const float *__restrict__ rho,
                                 ST *__restrict__ h)
{
    constexpr int D = Lattice<LAT>::D, Q = Lattice<LAT>::Q;
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    if (x >= g.nx) return;
    const int y = blockIdx.y, z = blockIdx.z;
    const unsigned n = entry(g, x, y, z), m = entry(gf, x, y, z);
    if (rho[n] < 0.0f) {   // solid: no populations
#pragma unroll
        for (int i = 0; i < Q; ++i) h[(size_t)i * g.N + n] = lbmf::from_f<ST>(0.0f);
        return;
    }
#pragma unroll
    for (int i = 0; i < Q; ++i) {
        float src = rho[source_node(g, D, i, x, y, z)];
        if (src < 0.0f) src = rho[n];   // bounced by n itself
        h[(size_t)i * g.N + n] =
            lbmf::from_f<ST>(shifted_of(f[(size_t)i * gf.N + m], src, weight_d(i, D)));
    }
}

// Population I/O of FP32 storage: `rows` rows of nx populations (of all
// directions, one after the other) from rows of pa entries of type A to rows of
// pb of type B. One population a thread and turn: a node a thread, 27 populations
// each, took 1.4 times as long on 16^3 (32 us against 22).
template <typename A, typename B>
__global__ void __launch_bounds__(256)
k_convert(unsigned rows, unsigned nx, unsigned pa, unsigned pb, const A *__restrict__ in, B *__restrict__ out)
{
    const size_t n = (size_t)rows * nx;
    for (size_t k = blockIdx.x * 256u + threadIdx.x; k < n; k += (size_t)gridDim.x * 256u) {
        size_t a = k, b = k;
        if (pa != nx || pb != nx) {
            const unsigned r = (unsigned)k / nx, x = (unsigned)k - r * nx;   // (at most 4e9 populations)
            a = (size_t)r * pa + x;
            b = (size_t)r * pb + x;
        }
        if constexpr (sizeof(B) == 8) out[b] = widen(in[a]);
        else                          out[b] = (B)in[a];
    }
}

// FP64 throughput probe: eight independent fused multiply-add chains per
// thread (two flops each), iters rounds, the chains' sum stored so that none
// is eliminated. a -> a b + c with b = 1 - 2^-20 and c = 2^-20 stays near 1
// (no overflow, no subnormals).
__global__ void k_fp64_fma_probe(double *__restrict__ out, int iters)
{
    double a[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) a[k] = 1.0 + 1e-3 * (threadIdx.x + k);
    const double b = 1.0 - 0x1p-20, c = 0x1p-20;
    for (int it = 0; it < iters; ++it)
#pragma unroll
        for (int k = 0; k < 8; ++k) a[k] = fma(a[k], b, c);
    double s = 0.0;
#pragma unroll
    for (int k = 0; k < 8; ++k) s += a[k];
    out[blockIdx.x * blockDim.x + threadIdx.x] = s;
}

}  // namespace lbmk
