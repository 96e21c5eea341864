// D2Q9 fused step for reduced storage (FP32 or 16-bit shifted populations,
// FP32 arithmetic): one 32 x 8 tile per block, in one shot.
//
// A 2D lattice of the sizes in use (64^2 .. 512^2) has few nodes and lives in
// L2, so what bounds it is latency and how many SMs take part, not
// bandwidth. A block therefore marches along nothing: every thread loads its
// own node and its share of the 2-node halo at once (one memory round trip),
// forms (rho, |psi|) and rho u_a^3 into shared memory, synchronises once,
// and collides its own node, whose populations and moments stayed in
// registers. Forming the halo's moments again in each tile costs 36 x 12 /
// (32 x 8) = 1.7 times the moments; they are a small part of the step.
// Measured (us per step, graph replays, FP32 / FP16-shifted, time 1) against the
// tile of 128 x 1 nodes marching along y that ran before, at its default
// chunk of 64 rows: 512^2 6.2 / 7.7 against 90 / 140 (17 / 25 at its best
// chunk, 4), 64^2 2.6 / 3.1 against 72. 32 x 4 tiles: the same up to 256^2,
// 10-20 % slower above.
// The arithmetic is that of the D3Q27 tile (node_moments, force_f,
// factors_f). In the frame of LatF<0> the 2D y axis is z.
//
// Included by the 8-row build of the fused tile only.
#pragma once

#include "lbm_fused_f32.cuh"
#include "lbm_pdl.cuh"

namespace lbmf2 {

using namespace lbmf;

constexpr int TX = 32, TY = 8, NT = TX * TY;   // the tile; one thread per node

struct Shared2 {
    static constexpr int AX = TX + 4, AY = TY + 4;   // (rho, |psi|) halo tile
    static constexpr int GX = TX + 2, GY = TY + 2;   // rho u^3 halo tile
    float2 rp[AY][AX];
    float g[2][GY][GX];   // rho u_x^3, rho u_y^3
};

// v modulo n for v >= -n, without a division for v < 2 n (a lattice narrower
// than the tile wraps more than once).
__device__ __forceinline__ int wrap_any(int v, int n)
{
    v = v < 0 ? v + n : v;
    if (v >= n) {
        v -= n;
        if (v >= n) v %= n;
    }
    return v;
}

// Halo node k of the tile: interior nodes first (a thread's first node is
// the one it collides), then the two rows above, the two below, and two
// columns on either side of each interior row.
__device__ __forceinline__ void halo2(int k, int &r, int &c)
{
    constexpr int AX = Shared2::AX, AY = Shared2::AY;
    if (k < NT) {
        r = (k >> 5) + 2;
        c = (k & 31) + 2;
        return;
    }
    int m = k - NT;
    if (m < 4 * AX) {
        const int q = m / AX;
        r = q < 2 ? q : AY - 4 + q;
        c = m - q * AX;
        return;
    }
    m -= 4 * AX;
    const int e = m & 3;
    r = 2 + (m >> 2);
    c = e < 2 ? e : AX - 4 + e;
}

template <bool MASK, typename ST, bool E64, bool REST>
__device__ __forceinline__ void tile2d(const GeoF &g, const PhysF &p, const uint8_t *__restrict__ mask,
                                       const ST *f, ST *__restrict__ fout, int *__restrict__ status, int bx,
                                       int by, Shared2 &sm, const float *rho_src, float *__restrict__ rho_dst)
{
    constexpr bool SHIFT = IsShifted<ST>::value;
    using L = LatF<0>;
    using S = Shared2;
    constexpr int Q = L::Q, NH = S::AX * S::AY, KA = (NH + NT - 1) / NT;
    const int tid = threadIdx.x;
    const int x0 = bx * TX, y0 = by * TY, nx = g.nx, ny = g.nz;
    const unsigned N = g.N;
    float fi[KA][Q];
    bool live[KA], solid[KA];
#pragma unroll
    for (int u = 0; u < KA; ++u) {
        const int k = tid + u * NT;
        live[u] = k < NH;
        int r, c;
        halo2(live[u] ? k : 0, r, c);
        const int x = wrap_any(x0 - 2 + c, nx), y = wrap_any(y0 - 2 + r, ny);
        const unsigned n = (unsigned)x + (unsigned)g.px * (unsigned)y;
        solid[u] = MASK && live[u] && mask[n];
        if (!live[u] || solid[u]) continue;
        if constexpr (SHIFT) {
            // population i: (w_i + h_i) times the density of its source node r - c_i,
            // or of the node itself where the source is solid (density -1)
            const int X[3] = {wrapf(x + 1, nx), x, wrapf(x - 1, nx)};
            const int Y[3] = {wrapf(y + 1, ny), y, wrapf(y - 1, ny)};
            float src[Q];
#pragma unroll
            for (int i = 0; i < Q; ++i)
                src[i] = rho_src[(unsigned)X[L::cx(i) + 1] + (unsigned)g.px * (unsigned)Y[L::cz(i) + 1]];
#pragma unroll
            for (int i = 0; i < Q; ++i) {
                const float own = MASK && src[i] < 0.0f ? src[Q / 2] : src[i];
                fi[u][i] = (weight_f<0>(i) + to_f(f[i * N + n])) * own;
            }
        } else {
#pragma unroll
            for (int i = 0; i < Q; ++i) fi[u][i] = to_f(f[i * N + n]);
        }
    }
    NodeM own = {};
    float psi0 = 0.0f;
#pragma unroll
    for (int u = 0; u < KA; ++u) {
        if (!live[u]) continue;
        int r, c;
        halo2(tid + u * NT, r, c);
        const bool ring1 = u == 0 || (c >= 1 && c < S::AX - 1 && r >= 1 && r < S::AY - 1);
        NodeM m = {};
        if (solid[u]) {
            m.rho = p.rho_w;
            m.d = p.spsi_w;
        } else {
            m = node_moments<0, E64>(p, fi[u], ring1);
        }
        const float psi = E64 && !solid[u] ? m.psi64 : sqrtf(fabsf(m.d));
        sm.rp[r][c] = f2(m.rho, psi);
        if (ring1) {
            sm.g[0][r - 1][c - 1] = m.gx;
            sm.g[1][r - 1][c - 1] = m.gz;
        }
        if (u == 0) {
            own = m;
            psi0 = psi;
        }
    }
    __syncthreads();
    const int tx = tid & 31, ty = tid >> 5, x = x0 + tx, y = y0 + ty;
    if (x >= nx || y >= ny || solid[0]) return;
    const unsigned n = (unsigned)x + (unsigned)g.px * (unsigned)y;
    const float rho = own.rho, spsi = (own.d > 0.0f ? 1.0f : -1.0f) * psi0;
    if (!(rho > 0.0f) || !isfinite(rho)) atomicOr(status, 1);
    if constexpr (SHIFT) rho_dst[n] = rho;   // source density of what this node pushes
    float F[3];
    force_f<0, E64>(p, rho, spsi, [&](int s, int cx, int, int cz) {
        return sm.rp[ty + 2 + s * cz][tx + 2 + s * cx];
    }, F);
    // Phi_aa = -(1 - omega/2) (g_a(r + e_a) - g_a(r - e_a)) / 2, the node's omega
    const float om = p.var_visc ? omega_var_f(p, rho) : p.omega;
    const float pref = p.var_visc ? p.phi_sign * (1.0f - 0.5f * om) : p.phi_pref;
    const float omw = p.var_visc ? 1.0f - om : p.omw;
    const float Phi[3] = {pref * 0.5f * (sm.g[0][ty + 1][tx + 2] - sm.g[0][ty + 1][tx]), 0.0f,
                          pref * 0.5f * (sm.g[1][ty + 2][tx + 1] - sm.g[1][ty][tx + 1])};
    const float inv = own.uv.w;
    const float un[3] = {own.uv.x, own.uv.y, own.uv.z};
    const PostF<0, REST, SHIFT> post(rho, inv, un, F, Phi, omw);
    // pushed to r + c_i (halfway bounce-back at solids)
    const int X[3] = {wrapf(x - 1, nx), x, wrapf(x + 1, nx)};
    const int Y[3] = {wrapf(y - 1, ny), y, wrapf(y + 1, ny)};
#pragma unroll
    for (int i = 0; i < Q; ++i) {
        const unsigned dst = (unsigned)X[L::cx(i) + 1] + (unsigned)g.px * (unsigned)Y[L::cz(i) + 1];
        if (MASK && mask[dst]) fout[(Q - 1 - i) * N + n] = from_f<ST>(post(i, fi[0]));
        else                   fout[i * N + dst] = from_f<ST>(post(i, fi[0]));
    }
}

template <bool MASK, typename ST, bool E64, bool REST>
__global__ void __launch_bounds__(NT)
k_step2d(GeoF g, PhysF p, const uint8_t *__restrict__ mask, const ST *f, ST *__restrict__ fout,
         const float *rho_src, float *__restrict__ rho_dst, int *__restrict__ status)
{
    __shared__ Shared2 sm;
    lbmpdl::step_trigger();
    lbmpdl::step_wait();
    tile2d<MASK, ST, E64, REST>(g, p, mask, f, fout, status, blockIdx.x, blockIdx.y, sm, rho_src, rho_dst);
}

// The same over the tiles of many lattices: block b takes item b.
template <typename ST, bool REST>
__global__ void __launch_bounds__(NT)
k_step2d_batch(const MemberF *__restrict__ members, const WorkItem *__restrict__ items)
{
    __shared__ Shared2 sm;
    const WorkItem w = items[blockIdx.x];
    const MemberF &m = members[w.member];
    lbmpdl::step_trigger();
    lbmpdl::step_wait();
    const ST *src = static_cast<const ST *>(m.src);
    ST *dst = static_cast<ST *>(m.dst);
    if (m.mask)
        tile2d<true, ST, false, REST>(m.g, m.p, m.mask, src, dst, m.status, w.bx, w.by, sm, m.rho_src, m.rho_dst);
    else
        tile2d<false, ST, false, REST>(m.g, m.p, m.mask, src, dst, m.status, w.bx, w.by, sm, m.rho_src, m.rho_dst);
}

}  // namespace lbmf2
