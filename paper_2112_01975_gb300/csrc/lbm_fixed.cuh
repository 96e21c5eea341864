// Sums of a node's populations in 64-bit fixed point.
//
// The moments of a node (density, momentum, second moments) are sums of its
// populations: 53 FP64 additions on D3Q27 for density and momentum alone,
// each as long as 76 integer issue slots, plus a conversion of the same
// length per population in 32- and 16-bit storage. Here the populations
// become 64-bit integers, so that their sums are exact; one integer-to-double
// conversion per moment rounds to 53 bits. With E the exponent of the node's
// largest population, unit and most that one population loses:
//   FP64     2^(E - 57)   half a unit (rounded to nearest)
//   FP32     2^(E - 57)   nothing down to 2^-34 of the largest, below that less
//                         than a unit (truncated)
//   shifted  2^(E - 56)   half a unit, and the 2^-60 or less of its source density's
//                         power of two that the product drops: 1.5 units in all
// which is less than the roundings of a sum in FP64 (2^-53 of the partial sum
// each). Against 80-bit arithmetic, density, u and U of FP64 D3Q27 and D2Q9
// drops are 1.1 (1 step) to 3 times (200 steps) closer than with FP64 sums;
// against exact sums of FP16 and BF16 D3Q27 populations the density is 2 and
// the momentum 1.5 to 2 times closer.
//
// Populations that are not positive normal numbers of a moderate range
// (negative ones, infinities and NaN among them), and in shifted storage those
// of which the largest is below 1/16 or so of a source's density, return
// false: the caller sums those nodes in FP64.
#pragma once

#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <stdint.h>

#include <type_traits>

namespace lbmk {

// The stored populations of a lattice: FP64, FP32, or 16-bit shifted values
// with the source densities of the buffer.
template <typename ST> struct Shifted {
    const ST *h;
    const float *rho_src;
};

// (w + h) rho in FP64 of float operands, as the stored value is defined; the
// conversions through the bit patterns (normal numbers and zero; others by
// the instruction).
__device__ __forceinline__ double widen(float v)
{
    const unsigned b = __float_as_uint(v), e = b & 0x7f800000u;
    if (e == 0u || e == 0x7f800000u) return (b << 1) == 0u ? __hiloint2double((int)b, 0) : (double)v;
    return __hiloint2double((int)((b & 0x80000000u) | (((b & 0x7fffffffu) >> 3) + 0x38000000u)), (int)(b << 29));
}

// s 2^e2 rounded to double (s != 0 needs 2^e2 s normal).
__device__ __forceinline__ double fixed_to_double(long long s, int e2)
{
    if (s == 0) return 0.0;
    const double d = (double)s;
    return __hiloint2double(__double2hiint(d) + e2 * (1 << 20), __double2loint(d));
}

// Mantissa v < 2^63 shifted right by k >= 1 places, rounded to nearest (a
// truncation would take 2^-58 of the density of a node on average, the same
// way in every step).
__device__ __forceinline__ long long shift_down(unsigned long long v, int k)
{
    return k > 63 ? 0 : (long long)((v + (1ull << (k - 1))) >> k);
}

// Node n = (x, y, z): q[i] 2^e2 = population i. skip: nothing is formed (the
// populations have been requested by then, beside what `skip` waits for).
template <int LAT>
__device__ __forceinline__ bool fixed_pops(const Geo &g, const double *f, unsigned n, int, int, int,
                                           long long *q, int &e2, bool skip)
{
    constexpr int Q = Lattice<LAT>::Q;
    double v[Q];
    unsigned top = 0;
#pragma unroll
    for (int i = 0; i < Q; ++i) v[i] = f[(size_t)i * g.N + n];
    if (skip) return true;
#pragma unroll
    for (int i = 0; i < Q; ++i) top = max(top, (unsigned)__double2hiint(v[i]));
    const int E = (int)(top >> 20);
    if (E < 128 || E >= 0x7ff) return false;   // (a sign bit makes E >= 2048)
    e2 = E - 1023 - 57;
#pragma unroll
    for (int i = 0; i < Q; ++i) {
        const unsigned hi = (unsigned)__double2hiint(v[i]);
        const unsigned long long m =
            ((unsigned long long)((hi & 0xfffffu) | 0x100000u) << 32 | (unsigned)__double2loint(v[i])) << 10;
        q[i] = shift_down(m, E + 5 - (int)(hi >> 20));
    }
    return true;
}

template <int LAT>
__device__ __forceinline__ bool fixed_pops(const Geo &g, const float *f, unsigned n, int, int, int,
                                           long long *q, int &e2, bool skip)
{
    constexpr int Q = Lattice<LAT>::Q;
    unsigned b[Q], top = 0;
#pragma unroll
    for (int i = 0; i < Q; ++i) b[i] = __float_as_uint(f[(size_t)i * g.N + n]);
    if (skip) return true;
#pragma unroll
    for (int i = 0; i < Q; ++i) top = max(top, b[i]);
    const int E = (int)(top >> 23);
    if (E < 72 || E >= 0xff) return false;
    e2 = E - 127 - 57;
#pragma unroll
    for (int i = 0; i < Q; ++i)   // exact down to 2^-34 of the largest
        q[i] = (long long)((unsigned long long)(((b[i] & 0x7fffffu) | 0x800000u) << 7) << 32 >>
                           min(E + 5 - (int)(b[i] >> 23), 63));
    return true;
}

// Shifted storage: (w_i + h_i) rho(r - c_i), the node's own density where the
// source is solid (density -1). w_i + h_i in units of 2^-62 (exact in FP16,
// whose values are multiples of 2^-24, and down to 2^-54 in BF16), times the
// 31-bit mantissa of the density. (Units of 2^-55 of the largest source density
// are as fast, but the density is off by 2.7e-16 rms, in FP64 sums 1.1e-16 and
// here 0.5e-16, and by up to 2e-13 beside a density 6.6e4 times as large.)
template <int LAT, typename ST>
__device__ __forceinline__ bool fixed_pops(const Geo &g, const Shifted<ST> &f, unsigned n, int x, int y, int z,
                                           long long *q, int &e2, bool skip)
{
    constexpr int D = Lattice<LAT>::D, Q = Lattice<LAT>::Q;
    constexpr double W1[3] = {1.0 / 6.0, 2.0 / 3.0, 1.0 / 6.0};
    const int X[3] = {wrapp(x + 1, g.nx), x, wrapm(x - 1, g.nx)};
    const int Y[3] = {wrapp(y + 1, g.ny), y, wrapm(y - 1, g.ny)};
    const int Z[3] = {D == 3 ? wrapp(z + 1, g.nz) : 0, z, D == 3 ? wrapm(z - 1, g.nz) : 0};
    float h[Q];
    unsigned s[Q], top = 0, htop = 0;
#pragma unroll
    for (int i = 0; i < Q; ++i) h[i] = lbmf::to_f(f.h[(size_t)i * g.N + n]);
#pragma unroll
    for (int i = 0; i < Q; ++i) {
        const unsigned src = entry(g, X[cxi(i) + 1], Y[cyi(i) + 1], Z[D == 3 ? czi(i) + 1 : 1]);
        s[i] = __float_as_uint(f.rho_src[src]);
    }
    if (skip) return true;
    const unsigned own = s[Q / 2];
    float largest = 0.0f;
#pragma unroll
    for (int i = 0; i < Q; ++i) {
        const float w = (float)(W1[cxi(i) + 1] * W1[cyi(i) + 1] * (D == 3 ? W1[czi(i) + 1] : 1.0));
        if (s[i] >> 31) s[i] = own;
        top = max(top, s[i]);
        htop = max(htop, __float_as_uint(h[i]) & 0x7fffffffu);
        largest = fmaxf(largest, fabsf((w + h[i]) * __uint_as_float(s[i])));
    }
    const int E = (int)(__float_as_uint(largest) >> 23), Es = (int)(top >> 23);
    // |h| < 1 keeps w + h and the product within 63 bits; Es >= 255: infinities,
    // NaN and negative densities
    if (E < 72 || Es >= 0xff || Es > E + 4 || htop >= 0x3f800000u) return false;
    e2 = E - 127 - 56;
#pragma unroll
    for (int i = 0; i < Q; ++i) {
        constexpr double unit = 4611686018427387904.0;   // 2^62
        long long wh = (long long)(W1[cxi(i) + 1] * W1[cyi(i) + 1] * (D == 3 ? W1[czi(i) + 1] : 1.0) * unit);
        const float a = h[i] * 1073741824.0f;   // 2^30
        if constexpr (std::is_same<ST, __half>::value) {
            wh += (long long)(int)a << 32;
        } else {
            const float ai = floorf(a);
            wh += ((long long)(int)ai << 32) + (unsigned)((a - ai) * 4294967296.0f);
        }
        const int m = (int)(((s[i] & 0x7fffffu) | 0x800000u) << 7);   // 2^30 <= m < 2^31
        const long long P = (long long)(int)(wh >> 32) * m + (long long)__umulhi((unsigned)wh, (unsigned)m);
        const int k = min(E + 4 - (int)(s[i] >> 23), 62);
        q[i] = (P + ((1ll << k) >> 1)) >> k;
    }
    return true;
}

// Population i in FP64.
template <int LAT>
__device__ __forceinline__ double pop_f64(const Geo &g, const double *f, int i, unsigned n, int, int, int)
{
    return f[(size_t)i * g.N + n];
}

template <int LAT>
__device__ __forceinline__ double pop_f64(const Geo &g, const float *f, int i, unsigned n, int, int, int)
{
    return widen(f[(size_t)i * g.N + n]);
}

template <int LAT, typename ST>
__device__ __forceinline__ double pop_f64(const Geo &g, const Shifted<ST> &f, int i, unsigned n, int x, int y, int z)
{
    constexpr int D = Lattice<LAT>::D;
    float src = f.rho_src[source_node(g, D, i, x, y, z)];
    if (src < 0.0f) src = f.rho_src[n];   // bounced by n itself
    return (weight_d(i, D) + widen(lbmf::to_f(f.h[(size_t)i * g.N + n]))) * widen(src);
}

// Density and momentum of node n; SECOND: also its second moments
// sum c_a c_b f (xx, yy[, zz], xy[, xz, yz]).
template <int LAT, bool SECOND, typename P>
__device__ __forceinline__ void node_sums(const Geo &g, const P &f, unsigned n, int x, int y, int z, double &rho,
                                          double *j, double *second = nullptr, bool skip = false)
{
    constexpr int D = Lattice<LAT>::D, Q = Lattice<LAT>::Q, NA = D == 3 ? 6 : 3;
    constexpr int CA[6] = {0, 1, D == 3 ? 2 : 0, 0, 0, 1};
    constexpr int CB[6] = {0, 1, D == 3 ? 2 : 1, 1, 2, 2};
    long long q[Q];
    int e2;
    if (fixed_pops<LAT>(g, f, n, x, y, z, q, e2, skip)) {
        if (skip) return;
        long long r = 0, jj[3] = {0, 0, 0}, ss[6] = {0, 0, 0, 0, 0, 0};
#pragma unroll
        for (int i = 0; i < Q; ++i) {
            const int c[3] = {cxi(i), cyi(i), D == 3 ? czi(i) : 0};
            r += q[i];
#pragma unroll
            for (int a = 0; a < D; ++a) jj[a] += c[a] * q[i];
            if (SECOND)
#pragma unroll
                for (int k = 0; k < NA; ++k) ss[k] += c[CA[k]] * c[CB[k]] * q[i];
        }
        rho = fixed_to_double(r, e2);
#pragma unroll
        for (int a = 0; a < D; ++a) j[a] = fixed_to_double(jj[a], e2);
        if (SECOND)
#pragma unroll
            for (int k = 0; k < NA; ++k) second[k] = fixed_to_double(ss[k], e2);
        return;
    }
    rho = j[0] = j[1] = j[2] = 0.0;
    if (SECOND)
#pragma unroll
        for (int k = 0; k < NA; ++k) second[k] = 0.0;
    for (int i = 0; i < Q; ++i) {
        const double fi = pop_f64<LAT>(g, f, i, n, x, y, z);
        const int c[3] = {cxi(i), cyi(i), D == 3 ? czi(i) : 0};
        rho += fi;
        for (int a = 0; a < D; ++a)
            if (c[a]) j[a] += c[a] > 0 ? fi : -fi;
        if (SECOND)
            for (int k = 0; k < NA; ++k) {
                const int cc = c[CA[k]] * c[CB[k]];
                if (cc) second[k] += cc > 0 ? fi : -fi;
            }
    }
}

}  // namespace lbmk
