// C ABI of the two-phase lattice Boltzmann library (declared in include/lbm.h).
#include <cuda.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>
#include <chrono>
#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <cstring>
#include <functional>
#include <map>
#include <new>
#include <thread>
#include <vector>

#include "lbm.h"
#include "lbm_fused_f32.cuh"
#include "lbm_fused_f32_r7.cuh"
#include "lbm_kernels.cuh"
#include "lbm_step2d.cuh"
#include "lbm_step_tma.h"

using lbmk::Geo;
using lbmk::Phys;
using lbmf::GeoF;
using lbmf::PhysF;

struct lbm_ctx {
    int lattice, D, Q;
    Geo geo;
    Phys phys;
    GeoF geof;     // FP32 fused step: 3D frame (D2Q9: ny = 1, nz = 2D y extent)
    PhysF physf;
    int tile_rows = 8;   // D3Q27 FP32 step: 32 x 8 (lbmf) or 32 x 7 (lbmf7) tiles
    int variant = LBM_FUSED_PLAIN;   // form of the fused step
    // D3Q27 reduced storage: the form and chunk follow the lattice
    // (choose_form) until the caller sets or tunes any of them
    bool auto_form = true;
    bool e64 = false;    // reduced storage: EOS, psi and force sums in FP64 (LBM_FLAG_EOS_F64)
    int storage, flags;
    double t_over_tc, tau;
    std::vector<uint8_t> mask_host, zsolid_host;
    bool any_solid = false;
    int sms = 148;         // SMs of the device
    int sweep_chunk = 16;  // planes per block of the D3Q27 force sweep (FP64 kernels); 0: direct sums
    int device;
    cudaStream_t own_stream = nullptr, stream = nullptr, cap_stream = nullptr;
    // device memory
    void *base = nullptr;
    bool owns_base = false;
    size_t bytes = 0;
    void *fv[2] = {nullptr, nullptr};   // population buffers (double, float or 16-bit)
    float *rs[2] = {nullptr, nullptr};  // shifted storage: source densities of buffer k
    double2 *rp = nullptr;
    double *u = nullptr, *gflux = nullptr /* D3Q27 reduced storage: the wall bits */, *partial = nullptr, *sums = nullptr;
    uint8_t *mask = nullptr;
    int *status = nullptr;
    int cur = 0;
    bool initialised = false, bad = false;
    cudaGraphExec_t graph = nullptr;        // two steps
    cudaGraphExec_t graph_long = nullptr;   // kLongSteps steps
    int64_t launches = 0;
    // status polling of long lbm_step calls: a pinned copy of the status word
    // and the event that marks its arrival
    int *poll_host = nullptr;
    cudaEvent_t poll_ev = nullptr;
    bool poll_pending = false;
    // D3Q27, FP32 with nx % 4 == 0 or shifted 16-bit with nx % 8 == 0: the
    // two population buffers as 4D tensors (x, y, z, i) for the TMA-staged
    // form (LBM_FUSED_WS_TMA)
    lbmf::BoxMaps tmaps[2];
    bool tmap_ready = false;
    // interpolated bounce-back: boundary nodes, their active links, wall distances
    int nb = 0;
    unsigned *bn = nullptr, *bmask = nullptr;
    double *bq = nullptr;
    char err[512] = {0};
};

namespace {

// Forget the captured steps (the form, chunk or kernels of a step change).
void drop_graphs(lbm_ctx *h)
{
    if (h->graph) cudaGraphExecDestroy(h->graph);
    if (h->graph_long) cudaGraphExecDestroy(h->graph_long);
    h->graph = h->graph_long = nullptr;
}

// Opt a kernel in to more than 48 KB of dynamic shared memory, once per
// device (the attribute belongs to the device the call runs on).
template <typename Kern>
void smem_opt_in(Kern kernel, int bytes, std::atomic<unsigned long long> &done)
{
    int dev = 0;
    cudaGetDevice(&dev);
    const unsigned long long bit = 1ull << (dev & 63);
    if (done.load() & bit) return;
    cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    done.fetch_or(bit);
}

constexpr size_t kAlign = 256;

size_t align_up(size_t v) { return (v + kAlign - 1) / kAlign * kAlign; }

struct Layout {
    size_t f0, f1, rs0, rs1, rp, u, g, mask, zs, partial, sums, status, total;
};

bool shifted(int storage) { return storage == LBM_F16S || storage == LBM_BF16S; }

size_t pop_bytes(int storage)
{
    return storage == LBM_F64 ? sizeof(double) : storage == LBM_F32 ? sizeof(float) : 2;
}

// planes: the fused step's march-axis extent (nz; ny for D2Q9).
Layout layout_for(int D, int Q, size_t N, int storage, size_t planes)
{
    Layout L;
    size_t o = 0;
    const size_t pb = pop_bytes(storage);
    // Either buffer, when it is the dead one between steps, also stages host
    // I/O: (1 + 2D) doubles per node (more than 9 floats on D2Q9).
    const size_t fb = pb * Q * N > sizeof(double) * (1 + 2 * D) * N ? pb * Q * N
                                                                   : sizeof(double) * (1 + 2 * D) * N;
    L.f0 = o; o = align_up(o + fb);
    L.f1 = o; o = align_up(o + fb);
    const size_t rsb = (storage == LBM_F16S || storage == LBM_BF16S) ? sizeof(float) * N : 0;
    L.rs0 = o; o = align_up(o + rsb);
    L.rs1 = o; o = align_up(o + rsb);
    L.rp = o; o = align_up(o + sizeof(double2) * N);
    L.u = o; o = align_up(o + sizeof(double) * D * N);
    L.g = o; o = align_up(o + sizeof(double) * D * N);
    L.mask = o; o = align_up(o + N);
    L.zs = o; o = align_up(o + planes);   // per-plane solid flags
    L.partial = o; o = align_up(o + sizeof(double) * 4 * lbmk::RED_BLOCKS);
    L.sums = o; o = align_up(o + sizeof(double) * 4);
    L.status = o; o = align_up(o + sizeof(int) * 4);
    L.total = o;
    return L;
}

// Row alignment of the TMA-staged forms: rows of 16 bytes, 4 FP32 or 8 16-bit
// populations.
int tma_nx_multiple(int storage) { return storage == LBM_F32 ? 4 : shifted(storage) ? 8 : 0; }

// Entries per row of the library's own fields: nx, in D3Q27 reduced storage
// rounded up so that every row starts on 16 bytes and lattices of any width
// have a TMA-staged form (unless entry numbers then leave 32 bits).
int row_pitch(int lattice, int nx, int ny, int nz, int storage)
{
    const int mult = tma_nx_multiple(storage);
    if (lattice != LBM_D3Q27 || !mult) return nx;
    const int px = (nx + mult - 1) / mult * mult;
    return (double)px * ny * nz * 27.0 <= 4.2e9 ? px : nx;
}

bool valid_shape(int lattice, int nx, int ny, int nz)
{
    if (lattice != LBM_D2Q9 && lattice != LBM_D3Q27) return false;
    if (nx < 5 || ny < 5) return false;
    if (lattice == LBM_D2Q9 && nz != 1) return false;
    if (lattice == LBM_D3Q27 && nz < 5) return false;
    // 32-bit node indices in the kernels
    if ((double)nx * ny * nz * 27.0 > 4.0e9) return false;
    return true;
}

int fail(lbm_ctx *h, int code, const char *fmt, ...)
{
    if (h) {
        va_list ap;
        va_start(ap, fmt);
        vsnprintf(h->err, sizeof(h->err), fmt, ap);
        va_end(ap);
    }
    return code;
}

#define CU(h, call)                                                                      \
    do {                                                                                 \
        cudaError_t e_ = (call);                                                         \
        if (e_ != cudaSuccess)                                                           \
            return fail((h), LBM_ECUDA, "%s: %s (%s:%d)", #call, cudaGetErrorString(e_), \
                        __FILE__, __LINE__);                                             \
    } while (0)

double eos_rtc(int eos, double a, double b)
{
    switch (eos) {
    case LBM_EOS_VDW: return 8.0 * a / (27.0 * b);
    case LBM_EOS_PR: return (0.0778 / 0.45724) * a / b;
    case LBM_EOS_RKS: return (0.08664 / 0.42748) * a / b;
    case LBM_EOS_CS: return (0.18727 / 0.4963) * a / b;
    case LBM_EOS_SC1: return -4.0;          // critical coupling G_c (Appendix G)
    case LBM_EOS_SC2: return -std::exp(2.0);
    }
    return NAN;
}

// The EOS's temperature parameter at T/Tc: R T for the cubic equations, the
// coupling G = G_c / (T/Tc) for Shan-Chen (kept in the RT slot).
double eos_temperature(int eos, double a, double b, double tr)
{
    const double c = eos_rtc(eos, a, b);
    return eos >= LBM_EOS_SC1 ? c / tr : tr * c;
}

double eos_alpha(int eos, double acentric, double tr)
{
    double m;
    if (eos == LBM_EOS_PR) m = 0.37464 + 1.54226 * acentric - 0.26992 * acentric * acentric;
    else if (eos == LBM_EOS_RKS) m = 0.480 + 1.574 * acentric - 0.176 * acentric * acentric;
    else return 1.0;
    const double s = 1.0 + m * (1.0 - std::sqrt(tr));
    return s * s;
}

// P - rho/3 in FP64 on the host (the EOS of the solid nodes' virtual density
// for the FP64-EOS form of the reduced-precision steps).
double excess_pressure_host(int eos, double a, double b, double RT, double aalpha, double r)
{
    const double br = b * r, rt = r * RT;
    double P;
    switch (eos) {
    case LBM_EOS_VDW: P = rt / (1.0 - br) - a * r * r; break;
    case LBM_EOS_PR: P = (rt * (1.0 + br * (2.0 - br)) - aalpha * r * r * (1.0 - br)) /
                         ((1.0 - br) * (1.0 + br * (2.0 - br))); break;
    case LBM_EOS_RKS: P = (rt * (1.0 + br) - aalpha * r * r * (1.0 - br)) / ((1.0 - br) * (1.0 + br)); break;
    case LBM_EOS_SC1: { const double q = 1.0 - std::exp(-r); P = r / 3.0 + RT / 6.0 * q * q; break; }
    case LBM_EOS_SC2: { const double q = std::exp(-1.0 / r); P = r / 3.0 + RT / 6.0 * q * q; break; }
    default: {
        const double e = 0.25 * br, om = 1.0 - e;
        P = rt * (1.0 + e + e * e - e * e * e) / (om * om * om) - a * r * r;
    }
    }
    return P - r / 3.0;
}

// Makespan of n_full blocks of cost cf, then n_tail of cost ct <= cf, each
// taken by the first of `slots` that is free.
double makespan(long long n_full, double cf, long long n_tail, double ct, long long slots)
{
    const long long k = n_full / slots, r = n_full % slots;
    const double lo = k * cf, hi = r ? lo + cf : lo;   // slots - r end at lo, r at hi
    if (n_tail == 0) return hi;
    double a = hi, b = hi + (n_tail / slots + 1) * ct;   // n_tail fit before b
    for (int it = 0; it < 40; ++it) {
        const double t = 0.5 * (a + b);
        const long long fit = (slots - r) * (long long)((t - lo) / ct + 1e-9) + r * (long long)((t - hi) / ct + 1e-9);
        if (fit >= n_tail) b = t;
        else               a = t;
    }
    return b;
}

dim3 node_block(const Geo &g)
{
    int bx = g.nx >= 128 ? 128 : ((g.nx + 31) / 32) * 32;
    return dim3(bx, 1, 1);
}

dim3 node_grid(const Geo &g)
{
    dim3 b = node_block(g);
    return dim3((g.nx + b.x - 1) / b.x, g.ny, g.nz);
}

void make_tensor_maps(lbm_ctx *h);

// The chunk of planes per block that ends the step first: a block of c planes
// marches through c + 4. `resident` blocks share an SM; two together take
// 1.31 times as long per plane as one alone (measured: 5.4 against 4.1 us,
// shifted storage at 128^3). The last, shorter chunk of each column fills the
// SMs that the whole ones leave. Measured, TMA-staged forms, the choice here
// against others: FP32 64^3 24.1 us (chunk 7; 8: 25.1), 128^3 104 (56; 64:
// 114, 16: 135), 160^3 187 (108; 54: 191), 256^3 723 (223; 64: 762);
// FP16-shifted 128^3 166 (29; 32: 179), 256^3 1093 (223; 64: 1174). Furthest
// from the best of a scan: 97x61x75 FP32 53.3 (50.5).
int best_chunk(const GeoF &g, int rows, int sms, int resident)
{
    const long long tiles = (long long)((g.nx + 31) / 32) * ((g.ny + rows - 1) / rows);
    int best = 1;
    double cost = 1e300;
    for (int c = 1; c <= g.nz; ++c) {
        const long long full = tiles * (g.nz / c), tail = g.nz % c ? tiles : 0;
        const double cf = c + 4.5, ct = g.nz % c + 4.5;
        double t = makespan(full, cf, tail, ct, sms);
        if (resident == 2 && full + tail > sms) t = 1.31 * makespan(full, cf, tail, ct, 2ll * sms);
        if (t <= cost) {
            cost = t;
            best = c;
        }
    }
    return best;
}

constexpr int kDefaultChunk3 = 16;

// Form and chunk of a D3Q27 handle of reduced storage that the caller has
// left open: with tensor maps the TMA-staged form of the storage, the
// fastest of the forms at every size measured, each at its best chunk (FP32
// 64^3 24.1 us against 34.8 for the Tensor Memory form, 128^3 104 against 154,
// 256^3 723 against 1127; FP16-shifted 128^3 166 against 190, 256^3 1093
// against 1363). The Tensor Memory form without tensor maps, where a column of the
// halo lies in no box (box_pos; 153 x 145 x 131 FP32: 206 us against 222) and,
// in shifted storage, where the tiles hang over the lattice by more than a
// tenth: there it reads less, while the TMA-staged form's nine copies cost the
// same (98 x 61 x 75: 66 us against 75, 45 x 37 x 60: 31 against 38; 150^3, which
// fills its tiles: 329 against 285). With the FP64 EOS the plain one. The fixed default before, plain at chunk 16: FP32 64^3 62, 128^3 184,
// 256^3 1208; FP16-shifted 258, 1649.
void choose_form(lbm_ctx *h)
{
    if (!h->auto_form || h->lattice != LBM_D3Q27 || h->storage == LBM_F64) return;
    const Geo &g = h->geo;
    const bool stray = g.nx % tma_nx_multiple(h->storage) == 1;   // a halo column in no box
    const double use = (double)g.nx * g.ny / (((g.nx + 31) / 32 * 32.0) * ((g.ny + 7) / 8 * 8.0));
    if (h->e64) h->variant = LBM_FUSED_PLAIN;
    else if (!h->tmap_ready || stray || (shifted(h->storage) && use < 0.9)) h->variant = LBM_FUSED_TMEM;
    else h->variant = h->storage == LBM_F32 ? LBM_FUSED_WS_TMA : LBM_FUSED_TM_TMA;
    h->geof.chunk = best_chunk(h->geof, 8, h->sms, h->variant == LBM_FUSED_WS_TMA ? 1 : 2);
}

// The caller sets one of form, tile and chunk: the others start from the
// plain form's.
void leave_auto_form(lbm_ctx *h)
{
    if (!h->auto_form) return;
    h->auto_form = false;
    if (h->lattice != LBM_D3Q27 || h->storage == LBM_F64) return;
    h->variant = LBM_FUSED_PLAIN;
    h->geof.chunk = kDefaultChunk3;
    drop_graphs(h);  // the captured graph holds the chosen form
}

// The wall bits of the planes within one of a solid node (4 bytes per node of
// those planes and 8 per plane of the lattice), in the region of rho u_a^3 (24
// bytes per node), which reduced storage does not use.
int make_wall_bits(lbm_ctx *h)
{
    if (h->lattice != LBM_D3Q27 || h->storage == LBM_F64 || !h->any_solid) return LBM_OK;
    const Geo &g = h->geo;
    std::vector<int> table(g.nz, -1), planes;   // number of each z's plane; z of each plane
    for (int z = 0; z < g.nz; ++z)
        if (h->zsolid_host[(z + g.nz - 1) % g.nz] || h->zsolid_host[z] || h->zsolid_host[(z + 1) % g.nz]) {
            table[z] = (int)planes.size();
            planes.push_back(z);
        }
    const size_t head = align_up(sizeof(int) * 2 * g.nz);
    if (head + sizeof(unsigned) * planes.size() * g.px * g.ny > sizeof(double) * 3 * g.N)
        return fail(h, LBM_EINVAL, "no room for the wall bits");   // not for any lattice of 5 or more nodes a side
    int *const walls = reinterpret_cast<int *>(h->gflux);
    unsigned *const w = reinterpret_cast<unsigned *>(reinterpret_cast<char *>(walls) + head);
    CU(h, cudaMemcpyAsync(walls, table.data(), sizeof(int) * g.nz, cudaMemcpyHostToDevice, h->stream));
    CU(h, cudaMemcpyAsync(walls + g.nz, planes.data(), sizeof(int) * planes.size(), cudaMemcpyHostToDevice,
                          h->stream));
    dim3 gr = node_grid(g);
    gr.z = (unsigned)planes.size();
    lbmk::k_wall_bits<<<gr, node_block(g), 0, h->stream>>>(g, h->mask, walls + g.nz, w);
    CU(h, cudaGetLastError());
    CU(h, cudaStreamSynchronize(h->stream));   // before the host vectors go
    h->geof.wplane = walls;
    h->geof.walls = w;
    return LBM_OK;
}

// Lay out the device memory (allocated here unless bound) and fill what stays
// as it is: masks, wall bits, tensor maps.
int lay_out(lbm_ctx *h)
{
    Layout L = layout_for(h->D, h->Q, h->geo.N, h->storage, h->geof.nz);
    if (!h->base) {
        void *p = nullptr;
        cudaError_t e = cudaMalloc(&p, L.total);
        if (e != cudaSuccess) {
            cudaGetLastError();
            return fail(h, LBM_ENOMEM, "cudaMalloc(%zu) failed: %s", L.total, cudaGetErrorString(e));
        }
        h->base = p;
        h->owns_base = true;
        h->bytes = L.total;
    }
    char *b = static_cast<char *>(h->base);
    h->fv[0] = b + L.f0;
    h->fv[1] = b + L.f1;
    if (shifted(h->storage)) {
        h->rs[0] = reinterpret_cast<float *>(b + L.rs0);
        h->rs[1] = reinterpret_cast<float *>(b + L.rs1);
    }
    h->rp = reinterpret_cast<double2 *>(b + L.rp);
    h->u = reinterpret_cast<double *>(b + L.u);
    h->gflux = reinterpret_cast<double *>(b + L.g);
    h->mask = reinterpret_cast<uint8_t *>(b + L.mask);
    h->geof.zsolid = reinterpret_cast<const uint8_t *>(b + L.zs);
    h->partial = reinterpret_cast<double *>(b + L.partial);
    h->sums = reinterpret_cast<double *>(b + L.sums);
    h->status = reinterpret_cast<int *>(b + L.status);
    // the mask with the rows' padding, if any, marked solid
    std::vector<uint8_t> padded;
    if (h->geo.px != h->geo.nx) {
        padded.assign(h->geo.N, 1);
        for (size_t r = 0; r < (size_t)h->geo.ny * h->geo.nz; ++r)
            memcpy(&padded[r * h->geo.px], &h->mask_host[r * h->geo.nx], h->geo.nx);
    }
    CU(h, cudaMemcpyAsync(h->mask, padded.empty() ? h->mask_host.data() : padded.data(), h->geo.N,
                          cudaMemcpyHostToDevice, h->stream));
    {   // planes of the fused step's march axis (z; the 2D y axis for D2Q9) that hold a solid
        const size_t plane = (size_t)h->geof.nx * h->geof.ny;
        h->zsolid_host.assign(h->geof.nz, 0);
        for (int z = 0; z < h->geof.nz; ++z) {
            uint8_t any = 0;
            for (size_t n = 0; n < plane; ++n) any |= h->mask_host[z * plane + n];
            h->zsolid_host[z] = any != 0;
        }
        CU(h, cudaMemcpyAsync(const_cast<uint8_t *>(h->geof.zsolid), h->zsolid_host.data(), h->geof.nz,
                              cudaMemcpyHostToDevice, h->stream));
    }
    CU(h, cudaMemsetAsync(h->status, 0, sizeof(int) * 4, h->stream));
    const int rc = make_wall_bits(h);
    if (rc != LBM_OK) return rc;
    CU(h, cudaStreamSynchronize(h->stream));
    make_tensor_maps(h);
    if (h->variant == LBM_FUSED_WS_TMA && !h->tmap_ready) h->variant = LBM_FUSED_WS_TMEM;
    if (h->variant == LBM_FUSED_TM_TMA && !h->tmap_ready) h->variant = LBM_FUSED_TMEM;
    choose_form(h);
    return LBM_OK;
}

// The device memory laid out, on the handle's first use of it. After a failure
// nothing is (fv[0] null): the next call starts over.
int ensure_memory(lbm_ctx *h)
{
    if (h->fv[0]) return LBM_OK;
    int rc;
    try {
        rc = lay_out(h);
    } catch (const std::bad_alloc &) {
        rc = fail(h, LBM_ENOMEM, "no host memory to lay out the lattice");
    }
    if (rc == LBM_OK) return rc;
    cudaStreamSynchronize(h->stream);   // copies from host memory that is about to go
    cudaGetLastError();
    h->fv[0] = nullptr;
    h->geof.wplane = nullptr;
    h->geof.walls = nullptr;
    if (h->owns_base) {
        cudaFree(h->base);
        h->base = nullptr;
        h->owns_base = false;
        h->bytes = 0;
    }
    return rc;
}

bool has_solid(const lbm_ctx *h) { return h->any_solid; }

// The two population buffers of a D3Q27 FP32 or shifted-storage handle as
// 4D tensors (x, y, z, i) of the stored type, each with the five box shapes
// of the TMA-staged forms (32 x 8, 32 x 2, W x 8, W x 2 and the one-copy
// (32 + 2 W) x 12 nodes of one plane, all 27 populations; W = 16 bytes of
// the type). Needs rows that start on 16 bytes (row_pitch) and the CUDA driver's tensor-map
// encoder, found through the runtime's entry-point query; leaves tmap_ready
// false when either is missing.
void make_tensor_maps(lbm_ctx *h)
{
    h->tmap_ready = false;
    const int mult = tma_nx_multiple(h->storage);
    if (h->lattice != LBM_D3Q27 || !mult || h->geo.px % mult || !h->fv[0]) return;
    using Encode = CUresult (*)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                const cuuint64_t *, const cuuint32_t *, const cuuint32_t *,
                                CUtensorMapInterleave, CUtensorMapSwizzle, CUtensorMapL2promotion,
                                CUtensorMapFloatOOBfill);
    void *fn = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &q) !=
            cudaSuccess ||
        q != cudaDriverEntryPointSuccess || !fn) {
        cudaGetLastError();
        return;
    }
    const Geo &g = h->geo;
    const cuuint64_t es = pop_bytes(h->storage);
    const CUtensorMapDataType dt = h->storage == LBM_F32    ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32
                                   : h->storage == LBM_F16S ? CU_TENSOR_MAP_DATA_TYPE_FLOAT16
                                                            : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16;
    const cuuint32_t w = (cuuint32_t)(16 / es);
    const cuuint64_t dims[4] = {(cuuint64_t)g.nx, (cuuint64_t)g.ny, (cuuint64_t)g.nz, 27};
    const cuuint64_t strides[3] = {(cuuint64_t)g.px * es, (cuuint64_t)g.px * g.ny * es, (cuuint64_t)g.N * es};
    const cuuint32_t estr[4] = {1, 1, 1, 1};
    for (int k = 0; k < 2; ++k) {
        CUtensorMap *m[5] = {&h->tmaps[k].mc, &h->tmaps[k].tc, &h->tmaps[k].ml, &h->tmaps[k].tl,
                             &h->tmaps[k].wide};
        const cuuint32_t wx[5] = {32, 32, w, w, 32 + 2 * w}, wy[5] = {8, 2, 8, 2, 12};
        for (int j = 0; j < 5; ++j) {
            const cuuint32_t box[4] = {wx[j], wy[j], 1, 27};
            if (reinterpret_cast<Encode>(fn)(m[j], dt, 4, h->fv[k], dims, strides, box, estr,
                                              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                                              CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                                              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
                return;
        }
    }
    h->tmap_ready = true;
}

// Whether the two kernels of the FP64 step overlap at their ends: D2Q9
// lattices of so few 32 x 2 tiles that both kernels' blocks have an SM each.
bool overlap64(const lbm_ctx *h)
{
    const Geo &g = h->geo;
    return h->lattice == LBM_D2Q9 && 2ll * ((g.nx + 31) / 32) * ((g.ny + 1) / 2) <= h->sms;
}

// The force sweep over the lattice (lbm_kernels.cuh) with the given body.
template <int LAT, typename Body>
void launch_sweep(lbm_ctx *h, cudaStream_t s, const Body &body)
{
    const Geo &g = h->geo;
    const int tx = (g.nx + lbmk::SWX - 1) / lbmk::SWX;
    if constexpr (LAT == 1) {
        const int chunk = h->sweep_chunk;
        if (chunk == 0) {
            lbmk::k_force_direct3<Body><<<node_grid(g), node_block(g), 0, s>>>(g, h->phys, h->rp, body);
            return;
        }
        const dim3 grid(tx, (g.ny + lbmk::SWY - 1) / lbmk::SWY, (g.nz + chunk - 1) / chunk);
        static std::atomic<unsigned long long> done{0};   // devices already opted in
        const int bytes = (int)sizeof(lbmk::SweepSmem3);
        smem_opt_in(lbmk::k_force_sweep3<Body>, bytes, done);
        lbmk::k_force_sweep3<Body><<<grid, lbmk::SWX * lbmk::SWY, bytes, s>>>(g, h->phys, h->rp, chunk, body);
    } else if (tx * ((g.ny + 7) / 8) < h->sms) {
        lbmpdl::launch_step(overlap64(h), lbmk::k_force_sweep2<2, 4, Body>, dim3(tx, (g.ny + 1) / 2), 128, 0, s, g, h->phys, h->rp,
                            body);
    } else {
        lbmpdl::launch_step(false, lbmk::k_force_sweep2<8, 8, Body>, dim3(tx, (g.ny + 7) / 8), 256, 0, s, g, h->phys, h->rp,
                            body);
    }
}

// Planes per block of the D3Q27 force sweep, or 0 for the direct sums of small
// lattices: a block's 8 warps share their SM's FP64 pipe (19 cycles an
// instruction), so the SM with the most blocks sets the time; a block of c
// planes also sums 4 more (46 of about 210 operations per node). Directly it
// is about 290 operations per node, but every SM has its share (32^3: 20 us
// against 33 at the best chunk, 44^3 66 against 70, 48^3 74 against 70).
int sweep_chunk(const Geo &g, int sms)
{
    const long long tiles = (long long)((g.nx + lbmk::SWX - 1) / lbmk::SWX) *
                            ((g.ny + lbmk::SWY - 1) / lbmk::SWY);
    // c planes cost 200 c + 256 (the proportion that picks the chunk of the scans);
    // two blocks share an SM at half speed each. The last, shorter chunk of each
    // column fills in (128^3: chunk 29 701 us, 14 705, 18 711, 32 768; 97x61x75:
    // 8 219, 9 242, 6 259; 160^3: 54 1272, 40 1442; 96^3: 24 316, 12 312).
    int best = 1;
    double cost = 1e300;
    for (int c = 1; c <= g.nz; ++c) {
        const long long full = tiles * (g.nz / c), tail = g.nz % c ? tiles : 0;
        const double cf = c * 200.0 + 256.0, ct = g.nz % c * 200.0 + 256.0;
        const double t = full + tail <= sms ? cf : 2.0 * makespan(full, cf, tail, ct, 2ll * sms);
        if (t < cost) {
            cost = t;
            best = c;
        }
    }
    const long long warps = (long long)g.ny * g.nz * ((g.nx + 31) / 32);
    const double direct = std::max(19.0 * ((warps + sms - 1) / sms), 64.0) * 290.0;
    return direct < 19.0 * 8.0 * cost ? 0 : best;
}

double *f64(lbm_ctx *h, int k) { return static_cast<double *>(h->fv[k]); }
float *f32(lbm_ctx *h, int k) { return static_cast<float *>(h->fv[k]); }

dim3 fused_grid(const GeoF &g, int rows = lbmf::LatF<1>::TY)
{
    using L = lbmf::LatF<1>;
    return dim3((g.nx + L::TX - 1) / L::TX, (g.ny + rows - 1) / rows, (g.nz + g.chunk - 1) / g.chunk);
}

// The same parameters as the 7-row build's types (one source, one layout).
template <typename T, typename U>
T as_layout(const U &u)
{
    static_assert(sizeof(T) == sizeof(U), "same source, same layout");
    T t;
    memcpy(&t, &u, sizeof t);
    return t;
}

template <bool MASK>
void launch_fused_r7(lbm_ctx *h, cudaStream_t s, const float *src, float *dst)
{
    using L = lbmf7::LatF<1>;
    if (h->variant == LBM_FUSED_TMEM) {
        static std::atomic<unsigned long long> done{0};   // devices already opted in
        const int bytes = (int)sizeof(lbmf7::SharedF<1>);
        smem_opt_in(lbmf7::k_step_f32_tm<1, MASK>, bytes, done);
        lbmf7::k_step_f32_tm<1, MASK><<<fused_grid(h->geof, L::TY), L::TX * L::TY, bytes, s>>>(
            as_layout<lbmf7::GeoF>(h->geof), as_layout<lbmf7::PhysF>(h->physf), h->mask, src, dst,
            h->status);
        return;
    }
    if (h->variant == LBM_FUSED_WARP_SPECIALISED) {
        static std::atomic<unsigned long long> done{0};   // devices already opted in
        const int bytes = (int)sizeof(lbmf7::SharedWS<1>);
        smem_opt_in(lbmf7::k_step_f32_ws<1, MASK>, bytes, done);
        lbmf7::k_step_f32_ws<1, MASK><<<fused_grid(h->geof, L::TY), 2 * L::TX * L::TY, bytes, s>>>(
            as_layout<lbmf7::GeoF>(h->geof), as_layout<lbmf7::PhysF>(h->physf), h->mask, src, dst,
            h->status);
        return;
    }
    static std::atomic<unsigned long long> done{0};   // devices already opted in
    const int bytes = (int)sizeof(lbmf7::SharedF<1>);
    smem_opt_in(lbmf7::k_step_f32<1, MASK>, bytes, done);
    lbmf7::k_step_f32<1, MASK><<<fused_grid(h->geof, L::TY), L::TX * L::TY, bytes, s>>>(
        as_layout<lbmf7::GeoF>(h->geof), as_layout<lbmf7::PhysF>(h->physf), h->mask, src, dst,
        h->status);
}

template <bool MASK>
void launch_fused_tm(lbm_ctx *h, cudaStream_t s, const float *src, float *dst)
{
    static std::atomic<unsigned long long> done{0};   // devices already opted in
    using L = lbmf::LatF<1>;
    const int bytes = (int)sizeof(lbmf::SharedF<1>);
    smem_opt_in(lbmf::k_step_f32_tm<1, MASK>, bytes, done);
    lbmf::k_step_f32_tm<1, MASK><<<fused_grid(h->geof), L::TX * L::TY, bytes, s>>>(
        h->geof, h->physf, h->mask, src, dst, h->status);
}

template <bool MASK>
void launch_fused_wstm(lbm_ctx *h, cudaStream_t s, const float *src, float *dst)
{
    static std::atomic<unsigned long long> done{0};   // devices already opted in
    using L = lbmf::LatF<1>;
    const int bytes = (int)sizeof(lbmf::SharedWS<1>);
    smem_opt_in(lbmf::k_step_f32_wstm<1, MASK>, bytes, done);
    lbmf::k_step_f32_wstm<1, MASK><<<fused_grid(h->geof), 2 * L::TX * L::TY, bytes, s>>>(
        h->geof, h->physf, h->mask, src, dst, h->status);
}

template <bool MASK>
void launch_fused_ws(lbm_ctx *h, cudaStream_t s, const float *src, float *dst)
{
    static std::atomic<unsigned long long> done{0};   // devices already opted in
    using L = lbmf::LatF<1>;
    const int bytes = (int)sizeof(lbmf::SharedWS<1>);
    smem_opt_in(lbmf::k_step_f32_ws<1, MASK>, bytes, done);
    lbmf::k_step_f32_ws<1, MASK><<<fused_grid(h->geof), 2 * L::TX * L::TY, bytes, s>>>(
        h->geof, h->physf, h->mask, src, dst, h->status);
}

template <bool MASK>
void launch_fused_e64(lbm_ctx *h, cudaStream_t s, const float *src, float *dst)
{
    static std::atomic<unsigned long long> done{0};   // devices already opted in
    using L = lbmf::LatF<1>;
    const int bytes = (int)sizeof(lbmf::SharedF<1>);
    smem_opt_in(lbmf::k_step_f32<1, MASK, true>, bytes, done);
    lbmf::k_step_f32<1, MASK, true><<<fused_grid(h->geof), L::TX * L::TY, bytes, s>>>(
        h->geof, h->physf, h->mask, src, dst, h->status);
}

// Whether `blocks` blocks of `threads` threads of a kernel leave its successor
// room for less than a block per SM, going by the blocks of it that an SM holds
// at once (its registers decide: 4 to 6 of the D2Q9 kernels' instantiations;
// asked once, the library is built for one architecture). D2Q9 with and without
// overlap, us a step: FP32, time 1 (6 an SM), 960x200 (4.9 blocks an SM) 5.14 /
// 5.00, 928x224 (5.3) 5.26 / 5.66; other times (5 an SM), 768x200 (3.9) 4.73 /
// 4.62, 704x240 (4.3) 4.76 / 5.14; FP16 960x200 6.67 / 6.04, 928x224 6.70 / 7.19
// and 768x200 5.65 / 5.27, 704x240 5.68 / 6.18.
template <typename Kern>
bool leaves_no_room(Kern kernel, long long blocks, int threads, int sms, std::atomic<int> &known)
{
    int n = known.load();
    if (n == 0) {
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kernel, threads, 0) != cudaSuccess || n < 1) {
            cudaGetLastError();
            return false;
        }
        known.store(n);
    }
    return blocks > (n - 1ll) * sms;
}

// The D2Q9 step of a reduced storage from population buffer k: one kernel,
// whatever form, chunk or tile the handle names (lbm_step2d.cuh).
template <typename ST, bool MASK, bool E64, bool REST>
void launch_2d_r(lbm_ctx *h, cudaStream_t s, int k)
{
    const GeoF &g = h->geof;
    const dim3 grid((g.nx + lbmf2::TX - 1) / lbmf2::TX, (g.nz + lbmf2::TY - 1) / lbmf2::TY);
    static std::atomic<int> known{0};
    const long long blocks = (long long)grid.x * grid.y;
    const bool overlap = lbmpdl::side_by_side(blocks, h->sms) ||
                         leaves_no_room(lbmf2::k_step2d<MASK, ST, E64, REST>, blocks, lbmf2::NT, h->sms, known);
    lbmpdl::launch_step(overlap, lbmf2::k_step2d<MASK, ST, E64, REST>, grid, lbmf2::NT, 0, s, g, h->physf, h->mask,
                        static_cast<const ST *>(h->fv[k]), static_cast<ST *>(h->fv[k ^ 1]), h->rs[k], h->rs[k ^ 1],
                        h->status);
}

template <typename ST, bool MASK, bool E64>
void launch_2d_m(lbm_ctx *h, cudaStream_t s, int k)
{
    if (lbmf::at_rest(h->physf)) launch_2d_r<ST, MASK, E64, true>(h, s, k);
    else                         launch_2d_r<ST, MASK, E64, false>(h, s, k);
}

template <typename ST>
void launch_2d(lbm_ctx *h, cudaStream_t s, int k)
{
    if (has_solid(h)) {
        if (h->e64) launch_2d_m<ST, true, true>(h, s, k);
        else        launch_2d_m<ST, true, false>(h, s, k);
    } else {
        if (h->e64) launch_2d_m<ST, false, true>(h, s, k);
        else        launch_2d_m<ST, false, false>(h, s, k);
    }
}

template <bool MASK>
void launch_fused_rest(lbm_ctx *h, cudaStream_t s, const float *src, float *dst)
{
    static std::atomic<unsigned long long> done{0};   // devices already opted in
    using L = lbmf::LatF<1>;
    const int bytes = (int)sizeof(lbmf::SharedF<1>);
    smem_opt_in(lbmf::k_step_f32<1, MASK, false, true>, bytes, done);
    lbmf::k_step_f32<1, MASK, false, true><<<fused_grid(h->geof), L::TX * L::TY, bytes, s>>>(
        h->geof, h->physf, h->mask, src, dst, h->status);
}

// One D3Q27 step of FP32 storage.
void launch_fused(lbm_ctx *h, cudaStream_t s, const float *src, float *dst)
{
    if (h->e64) {   // the plain 32 x 8 form only
        if (has_solid(h)) launch_fused_e64<true>(h, s, src, dst);
        else              launch_fused_e64<false>(h, s, src, dst);
        return;
    }
    if (h->tile_rows == 7) {
        if (has_solid(h)) launch_fused_r7<true>(h, s, src, dst);
        else              launch_fused_r7<false>(h, s, src, dst);
        return;
    }
    if (h->variant == LBM_FUSED_WARP_SPECIALISED) {
        if (has_solid(h)) launch_fused_ws<true>(h, s, src, dst);
        else              launch_fused_ws<false>(h, s, src, dst);
        return;
    }
    if (lbmf::at_rest(h->physf) && (h->variant == LBM_FUSED_TMEM || h->variant == LBM_FUSED_PLAIN)) {
        // nothing to keep between the phases: the two forms are one
        if (has_solid(h)) launch_fused_rest<true>(h, s, src, dst);
        else              launch_fused_rest<false>(h, s, src, dst);
        return;
    }
    if (h->variant == LBM_FUSED_TMEM) {
        if (has_solid(h)) launch_fused_tm<true>(h, s, src, dst);
        else              launch_fused_tm<false>(h, s, src, dst);
        return;
    }
    if (h->variant == LBM_FUSED_WS_TMA) {   // D3Q27, 32 x 8 tiles, tensor maps made
        lbmtma::launch(h->geof, h->physf, h->mask, h->tmaps[src == h->fv[0] ? 0 : 1], src, dst, h->status,
                       has_solid(h), s);
        return;
    }
    if (h->variant == LBM_FUSED_WS_TMEM) {   // D3Q27, 32 x 8 tiles
        if (has_solid(h)) launch_fused_wstm<true>(h, s, src, dst);
        else              launch_fused_wstm<false>(h, s, src, dst);
        return;
    }
    static std::atomic<unsigned long long> done_m{0}, done_f{0};   // devices already opted in
    using L = lbmf::LatF<1>;
    const int bytes = (int)sizeof(lbmf::SharedF<1>);
    const dim3 gr = fused_grid(h->geof);
    if (has_solid(h)) {
        smem_opt_in(lbmf::k_step_f32<1, true>, bytes, done_m);
        lbmf::k_step_f32<1, true><<<gr, L::TX * L::TY, bytes, s>>>(h->geof, h->physf, h->mask, src,
                                                                    dst, h->status);
    } else {
        smem_opt_in(lbmf::k_step_f32<1, false>, bytes, done_f);
        lbmf::k_step_f32<1, false><<<gr, L::TX * L::TY, bytes, s>>>(h->geof, h->physf, h->mask, src,
                                                                     dst, h->status);
    }
}

// One step of FP32 storage from population buffer k.
void launch_f32(lbm_ctx *h, cudaStream_t s, int k)
{
    if (h->lattice == LBM_D2Q9) launch_2d<float>(h, s, k);
    else                        launch_fused(h, s, f32(h, k), f32(h, k ^ 1));
}

template <typename ST, bool E64, bool MASK, bool REST = false>
void launch_shifted_e(lbm_ctx *h, cudaStream_t s, int k)
{
    static std::atomic<unsigned long long> done{0};   // devices already opted in
    const int bytes = (int)sizeof(lbmf::SharedS<1>);
    smem_opt_in(lbmf::k_step_shifted<1, ST, E64, MASK, REST>, bytes, done);
    using L = lbmf::LatF<1>;
    lbmf::k_step_shifted<1, ST, E64, MASK, REST><<<fused_grid(h->geof), L::TX * L::TY, bytes, s>>>(
        h->geof, h->physf, h->mask, static_cast<const ST *>(h->fv[k]), static_cast<ST *>(h->fv[k ^ 1]),
        h->rs[k], h->rs[k ^ 1], h->status);
}

template <typename ST, bool MASK>
void launch_shifted_tm(lbm_ctx *h, cudaStream_t s, int k)
{
    static std::atomic<unsigned long long> done{0};   // devices already opted in
    const int bytes = (int)sizeof(lbmf::SharedS<1>);
    smem_opt_in(lbmf::k_step_shifted_tm<1, ST, MASK>, bytes, done);
    using L = lbmf::LatF<1>;
    lbmf::k_step_shifted_tm<1, ST, MASK><<<fused_grid(h->geof), L::TX * L::TY, bytes, s>>>(
        h->geof, h->physf, h->mask, static_cast<const ST *>(h->fv[k]), static_cast<ST *>(h->fv[k ^ 1]),
        h->rs[k], h->rs[k ^ 1], h->status);
}

template <typename ST, bool MASK>
void launch_shifted_wstm(lbm_ctx *h, cudaStream_t s, int k)
{
    static std::atomic<unsigned long long> done{0};   // devices already opted in
    const int bytes = (int)sizeof(lbmf::SharedSWS<1>);
    smem_opt_in(lbmf::k_step_shifted_wstm<1, ST, MASK>, bytes, done);
    using L = lbmf::LatF<1>;
    lbmf::k_step_shifted_wstm<1, ST, MASK><<<fused_grid(h->geof), 2 * L::TX * L::TY, bytes, s>>>(
        h->geof, h->physf, h->mask, static_cast<const ST *>(h->fv[k]), static_cast<ST *>(h->fv[k ^ 1]),
        h->rs[k], h->rs[k ^ 1], h->status);
}

template <typename ST, bool MASK>
void launch_shifted_m(lbm_ctx *h, cudaStream_t s, int k)
{
    if (!h->e64 && h->variant == LBM_FUSED_WS_TMA) {   // tensor maps made
        lbmtma::launch_shifted(h->geof, h->physf, h->mask, h->tmaps[k], static_cast<const ST *>(h->fv[k]),
                               static_cast<ST *>(h->fv[k ^ 1]), h->rs[k], h->rs[k ^ 1], h->status, MASK, s);
        return;
    }
    if (!h->e64 && h->variant == LBM_FUSED_TM_TMA) {   // tensor maps made
        lbmtma::launch_shifted_tm(h->geof, h->physf, h->mask, h->tmaps[k], static_cast<const ST *>(h->fv[k]),
                                  static_cast<ST *>(h->fv[k ^ 1]), h->rs[k], h->rs[k ^ 1], h->status, MASK,
                                  s);
        return;
    }
    if (h->e64) launch_shifted_e<ST, true, MASK>(h, s, k);
    else if (lbmf::at_rest(h->physf) && (h->variant == LBM_FUSED_TMEM || h->variant == LBM_FUSED_PLAIN))
        launch_shifted_e<ST, false, MASK, true>(h, s, k);   // nothing to keep between the phases
    else if (h->variant == LBM_FUSED_TMEM) launch_shifted_tm<ST, MASK>(h, s, k);
    else if (h->variant == LBM_FUSED_WS_TMEM) launch_shifted_wstm<ST, MASK>(h, s, k);
    else launch_shifted_e<ST, false, MASK>(h, s, k);
}

template <typename ST>
void launch_shifted_t(lbm_ctx *h, cudaStream_t s, int k)
{
    if (has_solid(h)) launch_shifted_m<ST, true>(h, s, k);
    else              launch_shifted_m<ST, false>(h, s, k);
}

// One step of shifted storage from population buffer k.
void launch_shifted(lbm_ctx *h, cudaStream_t s, int k)
{
    const bool half = h->storage == LBM_F16S;
    if (h->lattice == LBM_D2Q9) {
        if (half) launch_2d<__half>(h, s, k);
        else      launch_2d<__nv_bfloat16>(h, s, k);
    } else {
        if (half) launch_shifted_t<__half>(h, s, k);
        else      launch_shifted_t<__nv_bfloat16>(h, s, k);
    }
}

// The collision of the FP64 step: the force sweep with its body, without the
// terms in 1 - omega where the relaxation time is 1 everywhere.
template <int LAT>
void launch_collide64(lbm_ctx *h, cudaStream_t s, const double *src, double *dst)
{
    if (h->phys.omega == 1.0 && !h->phys.var_visc)
        launch_sweep<LAT>(h, s, lbmk::CollideBody<LAT, true>{h->mask, src, dst, h->rp, h->u, h->gflux});
    else
        launch_sweep<LAT>(h, s, lbmk::CollideBody<LAT, false>{h->mask, src, dst, h->rp, h->u, h->gflux});
}

// One time step; returns the number of kernels launched (0 on error).
template <int LAT>
int launch_step(lbm_ctx *h, cudaStream_t s, int *nk)
{
    if (shifted(h->storage)) {
        launch_shifted(h, s, h->cur);
        *nk = 1;
    } else if (h->storage == LBM_F32) {
        launch_f32(h, s, h->cur);
        *nk = 1;
    } else {
        const dim3 gr = node_grid(h->geo), bl = node_block(h->geo);
        const double *src = f64(h, h->cur);
        double *dst = f64(h, h->cur ^ 1);
        lbmpdl::launch_step(overlap64(h), lbmk::k_macro<LAT, true, const double *>, gr, bl, 0, s, h->geo, h->phys, h->mask, src, h->rp,
                            h->u, h->gflux, h->status);
        launch_collide64<LAT>(h, s, src, dst);
        *nk = 2;
    }
    if (h->nb > 0) {   // interpolated bounce-back on the new state
        const int th = 128, bl = (h->nb + th - 1) / th;
        if (h->storage == LBM_F32)
            lbmk::k_interp_bounce_back<LAT, float><<<bl, th, 0, s>>>(h->geo, h->bn, h->bmask, h->bq,
                                                                     h->nb, f32(h, h->cur ^ 1));
        else
            lbmk::k_interp_bounce_back<LAT, double><<<bl, th, 0, s>>>(h->geo, h->bn, h->bmask, h->bq,
                                                                      h->nb, f64(h, h->cur ^ 1));
        *nk += 1;
    }
    CU(h, cudaGetLastError());
    h->cur ^= 1;
    return LBM_OK;
}

int step_plain(lbm_ctx *h, cudaStream_t s, int *nk_out = nullptr)
{
    int nk = 0;
    int rc = h->lattice == LBM_D2Q9 ? launch_step<0>(h, s, &nk) : launch_step<1>(h, s, &nk);
    if (rc == LBM_OK) h->launches += nk;
    if (nk_out) *nk_out = nk;
    return rc;
}

int kernels_per_step(const lbm_ctx *h) { return (h->storage == LBM_F64 ? 2 : 1) + (h->nb > 0); }

// Shifted storage I/O goes through a temporary FP64 copy of the populations.
struct TempF64 {
    double *p = nullptr;
    ~TempF64() { if (p) cudaFree(p); }
};

template <int LAT>
int decode_to(lbm_ctx *h, int k, double *out)
{
    const dim3 gr = node_grid(h->geo), bl = node_block(h->geo);
    if (h->storage == LBM_F16S)
        lbmk::k_decode_shifted<LAT, __half><<<gr, bl, 0, h->stream>>>(
            h->geo, static_cast<const __half *>(h->fv[k]), h->rs[k], out);
    else
        lbmk::k_decode_shifted<LAT, __nv_bfloat16><<<gr, bl, 0, h->stream>>>(
            h->geo, static_cast<const __nv_bfloat16 *>(h->fv[k]), h->rs[k], out);
    CU(h, cudaGetLastError());
    h->launches += 1;
    return LBM_OK;
}

template <int LAT, bool INIT = false>
int encode_from(lbm_ctx *h, const Geo &gf, const double *f)   // gf: the layout of f
{
    const dim3 gr = node_grid(h->geo), bl = node_block(h->geo);
    lbmk::k_density<LAT, INIT><<<gr, bl, 0, h->stream>>>(h->geo, gf, h->mask, f, h->rs[0], h->rs[1]);
    if (h->storage == LBM_F16S)
        lbmk::k_encode_shifted<LAT, __half><<<gr, bl, 0, h->stream>>>(
            h->geo, gf, f, h->rs[0], static_cast<__half *>(h->fv[0]));
    else
        lbmk::k_encode_shifted<LAT, __nv_bfloat16><<<gr, bl, 0, h->stream>>>(
            h->geo, gf, f, h->rs[0], static_cast<__nv_bfloat16 *>(h->fv[0]));
    CU(h, cudaGetLastError());
    h->launches += 2;
    h->cur = 0;
    return LBM_OK;
}

// Populations from rows of pa entries of type A to rows of pb of B.
template <typename A, typename B>
void convert_pops(lbm_ctx *h, int pa, int pb, const A *in, B *out)
{
    const Geo &g = h->geo;
    lbmk::k_convert<<<1024, 256, 0, h->stream>>>((unsigned)(h->Q * g.ny * g.nz), (unsigned)g.nx, (unsigned)pa,
                                                 (unsigned)pb, in, out);
}

int temp_alloc(lbm_ctx *h, TempF64 &t)
{
    const size_t bytes = sizeof(double) * (size_t)h->Q * h->geo.N;
    if (cudaMalloc(&t.p, bytes) != cudaSuccess) {
        cudaGetLastError();
        t.p = nullptr;
        return fail(h, LBM_ENOMEM, "no room for the FP64 copy of shifted populations");
    }
    return LBM_OK;
}

// An even number of steps (state buffer 0 -> 1 -> 0 ...) captured once on the
// library's own stream; replayed on the handle's stream.
int ensure_graph(lbm_ctx *h, cudaGraphExec_t &graph, int steps)
{
    if (graph) return LBM_OK;
    if (!h->cap_stream) CU(h, cudaStreamCreateWithFlags(&h->cap_stream, cudaStreamNonBlocking));
    cudaGraph_t g = nullptr;
    CU(h, cudaStreamBeginCapture(h->cap_stream, cudaStreamCaptureModeThreadLocal));
    const int saved = h->cur;
    int rc = LBM_OK;
    for (int k = 0; k < steps && rc == LBM_OK; ++k) rc = step_plain(h, h->cap_stream);
    h->launches -= steps * kernels_per_step(h);  // captured, not launched
    h->cur = saved;
    cudaError_t e = cudaStreamEndCapture(h->cap_stream, &g);
    if (rc != LBM_OK) {
        if (g) cudaGraphDestroy(g);
        return rc;
    }
    if (e != cudaSuccess) return fail(h, LBM_ECUDA, "graph capture: %s", cudaGetErrorString(e));
    e = cudaGraphInstantiate(&graph, g, 0);
    cudaGraphDestroy(g);
    if (e != cudaSuccess) {
        graph = nullptr;
        return fail(h, LBM_ECUDA, "graph instantiate: %s", cudaGetErrorString(e));
    }
    return LBM_OK;
}

int read_status(lbm_ctx *h)
{
    int st = 0;
    CU(h, cudaMemcpyAsync(&st, h->status, sizeof(int), cudaMemcpyDeviceToHost, h->stream));
    CU(h, cudaStreamSynchronize(h->stream));
    if (st) {
        h->bad = true;
        if (st & 8)
            return fail(h, LBM_ECUDA, "the TMA-staged step found its shared memory not 128-byte aligned");
        if (st & 2)
            return fail(h, LBM_ETIMEOUT, "a wait between the fused step's thread groups timed out");
        return fail(h, LBM_ENONFINITE, "a density became non-finite or non-positive");
    }
    return LBM_OK;
}

int check_ready(lbm_ctx *h)
{
    if (!h) return LBM_EINVAL;
    if (!h->initialised) return fail(h, LBM_ESTATE, "handle not initialised (call lbm_init)");
    return LBM_OK;
}

// fn(populations of buffer k) with their storage's type.
template <typename Fn>
void with_pops(const lbm_ctx *h, int k, const Fn &fn)
{
    switch (h->storage) {
    case LBM_F64: fn(static_cast<const double *>(h->fv[k])); break;
    case LBM_F32: fn(static_cast<const float *>(h->fv[k])); break;
    case LBM_F16S: fn(lbmk::Shifted<__half>{static_cast<const __half *>(h->fv[k]), h->rs[k]}); break;
    default: fn(lbmk::Shifted<__nv_bfloat16>{static_cast<const __nv_bfloat16 *>(h->fv[k]), h->rs[k]});
    }
}

// Side fields (rho, s psi) and u of the current state.
template <int LAT>
void launch_macro(lbm_ctx *h)
{
    with_pops(h, h->cur, [&](auto f) {
        lbmk::k_macro<LAT, false><<<node_grid(h->geo), node_block(h->geo), 0, h->stream>>>(
            h->geo, h->phys, h->mask, f, h->rp, h->u, nullptr, h->status);
    });
}

template <int LAT>
int launch_macro_and_out(lbm_ctx *h, double *rho, double *u, double *U)
{
    launch_macro<LAT>(h);
    if (U)
        launch_sweep<LAT>(h, h->stream, lbmk::MomentsBody<LAT>{h->mask, h->rp, h->u, rho, u, U});
    else
        lbmk::k_moments_out<LAT><<<node_grid(h->geo), node_block(h->geo), 0, h->stream>>>(
            h->geo, h->phys, h->mask, h->rp, h->u, rho, u);
    CU(h, cudaGetLastError());
    h->launches += 2;
    return LBM_OK;
}

template <int LAT>
int launch_pressure(lbm_ctx *h, double *out)
{
    launch_macro<LAT>(h);
    with_pops(h, h->cur, [&](auto f) {
        lbmk::k_pressure_tensor<LAT><<<node_grid(h->geo), node_block(h->geo), 0, h->stream>>>(
            h->geo, h->phys, h->mask, f, h->rp, out);
    });
    CU(h, cudaGetLastError());
    h->launches += 2;
    return LBM_OK;
}

template <int LAT>
int launch_init(lbm_ctx *h, const double *rho0, const double *u0)
{
    const dim3 gr = node_grid(h->geo), bl = node_block(h->geo);
    // side fields first: the initial force needs rho and s psi of every node
    lbmk::k_fill_solid<LAT><<<gr, bl, 0, h->stream>>>(h->geo, h->phys, h->mask, h->rp, h->u,
                                                      h->storage == LBM_F64 ? h->gflux : nullptr);
    lbmk::k_init_density<LAT><<<gr, bl, 0, h->stream>>>(h->geo, h->phys, h->mask, rho0, h->rp);
    h->launches += 3;
    if (shifted(h->storage)) {
        TempF64 t;
        int rc = temp_alloc(h, t);
        if (rc) return rc;
        lbmk::k_init<LAT><<<gr, bl, 0, h->stream>>>(h->geo, h->phys, h->mask, h->rp, u0, t.p);
        rc = encode_from<LAT, true>(h, h->geo, t.p);
        if (rc) return rc;
        CU(h, cudaGetLastError());
        CU(h, cudaStreamSynchronize(h->stream));   // before the temporary is freed
        return LBM_OK;
    }
    if (h->storage == LBM_F32)
        lbmk::k_init<LAT, float><<<gr, bl, 0, h->stream>>>(h->geo, h->phys, h->mask, h->rp, u0, f32(h, h->cur));
    else
        lbmk::k_init<LAT><<<gr, bl, 0, h->stream>>>(h->geo, h->phys, h->mask, h->rp, u0, f64(h, h->cur));
    CU(h, cudaGetLastError());
    return LBM_OK;
}

template <int LAT>
int launch_fill_solid(lbm_ctx *h)
{
    const dim3 gr = node_grid(h->geo), bl = node_block(h->geo);
    lbmk::k_fill_solid<LAT><<<gr, bl, 0, h->stream>>>(h->geo, h->phys, h->mask, h->rp, h->u,
                                                      h->storage == LBM_F64 ? h->gflux : nullptr);
    CU(h, cudaGetLastError());
    h->launches += 1;
    return LBM_OK;
}

template <int LAT>
int launch_reduce(lbm_ctx *h)
{
    with_pops(h, h->cur, [&](auto f) {
        lbmk::k_reduce_partial<LAT><<<lbmk::RED_BLOCKS, lbmk::RED_THREADS, 0, h->stream>>>(h->geo, h->mask, f,
                                                                                           h->partial);
    });
    lbmk::k_reduce_final<<<1, lbmk::RED_BLOCKS, 0, h->stream>>>(h->partial, h->sums);
    CU(h, cudaGetLastError());
    h->launches += 2;
    return LBM_OK;
}

// Between two graph replays the GPU idles for 1 to 3 us, as long as a step of a
// small lattice (64^2 FP32: 4.3 us a step with graphs of two steps, 2.6 with
// 16, and 32 gained 3 % on that). Sequences of at least twice that on lattices whose step is
// short (under about 50 us) replay graphs of kLongSteps steps.
constexpr int kLongSteps = 16;
constexpr unsigned kLongNodes = 1u << 20;

// Status polling of long step sequences: every kPollSteps steps the status word is copied to pinned host memory behind an
// event; before the next copy is queued the previous one is awaited, so the
// host runs at most one polling interval ahead of the device and a diverged
// lattice stops within two intervals.
constexpr int64_t kPollSteps = 64;

int ensure_poll(lbm_ctx *h)
{
    if (h->poll_host) return LBM_OK;
    CU(h, cudaHostAlloc(reinterpret_cast<void **>(&h->poll_host), sizeof(int), cudaHostAllocDefault));
    *h->poll_host = 0;
    CU(h, cudaEventCreateWithFlags(&h->poll_ev, cudaEventDisableTiming));
    return LBM_OK;
}

// Wait for the last queued status copy and act on it; queue the next one.
int poll_status(lbm_ctx *h)
{
    if (h->poll_pending) {
        CU(h, cudaEventSynchronize(h->poll_ev));
        h->poll_pending = false;
        if (*h->poll_host) {
            h->bad = true;
            return fail(h, LBM_ENONFINITE, "a density became non-finite or non-positive");
        }
    }
    CU(h, cudaMemcpyAsync(h->poll_host, h->status, sizeof(int), cudaMemcpyDeviceToHost, h->stream));
    CU(h, cudaEventRecord(h->poll_ev, h->stream));
    h->poll_pending = true;
    return LBM_OK;
}

}  // namespace

extern "C" {

int lbm_default_params(int eos, lbm_params *p)
{
    if (!p) return LBM_EINVAL;
    switch (eos) {
    case LBM_EOS_VDW: p->a = 9.0 / 49.0; p->b = 2.0 / 21.0; break;
    case LBM_EOS_PR:
    case LBM_EOS_RKS: p->a = 2.0 / 49.0; p->b = 2.0 / 21.0; break;
    case LBM_EOS_CS: p->a = 1.0; p->b = 4.0; break;
    case LBM_EOS_SC1:
    case LBM_EOS_SC2: p->a = 1.0; p->b = 1.0; break;   // not used by Shan-Chen
    default: return LBM_EINVAL;
    }
    p->acentric = 0.344;
    p->rho_w = 1.0;
    p->g[0] = p->g[1] = p->g[2] = 0.0;
    p->tau_v = 0.0;
    p->visc_rho[0] = 0.0;
    p->visc_rho[1] = 1.0;
    p->storage = LBM_F64;
    p->flags = 0;
    return LBM_OK;
}

size_t lbm_required_bytes(int lattice, int nx, int ny, int nz, int storage)
{
    if (!valid_shape(lattice, nx, ny, nz) || storage < LBM_F64 || storage > LBM_BF16S) return 0;
    const int D = lattice == LBM_D2Q9 ? 2 : 3, Q = lattice == LBM_D2Q9 ? 9 : 27;
    return layout_for(D, Q, (size_t)row_pitch(lattice, nx, ny, nz, storage) * ny * nz, storage,
                      lattice == LBM_D2Q9 ? ny : nz).total;
}

int lbm_create(lbm_handle *out, int lattice, int nx, int ny, int nz, int eos, double t_over_tc,
               double kappa, double tau, const uint8_t *solid_mask, const lbm_params *p)
{
    if (!out) return LBM_EINVAL;
    *out = nullptr;
    if (!valid_shape(lattice, nx, ny, nz)) return LBM_EINVAL;
    if (eos < LBM_EOS_VDW || eos > LBM_EOS_SC2) return LBM_EINVAL;
    if (!(t_over_tc > 0.0 && t_over_tc < 1.0) || !(kappa >= 0.0) || !(tau > 0.5)) return LBM_EINVAL;
    lbm_params prm;
    if (p) prm = *p;
    else lbm_default_params(eos, &prm);
    if (prm.storage < LBM_F64 || prm.storage > LBM_BF16S) return LBM_EINVAL;
    if (!(prm.a > 0.0) || !(prm.b > 0.0) || !(prm.rho_w > 0.0)) return LBM_EINVAL;
    for (int a = 0; a < 3; ++a)
        if (!std::isfinite(prm.g[a])) return LBM_EINVAL;
    if (prm.tau_v != 0.0 && !(prm.tau_v > 0.5 && prm.visc_rho[0] > 0.0 &&
                              prm.visc_rho[1] > prm.visc_rho[0] && std::isfinite(prm.tau_v)))
        return LBM_EINVAL;
    lbm_ctx *h = new (std::nothrow) lbm_ctx();
    if (!h) return LBM_ENOMEM;
    h->lattice = lattice;
    h->D = lattice == LBM_D2Q9 ? 2 : 3;
    h->Q = lattice == LBM_D2Q9 ? 9 : 27;
    h->geo.nx = nx; h->geo.ny = ny; h->geo.nz = nz;
    h->geo.M = (unsigned)((size_t)nx * ny * nz);
    h->geo.px = row_pitch(lattice, nx, ny, nz, prm.storage);
    h->geo.N = (unsigned)((size_t)h->geo.px * ny * nz);
    h->storage = prm.storage;
    h->flags = prm.flags;
    h->t_over_tc = t_over_tc;
    h->tau = tau;
    Phys &ph = h->phys;
    ph.eos = eos;
    ph.a = prm.a;
    ph.b = prm.b;
    ph.RT = eos_temperature(eos, prm.a, prm.b, t_over_tc);
    ph.alpha = eos_alpha(eos, prm.acentric, t_over_tc);
    ph.aalpha = ph.a * ph.alpha;
    ph.kappa = kappa;
    ph.kr = kappa * (lattice == LBM_D2Q9 ? -1.0 / 6.0 : -1.0 / 36.0);
    ph.omega = 1.0 / tau;
    ph.phi_pref = (prm.flags & LBM_FLAG_PHI_OFF) ? 0.0 : -(1.0 - 0.5 * ph.omega);
    ph.rho_w = prm.rho_w;
    for (int a = 0; a < 3; ++a) ph.g[a] = (a < (lattice == LBM_D2Q9 ? 2 : 3)) ? prm.g[a] : 0.0;
    ph.body = ph.g[0] != 0.0 || ph.g[1] != 0.0 || ph.g[2] != 0.0;
    ph.var_visc = prm.tau_v > 0.0 ? 1 : 0;
    ph.nu_l = (tau - 0.5) / 3.0;
    ph.nu_v = ph.var_visc ? (prm.tau_v - 0.5) / 3.0 : ph.nu_l;
    ph.visc_rv = prm.visc_rho[0];
    ph.visc_rl = prm.visc_rho[1];
    ph.phi_sign = (prm.flags & LBM_FLAG_PHI_OFF) ? 0.0 : -1.0;
    // FP32 fused step: D2Q9 runs in the 3D frame with one y row.
    h->geof.nx = nx;
    h->geof.ny = lattice == LBM_D2Q9 ? 1 : ny;
    h->geof.nz = lattice == LBM_D2Q9 ? ny : nz;
    h->geof.N = h->geo.N;
    h->geof.px = h->geo.px;
    h->geof.chunk = lattice == LBM_D2Q9 ? 64 : kDefaultChunk3;
    PhysF &pf = h->physf;
    pf.eos = eos;
    pf.a = (float)ph.a;
    pf.b = (float)ph.b;
    pf.RT = (float)ph.RT;
    pf.aalpha = (float)(ph.a * ph.alpha);
    pf.kappa = (float)kappa;
    pf.omega = (float)ph.omega;
    pf.omw = (float)(1.0 - ph.omega);
    pf.phi_pref = (float)ph.phi_pref;
    pf.rho_w = (float)prm.rho_w;
    pf.g[0] = (float)ph.g[0];
    pf.g[1] = lattice == LBM_D2Q9 ? 0.0f : (float)ph.g[1];
    pf.g[2] = lattice == LBM_D2Q9 ? (float)ph.g[1] : (float)ph.g[2];
    pf.var_visc = ph.var_visc;
    pf.nu_l = (float)ph.nu_l;
    pf.nu_v = (float)ph.nu_v;
    pf.visc_rl = (float)ph.visc_rl;
    pf.inv_drho = ph.var_visc ? (float)(1.0 / (ph.visc_rl - ph.visc_rv)) : 0.0f;
    pf.phi_sign = (float)ph.phi_sign;
    pf.da = ph.a;
    pf.db = ph.b;
    pf.dRT = ph.RT;
    pf.daalpha = ph.a * ph.alpha;
    pf.dkappa = kappa;
    h->e64 = (prm.flags & LBM_FLAG_EOS_F64) != 0;
    {
        // P - P0 of the solid density, in FP32
        const float r = pf.rho_w;
        float P;
        const float rep = r * pf.RT / (1.0f - pf.b * r);
        switch (eos) {
        case LBM_EOS_VDW: P = rep - pf.a * r * r; break;
        case LBM_EOS_PR: P = rep - pf.aalpha * r * r / (1.0f + 2.0f * pf.b * r - pf.b * pf.b * r * r); break;
        case LBM_EOS_RKS: P = rep - pf.aalpha * r * r / (1.0f + pf.b * r); break;
        case LBM_EOS_SC1: {
            const float q = 1.0f - std::exp(-r);
            P = r * (1.0f / 3.0f) + pf.RT / 6.0f * q * q;
            break;
        }
        case LBM_EOS_SC2: {
            const float q = std::exp(-1.0f / r);
            P = r * (1.0f / 3.0f) + pf.RT / 6.0f * q * q;
            break;
        }
        default: {
            const float e = 0.25f * pf.b * r, om = 1.0f - e;
            P = r * pf.RT * (1.0f + e + e * e - e * e * e) / (om * om * om) - pf.a * r * r;
        }
        }
        const float d = P - r * (1.0f / 3.0f);
        pf.spsi_w = d;
        if (h->e64) pf.spsi_w = (float)excess_pressure_host(eos, ph.a, ph.b, ph.RT, ph.a * ph.alpha, prm.rho_w);
    }
    h->mask_host.assign(h->geo.M, 0);
    if (solid_mask)
        for (size_t n = 0; n < h->geo.M; ++n) {
            h->mask_host[n] = solid_mask[n] ? 1 : 0;
            h->any_solid = h->any_solid || solid_mask[n];
        }
    if (cudaGetDevice(&h->device) != cudaSuccess ||
        cudaStreamCreateWithFlags(&h->own_stream, cudaStreamNonBlocking) != cudaSuccess) {
        cudaGetLastError();
        delete h;
        return LBM_ECUDA;
    }
    h->stream = h->own_stream;
    if (cudaDeviceGetAttribute(&h->sms, cudaDevAttrMultiProcessorCount, h->device) != cudaSuccess)
        cudaGetLastError();   // the default stands
    h->sweep_chunk = sweep_chunk(h->geo, h->sms);
    *out = h;
    return LBM_OK;
}

int lbm_bind_device_memory(lbm_handle h, void *dev, size_t bytes)
{
    if (!h || !dev) return LBM_EINVAL;
    if (h->fv[0]) return fail(h, LBM_ESTATE, "device memory already in use");
    if (reinterpret_cast<uintptr_t>(dev) % kAlign) return fail(h, LBM_EINVAL, "memory not 256-byte aligned");
    const size_t need = layout_for(h->D, h->Q, h->geo.N, h->storage, h->geof.nz).total;
    if (bytes < need) return fail(h, LBM_ENOMEM, "bound memory %zu < required %zu", bytes, need);
    h->base = dev;
    h->owns_base = false;
    h->bytes = bytes;
    return LBM_OK;
}

int lbm_set_stream(lbm_handle h, void *stream)
{
    if (!h) return LBM_EINVAL;
    h->stream = stream ? static_cast<cudaStream_t>(stream) : h->own_stream;
    return LBM_OK;
}

int lbm_init(lbm_handle h, const double *rho0, const double *u0, int on_device)
{
    if (!h || !rho0) return LBM_EINVAL;
    int rc = ensure_memory(h);
    if (rc) return rc;
    const size_t N = h->geo.M;
    h->cur = 0;
    const double *r = rho0, *v = u0;
    if (!on_device) {
        // stage through the second population buffer, dead between steps
        double *st = static_cast<double *>(h->fv[1]);
        CU(h, cudaMemcpyAsync(st, rho0, sizeof(double) * N, cudaMemcpyHostToDevice, h->stream));
        r = st;
        if (u0) {
            CU(h, cudaMemcpyAsync(st + N, u0, sizeof(double) * h->D * N, cudaMemcpyHostToDevice,
                                  h->stream));
            v = st + N;
        }
    }
    CU(h, cudaMemsetAsync(h->status, 0, sizeof(int), h->stream));
    rc = h->lattice == LBM_D2Q9 ? launch_init<0>(h, r, v) : launch_init<1>(h, r, v);
    if (rc) return rc;
    CU(h, cudaStreamSynchronize(h->stream));
    h->initialised = true;
    h->bad = false;
    return LBM_OK;
}

int lbm_step(lbm_handle h, int64_t n)
{
    int rc = check_ready(h);
    if (rc) return rc;
    if (n < 0) return fail(h, LBM_EINVAL, "negative step count");
    if (h->bad) return fail(h, LBM_ESTATE, "state holds a non-finite density; re-initialise");
    if (n >= 4) {
        if (h->cur != 0) {
            if ((rc = step_plain(h, h->stream))) return rc;
            --n;
        }
        const bool longer = n >= 2 * kLongSteps && h->geo.M <= kLongNodes;
        if ((rc = ensure_graph(h, h->graph, 2))) return rc;
        if (longer && (rc = ensure_graph(h, h->graph_long, kLongSteps))) return rc;
        if (n / 2 * 2 > kPollSteps && (rc = ensure_poll(h))) return rc;
        h->poll_pending = false;
        for (int64_t unpolled = 0; n >= 2;) {
            const int k = longer && n >= kLongSteps ? kLongSteps : 2;
            if (unpolled >= kPollSteps) {
                if ((rc = poll_status(h))) return rc;
                unpolled = 0;
            }
            CU(h, cudaGraphLaunch(k == 2 ? h->graph : h->graph_long, h->stream));
            h->launches += k * kernels_per_step(h);
            unpolled += k;
            n -= k;
        }
    }
    for (int64_t k = 0; k < n; ++k)
        if ((rc = step_plain(h, h->stream))) return rc;
    return LBM_OK;
}

int lbm_moments(lbm_handle h, double *rho, double *u, double *U, int on_device)
{
    int rc = check_ready(h);
    if (rc) return rc;
    const size_t N = h->geo.M, D = h->D;
    double *dr = rho, *du = u, *dU = U;
    if (!on_device) {
        double *st = static_cast<double *>(h->fv[h->cur ^ 1]);  // dead between steps
        dr = rho ? st : nullptr;
        du = u ? st + N : nullptr;
        dU = U ? st + N + D * N : nullptr;
    }
    rc = h->lattice == LBM_D2Q9 ? launch_macro_and_out<0>(h, dr, du, dU)
                                : launch_macro_and_out<1>(h, dr, du, dU);
    if (rc) return rc;
    if (!on_device) {
        if (rho) CU(h, cudaMemcpyAsync(rho, dr, sizeof(double) * N, cudaMemcpyDeviceToHost, h->stream));
        if (u) CU(h, cudaMemcpyAsync(u, du, sizeof(double) * D * N, cudaMemcpyDeviceToHost, h->stream));
        if (U) CU(h, cudaMemcpyAsync(U, dU, sizeof(double) * D * N, cudaMemcpyDeviceToHost, h->stream));
    }
    return read_status(h);
}

int lbm_set_wall_distances(lbm_handle h, const double *q)
{
    if (!h) return LBM_EINVAL;
    const size_t N = h->geo.M;
    const int Q = h->Q, D = h->D;
    const Geo &g = h->geo;
    std::vector<unsigned> bn, bm;
    std::vector<double> bq;
    if (q) {
        for (size_t n = 0; n < N; ++n) {
            if (h->mask_host[n]) continue;
            const int x = n % g.nx, y = (n / g.nx) % g.ny, z = n / ((size_t)g.nx * g.ny);
            unsigned m = 0;
            double qq[27] = {0.0};
            for (int i = 0; i < Q; ++i) {
                const int c[3] = {i % 3 - 1, (i / 3) % 3 - 1, D == 3 ? i / 9 - 1 : 0};
                const size_t nd = (size_t)((x + c[0] + g.nx) % g.nx) +
                                  (size_t)g.nx * (((y + c[1] + g.ny) % g.ny) +
                                                  (size_t)g.ny * ((z + c[2] + g.nz) % g.nz));
                const size_t nm = (size_t)((x - c[0] + g.nx) % g.nx) +
                                  (size_t)g.nx * (((y - c[1] + g.ny) % g.ny) +
                                                  (size_t)g.ny * ((z - c[2] + g.nz) % g.nz));
                const double qi = q[(size_t)i * N + n];
                if (!h->mask_host[nd] || !(qi > 0.0)) continue;
                if (!(qi <= 1.0)) return fail(h, LBM_EINVAL, "wall distance q > 1 at node %zu", n);
                if (h->mask_host[nm]) continue;   // no fluid node behind: stays halfway
                m |= 1u << i;
                qq[i] = qi;
            }
            if (m) {
                bn.push_back((unsigned)n);
                bm.push_back(m);
                bq.insert(bq.end(), qq, qq + Q);
            }
        }
    }
    if (h->stream) CU(h, cudaStreamSynchronize(h->stream));
    if (h->bn) cudaFree(h->bn);
    if (h->bmask) cudaFree(h->bmask);
    if (h->bq) cudaFree(h->bq);
    h->bn = h->bmask = nullptr;
    h->bq = nullptr;
    h->nb = 0;
    drop_graphs(h);  // the captured steps change
    if (bn.empty()) return LBM_OK;
    CU(h, cudaMalloc(&h->bn, sizeof(unsigned) * bn.size()));
    CU(h, cudaMalloc(&h->bmask, sizeof(unsigned) * bm.size()));
    CU(h, cudaMalloc(&h->bq, sizeof(double) * bq.size()));
    CU(h, cudaMemcpy(h->bn, bn.data(), sizeof(unsigned) * bn.size(), cudaMemcpyHostToDevice));
    CU(h, cudaMemcpy(h->bmask, bm.data(), sizeof(unsigned) * bm.size(), cudaMemcpyHostToDevice));
    CU(h, cudaMemcpy(h->bq, bq.data(), sizeof(double) * bq.size(), cudaMemcpyHostToDevice));
    h->nb = (int)bn.size();
    return LBM_OK;
}

int lbm_pressure_tensor(lbm_handle h, double *P, int on_device)
{
    int rc = check_ready(h);
    if (rc) return rc;
    if (!P) return fail(h, LBM_EINVAL, "null output");
    const size_t N = h->geo.M, na = h->D == 3 ? 6 : 3;
    // the dead population buffer holds (1 + 2D) N >= na N doubles
    double *out = on_device ? P : static_cast<double *>(h->fv[h->cur ^ 1]);
    rc = h->lattice == LBM_D2Q9 ? launch_pressure<0>(h, out) : launch_pressure<1>(h, out);
    if (rc) return rc;
    if (!on_device)
        CU(h, cudaMemcpyAsync(P, out, sizeof(double) * na * N, cudaMemcpyDeviceToHost, h->stream));
    return read_status(h);
}

int lbm_reduce(lbm_handle h, double *mass, double *momentum)
{
    int rc = check_ready(h);
    if (rc) return rc;
    if (!mass && !momentum) return LBM_EINVAL;
    rc = h->lattice == LBM_D2Q9 ? launch_reduce<0>(h) : launch_reduce<1>(h);
    if (rc) return rc;
    double s[4];
    CU(h, cudaMemcpyAsync(s, h->sums, sizeof(s), cudaMemcpyDeviceToHost, h->stream));
    rc = read_status(h);  // synchronises
    if (mass) *mass = s[0];
    if (momentum)
        for (int a = 0; a < h->D; ++a) momentum[a] = s[1 + a];
    return rc;
}

int lbm_get_populations(lbm_handle h, double *f, int on_device)
{
    int rc = check_ready(h);
    if (rc) return rc;
    if (!f) return LBM_EINVAL;
    const size_t N = h->geo.M, QN = (size_t)h->Q * N;
    if (shifted(h->storage)) {
        TempF64 t;   // of a host buffer; an aligned device buffer is written in place
        const bool direct = on_device && reinterpret_cast<uintptr_t>(f) % sizeof(double) == 0;
        if (!direct && (rc = temp_alloc(h, t))) return rc;
        double *out = direct ? f : t.p;
        rc = h->lattice == LBM_D2Q9 ? decode_to<0>(h, h->cur, out) : decode_to<1>(h, h->cur, out);
        if (rc) return rc;
        if (!direct) {
            CU(h, cudaMemcpyAsync(f, t.p, sizeof(double) * QN,
                                  on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost, h->stream));
            CU(h, cudaStreamSynchronize(h->stream));   // before the temporary is freed
        }
    } else if (h->storage == LBM_F32) {
        if (on_device) {
            convert_pops(h, h->geo.px, h->geo.nx, f32(h, h->cur), f);
            CU(h, cudaGetLastError());
            h->launches += 1;
        } else {
            const float *src = f32(h, h->cur);
            if (h->geo.px != h->geo.nx) {   // without the rows' padding, through the dead buffer
                convert_pops(h, h->geo.px, h->geo.nx, src, f32(h, h->cur ^ 1));
                CU(h, cudaGetLastError());
                h->launches += 1;
                src = f32(h, h->cur ^ 1);
            }
            std::vector<float> tmp(QN);
            CU(h, cudaMemcpyAsync(tmp.data(), src, sizeof(float) * QN, cudaMemcpyDeviceToHost, h->stream));
            CU(h, cudaStreamSynchronize(h->stream));
            for (size_t k = 0; k < QN; ++k) f[k] = tmp[k];
        }
    } else {
        CU(h, cudaMemcpyAsync(f, f64(h, h->cur), sizeof(double) * QN,
                              on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost,
                              h->stream));
    }
    rc = read_status(h);
    if (!on_device)
        for (size_t n = 0; n < N; ++n)
            if (h->mask_host[n])
                for (int i = 0; i < h->Q; ++i) f[(size_t)i * N + n] = 0.0;
    return rc;
}

int lbm_set_populations(lbm_handle h, const double *f, int on_device)
{
    if (!h || !f) return LBM_EINVAL;
    int rc = ensure_memory(h);
    if (rc) return rc;
    const size_t QN = (size_t)h->Q * h->geo.M;
    h->cur = 0;
    if (shifted(h->storage)) {
        TempF64 t;   // of a host buffer; an aligned device buffer is read in place
        const bool direct = on_device && reinterpret_cast<uintptr_t>(f) % sizeof(double) == 0;
        if (!direct) {
            if ((rc = temp_alloc(h, t))) return rc;
            CU(h, cudaMemcpyAsync(t.p, f, sizeof(double) * QN,
                                  on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice, h->stream));
        }
        const double *in = direct ? f : t.p;
        const Geo gu = lbmk::flat(h->geo);
        rc = h->lattice == LBM_D2Q9 ? encode_from<0>(h, gu, in) : encode_from<1>(h, gu, in);
        if (rc) return rc;
        if (!direct) CU(h, cudaStreamSynchronize(h->stream));   // before the temporary is freed
    } else if (h->storage == LBM_F32) {
        if (on_device) {
            convert_pops(h, h->geo.nx, h->geo.px, f, f32(h, 0));
            CU(h, cudaGetLastError());
            h->launches += 1;
        } else {
            std::vector<float> tmp(QN);
            for (size_t k = 0; k < QN; ++k) tmp[k] = (float)f[k];
            const bool pad = h->geo.px != h->geo.nx;   // the rows padded on the device, from the dead buffer
            CU(h, cudaMemcpyAsync(f32(h, pad), tmp.data(), sizeof(float) * QN, cudaMemcpyHostToDevice, h->stream));
            if (pad) {
                convert_pops(h, h->geo.nx, h->geo.px, f32(h, 1), f32(h, 0));
                CU(h, cudaGetLastError());
                h->launches += 1;
            }
            CU(h, cudaStreamSynchronize(h->stream));
        }
    } else {
        CU(h, cudaMemcpyAsync(f64(h, 0), f, sizeof(double) * QN,
                              on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice,
                              h->stream));
    }
    CU(h, cudaMemsetAsync(h->status, 0, sizeof(int), h->stream));
    rc = h->lattice == LBM_D2Q9 ? launch_fill_solid<0>(h) : launch_fill_solid<1>(h);
    if (rc) return rc;
    CU(h, cudaStreamSynchronize(h->stream));
    h->initialised = true;
    h->bad = false;
    return LBM_OK;
}

int lbm_sync(lbm_handle h, int timeout_ms)
{
    if (!h) return LBM_EINVAL;
    if (!h->initialised) return LBM_OK;
    if (timeout_ms >= 0) {
        cudaEvent_t ev;
        CU(h, cudaEventCreateWithFlags(&ev, cudaEventDisableTiming));
        cudaError_t e = cudaEventRecord(ev, h->stream);
        if (e != cudaSuccess) {
            cudaEventDestroy(ev);
            return fail(h, LBM_ECUDA, "cudaEventRecord: %s", cudaGetErrorString(e));
        }
        const auto t0 = std::chrono::steady_clock::now();
        for (;;) {
            e = cudaEventQuery(ev);
            if (e != cudaErrorNotReady) break;
            if (std::chrono::steady_clock::now() - t0 > std::chrono::milliseconds(timeout_ms)) {
                cudaEventDestroy(ev);
                return fail(h, LBM_ETIMEOUT, "work still running after %d ms", timeout_ms);
            }
            std::this_thread::sleep_for(std::chrono::microseconds(50));
        }
        cudaEventDestroy(ev);
        if (e != cudaSuccess) return fail(h, LBM_ECUDA, "stream error: %s", cudaGetErrorString(e));
    }
    return read_status(h);
}

int64_t lbm_launch_count(lbm_handle h) { return h ? h->launches : -1; }

int lbm_selftest_wait_timeout(long long limit_cycles, int *status_bits, double *ms)
{
    if (!status_bits || !ms || limit_cycles < 1 || limit_cycles > 2000000000ll) return LBM_EINVAL;
    int *st = nullptr;
    if (cudaMalloc(&st, sizeof(int)) != cudaSuccess) {
        cudaGetLastError();
        return LBM_ENOMEM;
    }
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    int rc = LBM_OK, host = 0;
    float t = 0.0f;
    if (cudaMemset(st, 0, sizeof(int)) != cudaSuccess || cudaEventCreate(&e0) != cudaSuccess ||
        cudaEventCreate(&e1) != cudaSuccess)
        rc = LBM_ECUDA;
    if (rc == LBM_OK) {
        cudaEventRecord(e0, 0);
        lbmf::k_wait_selftest<<<1, 64>>>(st, limit_cycles);
        cudaEventRecord(e1, 0);
        if (cudaEventSynchronize(e1) != cudaSuccess || cudaEventElapsedTime(&t, e0, e1) != cudaSuccess ||
            cudaMemcpy(&host, st, sizeof(int), cudaMemcpyDeviceToHost) != cudaSuccess)
            rc = LBM_ECUDA;
    }
    if (rc != LBM_OK) cudaGetLastError();
    if (e0) cudaEventDestroy(e0);
    if (e1) cudaEventDestroy(e1);
    cudaFree(st);
    if (rc == LBM_OK) {
        *status_bits = host;
        *ms = t;
    }
    return rc;
}

int lbm_probe_fp64_tflops(double *tflops)
{
    if (!tflops) return LBM_EINVAL;
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
        cudaGetLastError();
        return LBM_ECUDA;
    }
    const int threads = 256, blocks = 8 * sms, iters = 4096;
    double *out = nullptr;
    if (cudaMalloc(&out, sizeof(double) * threads * blocks) != cudaSuccess) {
        cudaGetLastError();
        return LBM_ENOMEM;
    }
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    int rc = LBM_OK;
    double best = 0.0;
    if (cudaEventCreate(&e0) != cudaSuccess || cudaEventCreate(&e1) != cudaSuccess) rc = LBM_ECUDA;
    for (int rep = 0; rep < 4 && rc == LBM_OK; ++rep) {   // the first launch warms up
        cudaEventRecord(e0, 0);
        lbmk::k_fp64_fma_probe<<<blocks, threads>>>(out, iters);
        cudaEventRecord(e1, 0);
        float ms = 0.0f;
        if (cudaEventSynchronize(e1) != cudaSuccess || cudaEventElapsedTime(&ms, e0, e1) != cudaSuccess) {
            rc = LBM_ECUDA;
            break;
        }
        const double tf = 2.0 * 8.0 * iters * (double)threads * blocks / (ms * 1e-3) / 1e12;
        if (rep > 0 && tf > best) best = tf;
    }
    if (rc != LBM_OK) cudaGetLastError();
    if (e0) cudaEventDestroy(e0);
    if (e1) cudaEventDestroy(e1);
    cudaFree(out);
    if (rc == LBM_OK) *tflops = best;
    return rc;
}

}  // extern "C"

struct lbm_batch_ctx {
    std::vector<lbm_ctx *> members;
    std::vector<int> cur0;   // each member's buffer index when the batch was made
    std::vector<cudaStream_t> prev;   // each member's stream before the batch
    int lattice = 0, storage = LBM_F32;
    cudaStream_t stream = nullptr;
    void *d_block = nullptr;   // the device memory of what follows
    lbmf::MemberF *d_members[2] = {nullptr, nullptr};   // step parity 0 and 1
    lbmf::WorkItem *d_items = nullptr;   // of the launches below, one after the other
    lbmf::BoxMaps *d_maps = nullptr;     // [member][buffer], TMA-staged launches
    // a step: launches of up to kBatchMembers TMA-staged D3Q27 members, and
    // one of all members that have no such form (or of all D2Q9 members)
    struct Launch {
        bool tma, solid, rest;   // rest: every member relaxes with time 1
        int first, n_items, eos;
        lbmf::BatchT args[2];   // TMA-staged: by step parity
    };
    std::vector<Launch> steps;
    int grid = 0, parity = 0;   // blocks of the plain launch
    cudaGraphExec_t graph = nullptr, graph_long = nullptr;   // two steps, kLongSteps steps
    long long nodes = 0;   // of all members
    int64_t launches = 0;
};

namespace {

template <typename ST>
void launch_batch_plain_shifted(lbm_batch_ctx *b, const lbmf::WorkItem *items, int n, int parity, cudaStream_t s)
{
    static std::atomic<unsigned long long> done{0};   // devices already opted in
    const int bytes = (int)sizeof(lbmf::SharedS<1>);
    smem_opt_in(lbmf::k_step_shifted_batch<1, ST>, bytes, done);
    lbmf::k_step_shifted_batch<1, ST><<<b->grid, lbmf::LatF<1>::TX * lbmf::LatF<1>::TY, bytes, s>>>(
        b->d_members[parity], items, n);
}

// D3Q27 members without tensor maps: no encoder in the CUDA driver, or rows that
// could not be padded (row_pitch).
void launch_batch_plain(lbm_batch_ctx *b, const lbmf::WorkItem *items, int n, int parity, cudaStream_t s)
{
    if (b->storage == LBM_F16S) launch_batch_plain_shifted<__half>(b, items, n, parity, s);
    else if (b->storage == LBM_BF16S) launch_batch_plain_shifted<__nv_bfloat16>(b, items, n, parity, s);
    else {
        static std::atomic<unsigned long long> done{0};   // devices already opted in
        const int bytes = (int)sizeof(lbmf::SharedF<1>);
        smem_opt_in(lbmf::k_step_f32_batch<1>, bytes, done);
        lbmf::k_step_f32_batch<1><<<b->grid, lbmf::LatF<1>::TX * lbmf::LatF<1>::TY, bytes, s>>>(
            b->d_members[parity], items, n);
    }
}

template <typename ST, bool REST>
void launch_batch_2d_r(lbm_batch_ctx *b, const lbmf::WorkItem *items, int n, int parity, cudaStream_t s)
{
    static std::atomic<int> known{0};
    const bool overlap = leaves_no_room(lbmf2::k_step2d_batch<ST, REST>, n, lbmf2::NT, b->members[0]->sms, known);
    lbmpdl::launch_step(overlap, lbmf2::k_step2d_batch<ST, REST>, n, lbmf2::NT, 0, s, b->d_members[parity], items);
}

template <typename ST>
void launch_batch_2d(lbm_batch_ctx *b, const lbmf::WorkItem *items, int n, bool rest, int parity, cudaStream_t s)
{
    if (rest) launch_batch_2d_r<ST, true>(b, items, n, parity, s);
    else      launch_batch_2d_r<ST, false>(b, items, n, parity, s);
}

// One step of every member.
void batch_launch(lbm_batch_ctx *b, int parity, cudaStream_t s)
{
    for (const lbm_batch_ctx::Launch &l : b->steps) {
        const lbmf::WorkItem *items = b->d_items + l.first;
        if (l.tma) {
            if (b->storage == LBM_F32) lbmtma::launch_batch(l.args[parity], items, l.n_items, l.eos, l.solid, l.rest, s);
            else if (b->storage == LBM_F16S)
                lbmtma::launch_batch_shifted<__half>(l.args[parity], items, l.n_items, l.solid, l.rest, s);
            else
                lbmtma::launch_batch_shifted<__nv_bfloat16>(l.args[parity], items, l.n_items, l.solid, l.rest, s);
        } else if (b->lattice != LBM_D2Q9) launch_batch_plain(b, items, l.n_items, parity, s);
        else if (b->storage == LBM_F32) launch_batch_2d<float>(b, items, l.n_items, l.rest, parity, s);
        else if (b->storage == LBM_F16S) launch_batch_2d<__half>(b, items, l.n_items, l.rest, parity, s);
        else launch_batch_2d<__nv_bfloat16>(b, items, l.n_items, l.rest, parity, s);
    }
}

// When the last of the items ends if each free one of `slots` takes the next:
// runs of (planes, number of items), a block of p planes taking p + 4.5. Slots
// that are free at the same time are kept as one entry.
double batch_end(const std::vector<std::pair<int, long long>> &runs, int slots)
{
    std::map<double, long long> free{{0.0, slots}};
    double end = 0.0;
    for (const auto &run : runs)
        for (long long left = run.second; left > 0;) {
            const auto first = free.begin();
            const double t = first->first + run.first + 4.5;
            const long long n = std::min(left, first->second);
            if (n == first->second) free.erase(first);
            else                    first->second -= n;
            free[t] += n;
            end = std::max(end, t);
            left -= n;
        }
    return end;
}

// Chunks of the members (by number) of one TMA-staged launch, and its items,
// longest first: members' march axes in equal parts of at most `cap` planes,
// with the cap that ends first when each free slot (SM, or half of one where two
// blocks are resident and the items need them, see best_chunk) takes the next
// item. Caps that make many times more items than there are slots balance no
// better and are not looked at.
std::vector<lbmf::WorkItem> batch_items(const std::vector<lbm_ctx *> &members, const std::vector<int> &which,
                                        int sms, int resident, std::vector<int> &chunks)
{
    const auto tiles = [&](size_t k) {
        const GeoF &g = members[which[k]]->geof;
        return (long long)((g.nx + 31) / 32) * ((g.ny + 7) / 8);
    };
    double best = 1e300;
    std::vector<int> seen;
    for (int cap : {1 << 30, 96, 64, 40, 24, 12, 8, 6, 4}) {
        std::vector<int> ch;
        std::map<int, long long, std::greater<int>> by_length;
        long long count = 0;
        for (size_t k = 0; k < which.size(); ++k) {
            const int nz = members[which[k]]->geof.nz, n = (nz + cap - 1) / cap, c = (nz + n - 1) / n;
            ch.push_back(c);
            by_length[c] += tiles(k) * (nz / c);
            if (nz % c) by_length[nz % c] += tiles(k);
            count += tiles(k) * ((nz + c - 1) / c);
        }
        if (ch == seen) continue;
        seen = ch;
        const bool shared = resident == 2 && count > sms;
        const int slots = shared ? 2 * sms : sms;
        const double cost = (shared ? 1.31 : 1.0) * batch_end({by_length.begin(), by_length.end()}, slots);
        if (cost < best) {
            best = cost;
            chunks = ch;
        }
        if (count > 10ll * slots) break;
    }
    struct Part { int k, len, bz; };
    std::vector<Part> parts;
    for (size_t k = 0; k < which.size(); ++k) {
        const int nz = members[which[k]]->geof.nz, c = chunks[k];
        for (int bz = 0; bz * c < nz; ++bz) parts.push_back({(int)k, std::min(c, nz - bz * c), bz});
    }
    std::stable_sort(parts.begin(), parts.end(), [](const Part &a, const Part &b) { return a.len > b.len; });
    std::vector<lbmf::WorkItem> items;
    for (const Part &q : parts) {
        const GeoF &g = members[which[q.k]]->geof;
        for (int by = 0; by < (g.ny + 7) / 8; ++by)
            for (int bx = 0; bx < (g.nx + 31) / 32; ++bx) items.push_back({q.k, bx, by, q.bz});
    }
    return items;
}

// `steps` (even) steps from parity 0, captured once.
int batch_graph(lbm_batch_ctx *b, cudaGraphExec_t &graph, int steps)
{
    if (graph) return LBM_OK;
    cudaStream_t cap = nullptr;
    if (cudaStreamCreateWithFlags(&cap, cudaStreamNonBlocking) != cudaSuccess) return LBM_ECUDA;
    cudaGraph_t gr = nullptr;
    cudaError_t e = cudaStreamBeginCapture(cap, cudaStreamCaptureModeThreadLocal);
    if (e == cudaSuccess) {
        for (int k = 0; k < steps; ++k) batch_launch(b, k & 1, cap);
        e = cudaStreamEndCapture(cap, &gr);
    }
    if (e == cudaSuccess) e = cudaGraphInstantiate(&graph, gr, 0);
    if (gr) cudaGraphDestroy(gr);
    cudaStreamDestroy(cap);
    if (e == cudaSuccess) return LBM_OK;
    graph = nullptr;
    cudaGetLastError();
    return LBM_ECUDA;
}

void batch_free(lbm_batch_ctx *b)
{
    if (!b) return;
    if (b->graph) cudaGraphExecDestroy(b->graph);
    if (b->graph_long) cudaGraphExecDestroy(b->graph_long);
    if (b->d_block) cudaFree(b->d_block);
    for (size_t k = 0; k < b->prev.size(); ++k) b->members[k]->stream = b->prev[k];
    if (b->stream) cudaStreamDestroy(b->stream);
    cudaGetLastError();
    delete b;
}

// b: the batch under construction, freed by the caller if this fails.
int batch_build(lbm_batch_ctx *&b, const lbm_handle *members, int count)
{
    const int lattice = members[0] ? members[0]->lattice : -1;
    const int storage = members[0] ? members[0]->storage : -1;
    if (storage == LBM_F64) return LBM_EINVAL;
    for (int k = 0; k < count; ++k) {
        lbm_ctx *h = members[k];
        if (!h || !h->initialised || h->bad || h->storage != storage || h->lattice != lattice ||
            h->nb > 0 ||   // interpolated bounce-back is not part of the batched step
            h->e64)        // nor the FP64-EOS form
            return LBM_EINVAL;
        for (int j = 0; j < k; ++j)
            if (members[j] == h) return LBM_EINVAL;   // a lattice at most once
    }
    b = new lbm_batch_ctx();
    b->lattice = lattice;
    b->storage = storage;
    b->members.assign(members, members + count);
    for (lbm_ctx *h : b->members) {
        b->cur0.push_back(h->cur);
        b->prev.push_back(h->stream);
        b->nodes += h->geo.M;
    }
    for (lbm_ctx *h : b->members) cudaStreamSynchronize(h->stream);
    if (cudaStreamCreateWithFlags(&b->stream, cudaStreamNonBlocking) != cudaSuccess) return LBM_ECUDA;
    int sms = 0, dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    sms = std::max(sms, 1);
    std::vector<lbmf::MemberF> desc[2];
    std::vector<lbmf::WorkItem> items, plain;
    std::vector<lbmf::BoxMaps> maps;
    std::vector<int> staged;   // members with a TMA-staged form
    for (int k = 0; k < count; ++k)
        if (lattice == LBM_D3Q27 && b->members[k]->tmap_ready) staged.push_back(k);
    for (int k = 0; k < count; ++k) {
        lbm_ctx *h = b->members[k];
        const bool tma = lattice == LBM_D3Q27 && h->tmap_ready;
        for (int par = 0; par < 2; ++par) maps.push_back(h->tmaps[par]);
        // D3Q27: 32 x 8 columns by z-chunks; D2Q9: 32 x 8 tiles of the (x, 2D y) plane
        const int tx = (h->geof.nx + 31) / 32;
        const int ty = ((lattice == LBM_D2Q9 ? h->geof.nz : h->geof.ny) + 7) / 8;
        GeoF geof = h->geof;
        if (h->auto_form && lattice == LBM_D3Q27) geof.chunk = kDefaultChunk3;   // the plain form's
        const int tz = lattice == LBM_D2Q9 ? 1 : (geof.nz + geof.chunk - 1) / geof.chunk;
        for (int par = 0; par < 2 && (int)staged.size() < count; ++par) {   // (staged launches carry theirs)
            lbmf::MemberF m;
            m.g = geof;
            m.p = h->physf;
            m.mask = h->any_solid ? h->mask : nullptr;
            m.src = h->fv[h->cur ^ par];
            m.dst = h->fv[h->cur ^ par ^ 1];
            m.rho_src = h->rs[h->cur ^ par];
            m.rho_dst = h->rs[h->cur ^ par ^ 1];
            m.status = h->status;
            m.tiles_x = tx;
            m.tiles_y = ty;
            desc[par].push_back(m);
        }
        if (!tma)
            for (int bz = 0; bz < tz; ++bz)
                for (int by = 0; by < ty; ++by)
                    for (int bx = 0; bx < tx; ++bx) plain.push_back({k, bx, by, bz});
        h->stream = b->stream;   // members' later work is ordered after the batch
    }
    // TMA-staged launches, of as many members each as come out even (the launches
    // of a step run one after the other), then the plain or D2Q9 one
    const size_t n_staged = (staged.size() + lbmf::kBatchMembers - 1) / lbmf::kBatchMembers;
    std::vector<std::vector<int>> which(n_staged), chunks(n_staged);
    b->steps.reserve(n_staged + 1);
    for (size_t g = 0; g < n_staged; ++g) {
        which[g].assign(staged.begin() + staged.size() * g / n_staged, staged.begin() + staged.size() * (g + 1) / n_staged);
        const std::vector<lbmf::WorkItem> part =
            batch_items(b->members, which[g], sms, storage == LBM_F32 ? 1 : 2, chunks[g]);
        b->steps.emplace_back();
        lbm_batch_ctx::Launch &l = b->steps.back();
        l.tma = true;
        l.first = (int)items.size();
        l.n_items = (int)part.size();
        items.insert(items.end(), part.begin(), part.end());
    }
    if (!plain.empty()) {
        b->steps.emplace_back();
        lbm_batch_ctx::Launch &l = b->steps.back();
        l.first = (int)items.size();
        l.n_items = (int)plain.size();
        l.rest = true;
        for (const lbm_ctx *h : b->members) l.rest = l.rest && lbmf::at_rest(h->physf);
        b->grid = std::min(l.n_items, 2 * sms);
        items.insert(items.end(), plain.begin(), plain.end());
    }
    // one block of device memory, filled by one copy: members of both parities,
    // tensor maps, items
    const size_t db = sizeof(lbmf::MemberF) * desc[0].size();
    const size_t mb = staged.empty() ? 0 : sizeof(lbmf::BoxMaps) * maps.size(), ib = sizeof(lbmf::WorkItem) * items.size();
    const size_t o_maps = 2 * align_up(db), o_items = o_maps + align_up(mb);
    std::vector<unsigned char> block(o_items + ib);
    for (int par = 0; par < 2; ++par)
        if (db) memcpy(&block[par * align_up(db)], desc[par].data(), db);
    if (mb) memcpy(&block[o_maps], maps.data(), mb);
    memcpy(&block[o_items], items.data(), ib);
    if (cudaMalloc(&b->d_block, block.size()) != cudaSuccess) return LBM_ENOMEM;
    char *const d = static_cast<char *>(b->d_block);
    for (int par = 0; par < 2; ++par) b->d_members[par] = reinterpret_cast<lbmf::MemberF *>(d + par * align_up(db));
    b->d_maps = reinterpret_cast<lbmf::BoxMaps *>(d + o_maps);
    b->d_items = reinterpret_cast<lbmf::WorkItem *>(d + o_items);
    for (size_t g = 0; g < n_staged; ++g) {
        lbm_batch_ctx::Launch &l = b->steps[g];
        l.eos = b->members[which[g][0]]->physf.eos;
        l.rest = true;
        for (size_t k = 0; k < which[g].size(); ++k) {
            const lbm_ctx *h = b->members[which[g][k]];
            l.solid = l.solid || h->any_solid;
            l.rest = l.rest && lbmf::at_rest(h->physf);
            if (h->physf.eos != l.eos) l.eos = -1;
            for (int par = 0; par < 2; ++par) {
                lbmf::MemberT &m = l.args[par].m[k];
                m.g = h->geof;
                m.g.chunk = chunks[g][k];
                m.p = h->physf;
                m.mask = h->mask;
                m.src = h->fv[h->cur ^ par];
                m.dst = h->fv[h->cur ^ par ^ 1];
                m.rho_src = h->rs[h->cur ^ par];
                m.rho_dst = h->rs[h->cur ^ par ^ 1];
                m.status = h->status;
                m.maps = b->d_maps + 2 * which[g][k] + (h->cur ^ par);
            }
        }
    }
    // on the batch's stream, which does not wait for the default one
    if (cudaMemcpyAsync(b->d_block, block.data(), block.size(), cudaMemcpyHostToDevice, b->stream) != cudaSuccess ||
        cudaStreamSynchronize(b->stream) != cudaSuccess) return LBM_ECUDA;
    return LBM_OK;
}

}  // namespace

extern "C" {

int lbm_batch_create(lbm_batch *out, const lbm_handle *members, int count)
{
    if (!out || !members || count < 1) return LBM_EINVAL;
    *out = nullptr;
    lbm_batch_ctx *b = nullptr;
    int rc;
    try {
        rc = batch_build(b, members, count);
    } catch (const std::bad_alloc &) {
        rc = LBM_ENOMEM;
    }
    if (rc == LBM_OK) *out = b;
    else              batch_free(b);
    return rc;
}

int lbm_batch_step(lbm_batch b, int64_t n)
{
    if (!b || n < 0) return LBM_EINVAL;
    for (lbm_ctx *h : b->members)
        if (h->bad) return LBM_ESTATE;
    if (n >= 4) {
        if (b->parity != 0) {
            batch_launch(b, b->parity, b->stream);
            b->parity ^= 1;
            ++b->launches;
            --n;
        }
        const bool longer = n >= 2 * kLongSteps && b->nodes <= (long long)kLongNodes;
        int rc = batch_graph(b, b->graph, 2);
        if (rc == LBM_OK && longer) rc = batch_graph(b, b->graph_long, kLongSteps);
        if (rc != LBM_OK) return rc;
        while (n >= 2) {
            const int k = longer && n >= kLongSteps ? kLongSteps : 2;
            if (cudaGraphLaunch(k == 2 ? b->graph : b->graph_long, b->stream) != cudaSuccess) return LBM_ECUDA;
            b->launches += k;
            n -= k;
        }
    }
    for (int64_t k = 0; k < n; ++k) {
        batch_launch(b, b->parity, b->stream);
        b->parity ^= 1;
        ++b->launches;
    }
    if (cudaGetLastError() != cudaSuccess) return LBM_ECUDA;
    return LBM_OK;
}

int lbm_batch_sync(lbm_batch b)
{
    if (!b) return LBM_EINVAL;
    if (cudaStreamSynchronize(b->stream) != cudaSuccess) return LBM_ECUDA;
    // members' state buffers follow the batch parity; their moments, reductions
    // and population reads are valid between lbm_batch_sync and the next step
    int bad = LBM_OK;
    for (size_t k = 0; k < b->members.size(); ++k) {
        lbm_ctx *h = b->members[k];
        h->cur = b->cur0[k] ^ b->parity;
        int rc = read_status(h);
        if (rc && !bad) bad = rc;
    }
    return bad;
}

int64_t lbm_batch_launch_count(lbm_batch b) { return b ? b->launches : -1; }

void lbm_batch_destroy(lbm_batch b)
{
    if (!b) return;
    cudaStreamSynchronize(b->stream);
    for (size_t k = 0; k < b->members.size(); ++k) b->members[k]->cur = b->cur0[k] ^ b->parity;
    batch_free(b);
}

int lbm_time_kernels(lbm_handle h, int64_t n, double *ms)
{
    int rc = check_ready(h);
    if (rc) return rc;
    if (n < 1 || !ms) return fail(h, LBM_EINVAL, "need n >= 1 and an output array");
    if (h->bad) return fail(h, LBM_ESTATE, "state holds a non-finite density; re-initialise");
    std::vector<cudaEvent_t> ev(3 * n);
    for (auto &e : ev) CU(h, cudaEventCreate(&e));
    const dim3 gr = node_grid(h->geo), bl = node_block(h->geo);
    const bool fused = h->storage != LBM_F64;
    for (int64_t k = 0; k < n; ++k) {
        CU(h, cudaEventRecord(ev[3 * k], h->stream));
        if (fused) {
            CU(h, cudaEventRecord(ev[3 * k + 1], h->stream));
            if (shifted(h->storage)) launch_shifted(h, h->stream, h->cur);
            else                     launch_f32(h, h->stream, h->cur);
            h->launches += 1;
        } else {
            const double *src = f64(h, h->cur);
            double *dst = f64(h, h->cur ^ 1);
            if (h->lattice == LBM_D2Q9)
                lbmk::k_macro<0, true><<<gr, bl, 0, h->stream>>>(h->geo, h->phys, h->mask, src, h->rp,
                                                           h->u, h->gflux, h->status);
            else
                lbmk::k_macro<1, true><<<gr, bl, 0, h->stream>>>(h->geo, h->phys, h->mask, src, h->rp,
                                                           h->u, h->gflux, h->status);
            CU(h, cudaEventRecord(ev[3 * k + 1], h->stream));
            if (h->lattice == LBM_D2Q9) launch_collide64<0>(h, h->stream, src, dst);
            else                        launch_collide64<1>(h, h->stream, src, dst);
            h->launches += 2;
        }
        CU(h, cudaEventRecord(ev[3 * k + 2], h->stream));
        CU(h, cudaGetLastError());
        h->cur ^= 1;
    }
    CU(h, cudaStreamSynchronize(h->stream));
    double t0 = 0.0, t1 = 0.0;
    for (int64_t k = 0; k < n; ++k) {
        float a = 0.f, b = 0.f;
        CU(h, cudaEventElapsedTime(&a, ev[3 * k], ev[3 * k + 1]));
        CU(h, cudaEventElapsedTime(&b, ev[3 * k + 1], ev[3 * k + 2]));
        t0 += a;
        t1 += b;
    }
    for (auto &e : ev) cudaEventDestroy(e);
    ms[0] = t0 / n;
    ms[1] = t1 / n;
    return read_status(h);
}

int lbm_autotune(lbm_handle h, int *chunk_out)
{
    int rc = check_ready(h);
    if (rc) return rc;
    if (h->storage == LBM_F64) {
        if (chunk_out) *chunk_out = 0;
        return LBM_OK;   // the FP64 step has no tile parameters
    }
    if (h->bad) return fail(h, LBM_ESTATE, "state holds a non-finite density; re-initialise");
    if (h->lattice == LBM_D2Q9) {   // nor has the D2Q9 step: its chunk changes nothing
        if ((rc = read_status(h))) return rc;
        if (chunk_out) *chunk_out = h->geof.chunk;
        return LBM_OK;
    }
    const size_t bytes = pop_bytes(h->storage) * (size_t)h->Q * h->geo.N;
    const size_t rbytes = shifted(h->storage) ? sizeof(float) * h->geo.N : 0;
    void *save = nullptr;
    if (cudaMalloc(&save, bytes + rbytes) != cudaSuccess) {
        cudaGetLastError();
        return fail(h, LBM_ENOMEM, "autotune: no room to save the state");
    }
    CU(h, cudaMemcpyAsync(save, h->fv[h->cur], bytes, cudaMemcpyDeviceToDevice, h->stream));
    if (rbytes)
        CU(h, cudaMemcpyAsync(static_cast<char *>(save) + bytes, h->rs[h->cur], rbytes,
                              cudaMemcpyDeviceToDevice, h->stream));
    const int nz = h->geof.nz;
    // plane chunks per CTA; on a march axis longer than 128 planes also 10/16
    // .. 16/16 of it: one long chunk per column and a short one after it,
    // whose blocks (launched after all long ones) fill the last wave
    std::vector<int> cands = {4, 6, 8, 11, 13, 16, 22, 26, 32, 43, 64, 128};
    if (nz > 128)
        for (int k = 10; k <= 16; ++k) cands.push_back(std::max(129, nz * k / 16));
    for (int resident : {1, 2}) cands.push_back(best_chunk(h->geof, 8, h->sms, resident));
    std::sort(cands.begin(), cands.end());
    const int chunk0 = h->geof.chunk, rows0 = h->tile_rows;   // restored on failure
    const bool auto0 = h->auto_form;
    h->auto_form = false;
    // every form of the storage; FP32 also 32 x 8 and 32 x 7 tiles (the forms up
    // to LBM_FUSED_TMEM)
    const bool fp32 = h->storage == LBM_F32 && !h->e64;   // the FP64-EOS form is plain 32 x 8
    const int variant0 = h->variant;
    int best = h->geof.chunk, best_rows = h->tile_rows, best_variant = h->variant;
    double best_ms = 1e30;
    for (int var = 0; var <= LBM_FUSED_TM_TMA && rc == LBM_OK; ++var) {
        // shifted storage: no warp-specialised form without Tensor Memory
        if (var > 0 && (h->e64 || (!fp32 && var == LBM_FUSED_WARP_SPECIALISED))) continue;
        if ((var == LBM_FUSED_WS_TMA || var == LBM_FUSED_TM_TMA) && !h->tmap_ready) continue;
        if (var == LBM_FUSED_TM_TMA && !shifted(h->storage)) continue;   // a form of shifted storage
        h->variant = var;
        for (int rows : {8, 7}) {
            if (rows == 7 && (!fp32 || var >= LBM_FUSED_WS_TMEM)) continue;
            h->tile_rows = rows;
            for (size_t j = 0; j < cands.size(); ++j) {
                const int c = cands[j];
                if ((c > nz && j != 0) || (j > 0 && c == cands[j - 1])) continue;
                h->geof.chunk = c;
                double ms[2];
                rc = lbm_time_kernels(h, 1, ms);                  // warm-up
                if (rc == LBM_OK) rc = lbm_time_kernels(h, 6, ms);
                if (rc != LBM_OK) break;
                if (ms[1] < best_ms) { best_ms = ms[1]; best = c; best_rows = rows; best_variant = var; }
            }
            if (rc != LBM_OK) break;
        }
    }
    // the best candidate, or on failure the kernel, chunk and tile the handle
    // had; a graph captured before the search may hold either, so it is dropped
    h->tile_rows = rc == LBM_OK ? best_rows : rows0;
    h->geof.chunk = rc == LBM_OK ? best : chunk0;
    h->variant = rc == LBM_OK ? best_variant : variant0;
    if (rc != LBM_OK) h->auto_form = auto0;
    drop_graphs(h);
    cudaError_t e = cudaMemcpyAsync(h->fv[0], save, bytes, cudaMemcpyDeviceToDevice, h->stream);
    if (e == cudaSuccess && rbytes)
        e = cudaMemcpyAsync(h->rs[0], static_cast<char *>(save) + bytes, rbytes,
                            cudaMemcpyDeviceToDevice, h->stream);
    cudaStreamSynchronize(h->stream);
    cudaFree(save);
    if (e != cudaSuccess) return fail(h, LBM_ECUDA, "autotune restore: %s", cudaGetErrorString(e));
    h->cur = 0;
    if (rc != LBM_OK) return rc;
    if (chunk_out) *chunk_out = best;
    return LBM_OK;
}

int lbm_get_tile(lbm_handle h, int *tile_x, int *tile_y)
{
    if (!h) return LBM_EINVAL;
    int tx = 0, ty = 0;
    if (h->storage != LBM_F64) {
        tx = h->lattice == LBM_D2Q9 ? lbmf::LatF<0>::TX : lbmf::LatF<1>::TX;
        ty = h->lattice == LBM_D2Q9 ? lbmf::LatF<0>::TY
             : (h->tile_rows == 7 && h->storage == LBM_F32) ? 7 : lbmf::LatF<1>::TY;
    }
    if (tile_x) *tile_x = tx;
    if (tile_y) *tile_y = ty;
    return LBM_OK;
}

int lbm_set_tile(lbm_handle h, int tile_y)
{
    if (!h) return LBM_EINVAL;
    if (h->lattice != LBM_D3Q27 || h->storage != LBM_F32)
        return fail(h, LBM_EINVAL, "the tile height is a parameter of the D3Q27 FP32 step only");
    if (tile_y != 7 && tile_y != 8) return fail(h, LBM_EINVAL, "tile height must be 7 or 8");
    if (tile_y == 7 && h->e64) return fail(h, LBM_EINVAL, "the FP64-EOS step runs 8-row tiles");
    if (tile_y == 7 && !h->auto_form && h->variant >= LBM_FUSED_WS_TMEM)
        return fail(h, LBM_EINVAL, "the warp-specialised Tensor Memory forms run 8-row tiles");
    leave_auto_form(h);
    if (h->tile_rows != tile_y) drop_graphs(h);  // the captured graph holds the other kernel
    h->tile_rows = tile_y;
    return LBM_OK;
}

int lbm_set_fused_variant(lbm_handle h, int variant)
{
    if (!h) return LBM_EINVAL;
    if (variant < LBM_FUSED_PLAIN || variant > LBM_FUSED_TM_TMA)
        return fail(h, LBM_EINVAL, "unknown fused-step variant %d", variant);
    if (variant == LBM_FUSED_TM_TMA && !shifted(h->storage))
        return fail(h, LBM_EINVAL, "the one-group TMA-staged form is a form of shifted storage");
    if (variant >= LBM_FUSED_WS_TMEM && (h->lattice != LBM_D3Q27 || h->tile_rows != 8))
        return fail(h, LBM_EINVAL, "the warp-specialised Tensor Memory forms run D3Q27 32 x 8 tiles");
    // with the memory laid out the tensor maps decide (rows are padded for them,
    // so that what lbm_autotune or the handle chose can be set); before that, the width
    const int mult = tma_nx_multiple(h->storage);
    if ((variant == LBM_FUSED_WS_TMA || variant == LBM_FUSED_TM_TMA) &&
        (!mult || (h->fv[0] ? !h->tmap_ready : h->geo.nx % mult != 0)))
        return fail(h, LBM_EINVAL, "the TMA-staged forms need FP32 or shifted storage and the CUDA driver's tensor-map "
                                   "encoder and, before the memory is laid out, nx a multiple of 4 (FP32) or 8 (shifted)");
    if (h->storage == LBM_F64 && variant != LBM_FUSED_PLAIN)
        return fail(h, LBM_EINVAL, "the FP64 step has one form");
    if (h->e64 && variant != LBM_FUSED_PLAIN)
        return fail(h, LBM_EINVAL, "the FP64-EOS step has one form");
    if (shifted(h->storage) && variant == LBM_FUSED_WARP_SPECIALISED)
        return fail(h, LBM_EINVAL, "shifted storage has the plain and the Tensor Memory forms");
    leave_auto_form(h);
    if (h->variant != variant) drop_graphs(h);  // the captured graph holds the other kernel
    h->variant = variant;
    return LBM_OK;
}

int lbm_get_fused_variant(lbm_handle h, int *variant)
{
    if (!h || !variant) return LBM_EINVAL;
    *variant = h->variant;
    return LBM_OK;
}

int lbm_set_chunk(lbm_handle h, int chunk)
{
    if (!h) return LBM_EINVAL;
    if (chunk < 1) return fail(h, LBM_EINVAL, "chunk must be >= 1");
    leave_auto_form(h);
    if (h->geof.chunk != chunk) drop_graphs(h);
    h->geof.chunk = chunk;
    return LBM_OK;
}

const char *lbm_last_error(lbm_handle h) { return h ? h->err : "null handle"; }

void lbm_destroy(lbm_handle h)
{
    if (!h) return;
    if (h->stream) cudaStreamSynchronize(h->stream);
    drop_graphs(h);
    if (h->cap_stream) cudaStreamDestroy(h->cap_stream);
    if (h->owns_base && h->base) cudaFree(h->base);
    if (h->bn) cudaFree(h->bn);
    if (h->bmask) cudaFree(h->bmask);
    if (h->bq) cudaFree(h->bq);
    if (h->own_stream) cudaStreamDestroy(h->own_stream);
    if (h->poll_ev) cudaEventDestroy(h->poll_ev);
    if (h->poll_host) cudaFreeHost(h->poll_host);
    cudaGetLastError();
    delete h;
}

}  // extern "C"
