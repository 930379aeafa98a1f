// roeam3_api.cu — host implementation of the 3D C ABI declared in include/roeam3.h.
//
// Owns the device memory of a batch of 3D grids (pitched rows of cells, each a quad and a tail of
// values), builds the work units of the 3D stage kernel (a rectangle of columns by a segment of
// planes), and drives the three fused stage launches of each SSP-RK3 step with per-grid time steps
// read on the device.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <cstring>
#include <utility>
#include <vector>

#include "roeam.h"
#include "roeam3.h"
#include "roeam3_internal.h"

using namespace roeam;

namespace {

roeam_status fail3(roeam_status st, const char *fmt, ...)
{
    char buf[512];
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(buf, sizeof(buf), fmt, ap);
    va_end(ap);
    return (roeam_status)record_error(st, buf);
}

#define CUDA_TRY3(expr)                                                                                      \
    do {                                                                                                     \
        cudaError_t e_ = (expr);                                                                             \
        if (e_ != cudaSuccess)                                                                               \
            return fail3(e_ == cudaErrorMemoryAllocation ? ROEAM_E_OOM : ROEAM_E_CUDA, "%s: %s (%s:%d)", #expr, \
                         cudaGetErrorString(e_), __FILE__, __LINE__);                                        \
    } while (0)

long long round_up3(long long a, long long m) { return (a + m - 1) / m * m; }

}  // namespace

struct roeam3_grid {
    int device = 0;
    cudaStream_t stream = nullptr;
    int precision = 32, nscal = 0, nv = 5, count = 0;
    size_t esize = 4;
    std::vector<GridDev3> hg;
    GridDev3 *d_grids = nullptr;
    void *d_coef = nullptr;
    void *U = nullptr, *A = nullptr, *B = nullptr;
    long long total_elems = 0, total_packed = 0, max_cells = 0;
    int4 *d_units = nullptr;
    int nunits = 0, threads = 0;
    size_t smem = 0;
    unsigned long long *rate = nullptr;   // 2 x count slots, alternating by step parity
    int parity = 0;
    unsigned *status = nullptr;
    double *staging = nullptr;            // float64 packed copy on the device
    double *partials = nullptr;
    double *h_red = nullptr;              // pinned
    unsigned *h_status = nullptr;         // pinned
    unsigned long long *h_rate = nullptr; // pinned
    unsigned long long launches = 0;
};

namespace {

roeam_status validate3(int count, const roeam3_grid_desc *d)
{
    if (count < 1 || !d) return fail3(ROEAM_E_ARG, "count must be >= 1 and descs non-null");
    if (count > 65535) return fail3(ROEAM_E_ARG, "count must be <= 65535 grids per handle");
    for (int k = 0; k < count; ++k) {
        const roeam3_grid_desc &q = d[k];
        const roeam_params &p = q.p;
        if (q.ni < 1 || q.nj < 1 || q.nk < 1 || q.ni > 65535 || q.nj > 65535 || q.nk > 65535)
            return fail3(ROEAM_E_ARG, "grid %d: ni, nj, nk must be in 1..65535", k);
        if ((long long)q.ni * q.nj * q.nk > (1ll << 28)) return fail3(ROEAM_E_ARG, "grid %d: too many cells", k);
        if (!(q.dx > 0.0) || !(q.dy > 0.0) || !(q.dz > 0.0)) return fail3(ROEAM_E_ARG, "grid %d: dx, dy, dz must be > 0", k);
        if (q.nscal < 0 || q.nscal > ROEAM3_MAX_SCALARS) return fail3(ROEAM_E_ARG, "grid %d: nscal must be 0..3", k);
        if (q.nscal != d[0].nscal) return fail3(ROEAM_E_ARG, "grid %d: nscal differs within the batch", k);
        if (q.reserved_ != 0) return fail3(ROEAM_E_ARG, "grid %d: reserved_ must be 0", k);
        if (!(p.gamma > 1.0)) return fail3(ROEAM_E_ARG, "grid %d: gamma must be > 1", k);
        if (!(p.m_ref > 0.0)) return fail3(ROEAM_E_ARG, "grid %d: m_ref must be > 0", k);
        if (!(p.u_ref > 0.0)) return fail3(ROEAM_E_ARG, "grid %d: u_ref must be > 0", k);
        if (!(p.eps2 >= 0.0)) return fail3(ROEAM_E_ARG, "grid %d: eps2 must be >= 0", k);
        if (p.eps1 != 0 && p.eps1 != 1) return fail3(ROEAM_E_ARG, "grid %d: eps1 must be 0 or 1", k);
        if (p.use_s1 != 0 && p.use_s1 != 1) return fail3(ROEAM_E_ARG, "grid %d: use_s1 must be 0 or 1", k);
        if (p.xi_form != 0 && p.xi_form != 1) return fail3(ROEAM_E_ARG, "grid %d: xi_form must be 0 or 1", k);
        if (p.recon != ROEAM_RECON_FIRST) return fail3(ROEAM_E_ARG, "grid %d: the 3D path is first order (recon 0)", k);
        if (p.scheme || p.dup_mode || p.no_ufix || p.xi_roe || p.harten != 0.0 || p.reserved_)
            return fail3(ROEAM_E_ARG, "grid %d: the 3D path has no ablation variants", k);
        if (p.precision != 32 && p.precision != 64) return fail3(ROEAM_E_ARG, "grid %d: precision must be 32 or 64", k);
        if (p.precision != d[0].p.precision) return fail3(ROEAM_E_ARG, "grid %d: precision differs within the batch", k);
        for (int s = 0; s < 6; ++s)
            if (q.bc[s] < 0 || q.bc[s] > 3) return fail3(ROEAM_E_ARG, "grid %d: bad boundary type on side %d", k, s);
        for (int a = 0; a < 3; ++a)
            if ((q.bc[2 * a] == ROEAM_BC_PERIODIC) != (q.bc[2 * a + 1] == ROEAM_BC_PERIODIC))
                return fail3(ROEAM_E_ARG, "grid %d: PERIODIC must be set on both sides of axis %d", k, a);
        for (int s = 0; s < 6; ++s)
            if (q.bc[s] == ROEAM_BC_INFLOW && !(q.inflow[0] > 0.0 && q.inflow[4] > 0.0))
                return fail3(ROEAM_E_ARG, "grid %d: inflow density and pressure must be > 0", k);
    }
    return ROEAM_OK;
}

template <typename T>
GridCoef3<T> make_coef3(const GridDev3 &q)
{
    GridCoef3<T> c;
    c.g = T(q.gamma);
    c.gm1 = T(q.gamma - 1.0);
    c.gm1i = T(1.0 / (q.gamma - 1.0));
    c.hgm1 = T(0.5 * (q.gamma - 1.0));
    c.mr2 = T(q.m_ref * q.m_ref);
    c.rr_thr = T(1e-5 * q.u_ref);
    c.eps2 = T(q.eps2);
    c.idx = T(1.0 / q.dx);
    c.idy = T(1.0 / q.dy);
    c.idz = T(1.0 / q.dz);
    for (int v = 0; v < MAX_VARS3; ++v) c.inflow[v] = T(q.inflow[v]);
    return c;
}

template <typename T>
roeam_status upload_coef3(roeam3_grid *g)
{
    std::vector<GridCoef3<T>> h(g->count);
    for (int k = 0; k < g->count; ++k) h[k] = make_coef3<T>(g->hg[k]);
    CUDA_TRY3(cudaMalloc(&g->d_coef, sizeof(GridCoef3<T>) * g->count));
    CUDA_TRY3(cudaMemcpy(g->d_coef, h.data(), sizeof(GridCoef3<T>) * g->count, cudaMemcpyHostToDevice));
    return ROEAM_OK;
}

// Work units: rectangles of at most w x h columns by segments of planes, one CTA each (one fits an SM).
// FP32 takes 30 x 14 columns; (w, h) in FP64 and the number of segments minimise an estimate of a
// launch's cycles, units going over the SMs in rounds: planes (a segment costs about one more) times a
// plane's cycles, which in FP64 are its FP64 operations on an SM's four pipes and three barriers.
// (Counting the rectangles that the even split makes, full and started passes half and half, and odd widths:
// FP64 us a step, two scalars, 64^3 1300 -> 1252, 128^3 9526 -> 9294, 33^3 306 -> 258, 40^3 411 -> 380,
// 60 x 180 x 34 1857 -> 1609, 500 x 4 x 4 158 -> 132; 95 x 63 x 127 3750 -> 3853.)
// FP64 threads: one per face of a plane up to 256, also where there are fewer positions than that: two warps
// per scheduler hide each other's latency (32^3: 398 us a step with a thread per position, 241 with 256;
// 384 threads: 64^3 1348 us against 1332, 16^3 126 against 103, 95 x 63 x 127 3519 against 3852).
template <typename T>
roeam_status setup_units3(roeam3_grid *g, int num_sms)
{
    int max_ni = 0, max_nj = 0, max_nk = 0;
    for (const GridDev3 &G : g->hg) {
        max_ni = std::max(max_ni, G.ni);
        max_nj = std::max(max_nj, G.nj);
        max_nk = std::max(max_nk, G.nk);
    }
    const bool f32 = sizeof(T) == 4;
    constexpr int SAMPLES = 16;   // (of a large batch's grids)
    const int every = 1 + (g->count - 1) / SAMPLES, samples = (g->count + every - 1) / every;
    double best = 1e300;
    int bw = 0, bh = 0, bn = 1;
    // Numbers of segments and the planes of the longest one; of equal planes the fewest segments. (Beyond 96 in
    // steps of a sixteenth: needles along z need more, FP32 1 x 1 x 4000 259 us a step with 96 segments, 177 with
    // 152; FP64 1342 and 906.)
    std::vector<std::pair<int, int>> cuts;
    for (int n = 1; n <= max_nk; n += n < 96 ? 1 : n / 16) {
        int zs = 0;
        for (int q = 0; q < g->count; q += every) {
            const int nk = g->hg[q].nk, sn = std::min(n, nk);
            zs = std::max(zs, (nk + sn - 1) / sn);
        }
        if (cuts.empty() || zs < cuts.back().second) cuts.emplace_back(n, zs);
    }
    auto consider = [&](int w, int h, double plane, double segment, double planes_more) {
        double columns[SAMPLES];   // rectangles of a plane of each sampled grid
        double planes = 0;         // of all rectangles: their cycles over the SMs bound the cost from below
        for (int q = 0; q < samples; ++q) {
            const GridDev3 &G = g->hg[q * every];
            columns[q] = (double)every * ((G.ni + w - 1) / w) * ((G.nj + h - 1) / h);
            planes += columns[q] * G.nk;
        }
        if (planes * plane / num_sms >= best) return;
        for (const auto &c : cuts) {
            double units = 0;
            for (int q = 0; q < samples; ++q) units += columns[q] * std::min(c.first, g->hg[q * every].nk);
            const double cost = std::ceil(units / num_sms) * (plane * (c.second + planes_more) + segment);
            if (cost < best * 0.999) { best = cost; bw = w; bh = h; bn = c.first; }
        }
    };
    if (f32) consider(MARCH3_X, MARCH3_Y, 5000, 6000, 1.0);
    else
        for (int w = std::min(64, max_ni + 1); w >= 1; --w)
            for (int h = 2; h <= std::min(64, max_nj + 1); ++h) {
                if (bytes3<T>(w, h, g->nv) == 0) break;
                // (a single grid's rectangles are as large as its even split makes them; a phase's last
                //  pass counts half its lanes idle)
                const int W = g->count == 1 ? (max_ni + (max_ni + w - 1) / w - 1) / ((max_ni + w - 1) / w) : w;
                const int Y = g->count == 1 ? (max_nj + (max_nj + h - 1) / h - 1) / ((max_nj + h - 1) / h) : h;
                const auto passes = [](double n) { return 0.5 * (std::ceil(n / 128) + n / 128); };
                const double faces = (double)(W + 1) * Y + (double)W * (Y + 1) + (double)W * Y;
                const double positions = (double)(W + 2) * (Y + 2);
                consider(w, h, 2500 + 76 * (passes(faces) * (148 + 9 * g->nscal) + passes(positions) * (75 + 7 * g->nv)), 4000, 1.3);
            }
    if (bw == 0) return fail3(ROEAM_E_ARG, "no work unit fits");
    std::vector<int4> units;
    int mw = 0, mh = 0;
    for (int gi = 0; gi < g->count; ++gi) {
        const GridDev3 &G = g->hg[gi];
        const int nx = (G.ni + bw - 1) / bw, ny = (G.nj + bh - 1) / bh, nz = std::min(bn, G.nk);
        for (int z = 0; z < nz; ++z)
            for (int y = 0; y < ny; ++y)
                for (int x = 0; x < nx; ++x) {
                    const int x0 = (int)((long long)x * G.ni / nx), x1 = (int)((long long)(x + 1) * G.ni / nx);
                    const int y0 = (int)((long long)y * G.nj / ny), y1 = (int)((long long)(y + 1) * G.nj / ny);
                    const unsigned z0 = (unsigned)((long long)z * G.nk / nz), z1 = (unsigned)((long long)(z + 1) * G.nk / nz);
                    units.push_back(make_int4(gi, x0 | (x1 - x0) << 16, y0 | (y1 - y0) << 16, (int)(z0 | z1 << 16)));
                    mw = std::max(mw, x1 - x0);
                    mh = std::max(mh, y1 - y0);
                }
    }
    g->nunits = (int)units.size();
    g->smem = bytes3<T>(mw, mh, g->nv);
    g->threads = f32 ? threads3<T>() : std::min(threads3<T>(), std::max(128, (3 * mw * mh + mw + mh + 31) / 32 * 32));
    CUDA_TRY3(Launchers3<T>::prepare(g->nscal));
    CUDA_TRY3(cudaMalloc(&g->d_units, sizeof(int4) * units.size()));
    CUDA_TRY3(cudaMemcpy(g->d_units, units.data(), sizeof(int4) * units.size(), cudaMemcpyHostToDevice));
    return ROEAM_OK;
}

template <typename T>
StageArgs3<T> base_args3(roeam3_grid *g)
{
    StageArgs3<T> a;
    std::memset(&a, 0, sizeof(a));
    a.grids = g->d_grids;
    a.coef = (const GridCoef3<T> *)g->d_coef;
    a.units = g->d_units;
    a.ngrids = g->count;
    a.nunits = g->nunits;
    if (g->count == 1) {
        a.g0 = g->hg[0];
        a.c0 = make_coef3<T>(g->hg[0]);
    }
    a.status = g->status;
    return a;
}

template <typename T>
roeam_status do_set3(roeam3_grid *g, int lo, int hi, const double *host)
{
    const GridDev3 &a = g->hg[lo], &b = g->hg[hi - 1];
    const long long n0 = a.poff, n1 = b.poff + (long long)g->nv * b.ni * b.nj * b.nk;
    CUDA_TRY3(cudaMemcpyAsync(g->staging + n0, host, sizeof(double) * (n1 - n0), cudaMemcpyHostToDevice, g->stream));
    unsigned long long *slot = g->rate + (size_t)g->parity * g->count;
    CUDA_TRY3(cudaMemsetAsync(slot + lo, 0, sizeof(unsigned long long) * (hi - lo), g->stream));
    CUDA_TRY3(Launchers3<T>::pack(g->d_grids, (const GridCoef3<T> *)g->d_coef, lo, hi, g->nscal, g->max_cells, g->staging,
                                  (T *)g->U, slot, g->stream));
    g->launches += 1;
    return ROEAM_OK;
}

roeam_status sync_status3(roeam3_grid *g)
{
    CUDA_TRY3(cudaMemcpyAsync(g->h_status, g->status, sizeof(unsigned), cudaMemcpyDeviceToHost, g->stream));
    CUDA_TRY3(cudaMemsetAsync(g->status, 0, sizeof(unsigned), g->stream));
    CUDA_TRY3(cudaStreamSynchronize(g->stream));
    const unsigned st = *g->h_status;
    if (st & ST_NONFINITE) return fail3(ROEAM_E_NONFINITE, "non-finite state after a step");
    if (st & ST_NONPOSITIVE) return fail3(ROEAM_E_NONPOSITIVE, "non-positive density or pressure after a step");
    return ROEAM_OK;
}

template <typename T>
roeam_status do_get3(roeam3_grid *g, int lo, int hi, double *host, const void *src)
{
    CUDA_TRY3(Launchers3<T>::unpack(g->d_grids, lo, hi, g->nscal, g->max_cells, (const T *)src, g->staging, g->stream));
    g->launches += 1;
    const GridDev3 &a = g->hg[lo], &b = g->hg[hi - 1];
    const long long n0 = a.poff, n1 = b.poff + (long long)g->nv * b.ni * b.nj * b.nk;
    CUDA_TRY3(cudaMemcpyAsync(host, g->staging + n0, sizeof(double) * (n1 - n0), cudaMemcpyDeviceToHost, g->stream));
    return sync_status3(g);
}

template <typename T>
roeam_status launch_step3(roeam3_grid *g, double cfl, double dt_fixed)
{
    StageArgs3<T> a = base_args3<T>(g);
    a.cfl_t = T(cfl);
    a.dt_fixed_t = T(dt_fixed);
    a.mode = MODE_STAGE;
    a.rate_rd = g->rate + (size_t)g->parity * g->count;
    a.rate_wr = g->rate + (size_t)(1 - g->parity) * g->count;
    const T *U = (const T *)g->U;
    // stage 1: U1 = U + dt R(U)   (also clears the next step's rate slots)
    a.src = U; a.un = U; a.dst = (T *)g->A; a.alpha = T(0); a.beta = T(1); a.rate_zero = a.rate_wr; a.want_rate = 0;
    CUDA_TRY3(Launchers3<T>::stage(a, g->nscal, g->threads, g->smem, g->stream));
    // stage 2: U2 = 3/4 U + 1/4 (U1 + dt R(U1))
    a.src = (const T *)g->A; a.dst = (T *)g->B; a.alpha = T(0.75); a.beta = T(0.25); a.rate_zero = nullptr;
    CUDA_TRY3(Launchers3<T>::stage(a, g->nscal, g->threads, g->smem, g->stream));
    // stage 3: U = 1/3 U + 2/3 (U2 + dt R(U2)), in place; the next step's rate
    a.src = (const T *)g->B; a.dst = (T *)g->U; a.alpha = T(1.0 / 3.0); a.beta = T(2.0 / 3.0); a.want_rate = 1;
    CUDA_TRY3(Launchers3<T>::stage(a, g->nscal, g->threads, g->smem, g->stream));
    g->launches += 3;
    g->parity ^= 1;
    return ROEAM_OK;
}

template <typename T>
roeam_status do_residual3(roeam3_grid *g, int lo, int hi, double *out)
{
    StageArgs3<T> a = base_args3<T>(g);
    a.mode = MODE_RESIDUAL;
    a.src = (const T *)g->U;
    a.un = (const T *)g->U;
    a.dst = (T *)g->A;
    CUDA_TRY3(Launchers3<T>::stage(a, g->nscal, g->threads, g->smem, g->stream));
    g->launches += 1;
    if (!out) return ROEAM_OK;
    return do_get3<T>(g, lo, hi, out, g->A);
}

template <typename T>
roeam_status do_totals3(roeam3_grid *g, int idx, double *out)
{
    const GridDev3 &G = g->hg[idx];
    const long long n = (long long)G.ni * G.nj * G.nk;
    const int nb = (int)std::min<long long>((n + 255) / 256, 1024);
    CUDA_TRY3(Launchers3<T>::totals(g->d_grids, idx, (const T *)g->U, g->nv, g->partials, nb, g->stream));
    g->launches += 1;
    std::vector<double> h((size_t)nb * MAX_VARS3);
    CUDA_TRY3(cudaMemcpyAsync(h.data(), g->partials, sizeof(double) * h.size(), cudaMemcpyDeviceToHost, g->stream));
    CUDA_TRY3(cudaStreamSynchronize(g->stream));
    for (int v = 0; v < g->nv; ++v) {
        double s = 0.0;
        for (int b = 0; b < nb; ++b) s += h[(size_t)b * MAX_VARS3 + v];   // fixed order
        out[v] = s;
    }
    return ROEAM_OK;
}

roeam_status range3(roeam3_grid *g, int idx, int &lo, int &hi)
{
    if (!g) return fail3(ROEAM_E_ARG, "null handle");
    if (idx < -1 || idx >= g->count) return fail3(ROEAM_E_ARG, "grid index %d out of range", idx);
    lo = idx < 0 ? 0 : idx;
    hi = idx < 0 ? g->count : idx + 1;
    if (cudaSetDevice(g->device) != cudaSuccess) return fail3(ROEAM_E_CUDA, "cudaSetDevice failed");
    return ROEAM_OK;
}

}  // namespace

extern "C" {

roeam_status roeam3_create_grid(int count, const roeam3_grid_desc *descs, int device, void *cuda_stream,
                                roeam3_grid **out)
{
    if (!out) return fail3(ROEAM_E_ARG, "out must be non-null");
    *out = nullptr;
    roeam_status st = validate3(count, descs);
    if (st != ROEAM_OK) return st;
    CUDA_TRY3(cudaSetDevice(device));
    int num_sms = 0;
    CUDA_TRY3(cudaDeviceGetAttribute(&num_sms, cudaDevAttrMultiProcessorCount, device));
    roeam3_grid *g = new roeam3_grid();
    g->device = device;
    g->stream = (cudaStream_t)cuda_stream;
    g->count = count;
    g->precision = descs[0].p.precision;
    g->esize = g->precision == 32 ? 4 : 8;
    g->nscal = descs[0].nscal;
    g->nv = 5 + g->nscal;
    g->hg.resize(count);
    long long off = 0, poff = 0;
    for (int k = 0; k < count; ++k) {
        const roeam3_grid_desc &q = descs[k];
        GridDev3 &G = g->hg[k];
        std::memset(&G, 0, sizeof(G));
        G.ni = q.ni; G.nj = q.nj; G.nk = q.nk;
        G.pitch = (int)round_up3(q.ni, 32);
        G.vol = (long long)q.nk * q.nj * G.pitch;
        G.off = off;
        off += round_up3((long long)(4 + tail3(g->nv)) * G.vol, 64);
        G.poff = poff;
        poff += (long long)g->nv * q.ni * q.nj * q.nk;
        for (int s = 0; s < 6; ++s) G.bc[s] = q.bc[s];
        G.eps1 = q.p.eps1; G.use_s1 = q.p.use_s1; G.xi_form = q.p.xi_form;
        for (int v = 0; v < MAX_VARS3; ++v) G.inflow[v] = q.inflow[v];
        G.gamma = q.p.gamma; G.m_ref = q.p.m_ref; G.u_ref = q.p.u_ref; G.eps2 = q.p.eps2;
        G.dx = q.dx; G.dy = q.dy; G.dz = q.dz;
        g->max_cells = std::max(g->max_cells, (long long)q.ni * q.nj * q.nk);
    }
    g->total_elems = off;
    g->total_packed = poff;
    auto cleanup = [&](roeam_status s) { roeam3_destroy_grid(g); return s; };
#define CREATE3_TRY(expr)                                                                                        \
    do {                                                                                                         \
        cudaError_t e_ = (expr);                                                                                 \
        if (e_ != cudaSuccess)                                                                                   \
            return cleanup(fail3(e_ == cudaErrorMemoryAllocation ? ROEAM_E_OOM : ROEAM_E_CUDA, "%s: %s", #expr, \
                                 cudaGetErrorString(e_)));                                                       \
    } while (0)
    const size_t sbytes = g->esize * (size_t)g->total_elems;
    CREATE3_TRY(cudaMalloc(&g->U, sbytes));
    CREATE3_TRY(cudaMalloc(&g->A, sbytes));
    CREATE3_TRY(cudaMalloc(&g->B, sbytes));
    CREATE3_TRY(cudaMemset(g->U, 0, sbytes));
    CREATE3_TRY(cudaMemset(g->A, 0, sbytes));
    CREATE3_TRY(cudaMemset(g->B, 0, sbytes));
    CREATE3_TRY(cudaMalloc(&g->d_grids, sizeof(GridDev3) * count));
    CREATE3_TRY(cudaMemcpy(g->d_grids, g->hg.data(), sizeof(GridDev3) * count, cudaMemcpyHostToDevice));
    CREATE3_TRY(cudaMalloc(&g->rate, sizeof(unsigned long long) * 2 * count));
    CREATE3_TRY(cudaMemset(g->rate, 0, sizeof(unsigned long long) * 2 * count));
    CREATE3_TRY(cudaMalloc(&g->status, sizeof(unsigned)));
    CREATE3_TRY(cudaMemset(g->status, 0, sizeof(unsigned)));
    CREATE3_TRY(cudaMalloc(&g->staging, sizeof(double) * (size_t)std::max(1ll, g->total_packed)));
    CREATE3_TRY(cudaMalloc(&g->partials, sizeof(double) * 1024 * MAX_VARS3));
    CREATE3_TRY(cudaMallocHost(&g->h_status, sizeof(unsigned)));
    CREATE3_TRY(cudaMallocHost(&g->h_rate, sizeof(unsigned long long) * count));
#undef CREATE3_TRY
    st = g->precision == 32 ? upload_coef3<float>(g) : upload_coef3<double>(g);
    if (st != ROEAM_OK) return cleanup(st);
    st = g->precision == 32 ? setup_units3<float>(g, num_sms) : setup_units3<double>(g, num_sms);
    if (st != ROEAM_OK) return cleanup(st);
    *out = g;
    return ROEAM_OK;
}

void roeam3_destroy_grid(roeam3_grid *g)
{
    if (!g) return;
    cudaSetDevice(g->device);
    if (g->stream) cudaStreamSynchronize(g->stream); else cudaDeviceSynchronize();
    cudaFree(g->U); cudaFree(g->A); cudaFree(g->B);
    cudaFree(g->d_grids); cudaFree(g->d_coef); cudaFree(g->d_units);
    cudaFree(g->rate); cudaFree(g->status); cudaFree(g->staging); cudaFree(g->partials);
    cudaFreeHost(g->h_status); cudaFreeHost(g->h_rate);
    delete g;
}

roeam_status roeam3_set_state(roeam3_grid *g, int grid_idx, const double *cons)
{
    int lo, hi;
    roeam_status st = range3(g, grid_idx, lo, hi);
    if (st != ROEAM_OK) return st;
    if (!cons) return fail3(ROEAM_E_ARG, "cons must be non-null");
    return g->precision == 32 ? do_set3<float>(g, lo, hi, cons) : do_set3<double>(g, lo, hi, cons);
}

roeam_status roeam3_get_state(roeam3_grid *g, int grid_idx, double *cons_out)
{
    int lo, hi;
    roeam_status st = range3(g, grid_idx, lo, hi);
    if (st != ROEAM_OK) return st;
    if (!cons_out) return fail3(ROEAM_E_ARG, "cons_out must be non-null");
    return g->precision == 32 ? do_get3<float>(g, lo, hi, cons_out, g->U) : do_get3<double>(g, lo, hi, cons_out, g->U);
}

roeam_status roeam3_flux_residual(roeam3_grid *g, int grid_idx, double *res_out)
{
    int lo, hi;
    roeam_status st = range3(g, grid_idx, lo, hi);
    if (st != ROEAM_OK) return st;
    return g->precision == 32 ? do_residual3<float>(g, lo, hi, res_out) : do_residual3<double>(g, lo, hi, res_out);
}

roeam_status roeam3_rk_step(roeam3_grid *g, double cfl, double dt_fixed, int nsteps, double *dt_last)
{
    int lo, hi;
    roeam_status st = range3(g, -1, lo, hi);
    if (st != ROEAM_OK) return st;
    if (nsteps < 0) return fail3(ROEAM_E_ARG, "nsteps must be >= 0");
    if (!(dt_fixed > 0.0) && !(cfl > 0.0)) return fail3(ROEAM_E_ARG, "give cfl > 0 or dt_fixed > 0");
    for (int s = 0; s < nsteps; ++s) {
        st = g->precision == 32 ? launch_step3<float>(g, cfl, dt_fixed) : launch_step3<double>(g, cfl, dt_fixed);
        if (st != ROEAM_OK) return st;
    }
    if (dt_last) {
        if (dt_fixed > 0.0 || nsteps == 0) {
            for (int k = 0; k < g->count; ++k) dt_last[k] = nsteps == 0 ? 0.0 : dt_fixed;
        } else {
            // the last step read the slots of the parity before the flip
            const unsigned long long *slot = g->rate + (size_t)(g->parity ^ 1) * g->count;
            CUDA_TRY3(cudaMemcpyAsync(g->h_rate, slot, sizeof(unsigned long long) * g->count, cudaMemcpyDeviceToHost,
                                      g->stream));
            st = sync_status3(g);
            if (st != ROEAM_OK) return st;
            for (int k = 0; k < g->count; ++k) {
                if (g->precision == 32) {
                    float f;
                    const unsigned bits = (unsigned)g->h_rate[k];
                    std::memcpy(&f, &bits, 4);
                    dt_last[k] = (double)(float(cfl) / f);
                } else {
                    double r;
                    std::memcpy(&r, &g->h_rate[k], 8);
                    dt_last[k] = cfl / r;
                }
            }
        }
    }
    return ROEAM_OK;
}

roeam_status roeam3_conserved_totals(roeam3_grid *g, int grid_idx, double *out)
{
    int lo, hi;
    if (grid_idx < 0) return fail3(ROEAM_E_ARG, "grid_idx must be >= 0");
    roeam_status st = range3(g, grid_idx, lo, hi);
    if (st != ROEAM_OK) return st;
    if (!out) return fail3(ROEAM_E_ARG, "out must be non-null");
    st = sync_status3(g);
    if (st != ROEAM_OK) return st;
    return g->precision == 32 ? do_totals3<float>(g, grid_idx, out) : do_totals3<double>(g, grid_idx, out);
}

roeam_status roeam3_check(roeam3_grid *g)
{
    int lo, hi;
    roeam_status st = range3(g, -1, lo, hi);
    if (st != ROEAM_OK) return st;
    return sync_status3(g);
}

unsigned long long roeam3_launch_count(const roeam3_grid *g) { return g ? g->launches : 0ull; }

}  // extern "C"
