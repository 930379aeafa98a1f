// roeam3_internal.h — device-side descriptors and launch entry points of the 3D path (Cartesian
// grids with passive scalars), shared by roeam3_api.cu and the 3D kernel translation units.
// Not part of the public ABI.
#pragma once

#include "roeam_internal.h"

namespace roeam {

constexpr int MAX_SCALARS = 3;
constexpr int MAX_VARS3 = 5 + MAX_SCALARS;

// Per-grid descriptor of a 3D grid, resident in device memory.
struct GridDev3 {
    long long off;     // element offset of this grid in the state buffers: quads (rho, rho u, rho v, rho w)
                       // of its cells at off + 4 c, c = (k nj + j) pitch + i, then their tails
                       // (rho E, scalars; tail3(nv) values) at off + 4 vol + tail3(nv) c
    long long vol;     // cells held (nk * nj * pitch)
    long long poff;    // element offset of this grid in the packed host layout [nv][nk][nj][ni]
    int ni, nj, nk, pitch;
    int bc[6];         // W, E, S, N, B, T
    int eps1, use_s1, xi_form, pad_;
    double inflow[MAX_VARS3];   // rho, u, v, w, p, k_1..
    double gamma, m_ref, u_ref, eps2;
    double dx, dy, dz;
};

// Per-grid constants in the working precision.
template <typename T>
struct GridCoef3 {
    T g, gm1, gm1i, hgm1, mr2, rr_thr, eps2;
    T idx, idy, idz;             // 1/dx, 1/dy, 1/dz
    T inflow[MAX_VARS3];
};

// Values beyond the first four of a cell of nv variables (three are stored as four, so that a tail is
// one aligned access).
__host__ __device__ constexpr int tail3(int nv) { return nv - 4 == 3 ? 4 : nv - 4; }

// Threads per CTA of the 3D stage kernel (FP64: at most), and the cells of an FP32 unit: 32 columns by a
// row per warp, less the halo.
template <typename T> __host__ __device__ constexpr int threads3() { return sizeof(T) == 4 ? 512 : 256; }
constexpr int MARCH3_X = 30, MARCH3_Y = threads3<float>() / 32 - 2;

// Shared memory of the 3D stage kernel for a rectangle of w x h cells, or 0 if it does not fit.
// FP32 (whatever the rectangle): per thread two buffers of exchanged fields (9 + scalars cell values, 3
// ratios, nv fluxes), four raw cells and two of U^n. FP64: a record of rec3 values per position (cells and
// a halo of one), at most two positions per thread.
__host__ __device__ constexpr int rec3(int nv) { return ((56 + 12 * tail3(nv) + 6 + 3) / 4 | 1) * 4; }
template <typename T> inline size_t bytes3(int w, int h, int nv)
{
    if (sizeof(T) == 4)
        return w <= MARCH3_X && h <= MARCH3_Y ? sizeof(T) * threads3<T>() * (2 * (4 + nv + 3 + nv) + 6 * (4 + tail3(nv))) : 0;
    const size_t b = sizeof(T) * (size_t)(w + 2) * (h + 2) * rec3(nv);
    return b <= TILE_SMEM_MAX && (w + 2) * (h + 2) <= 2 * threads3<T>() ? b : 0;
}

template <typename T>
struct StageArgs3 {
    const GridDev3 *grids;
    const GridCoef3<T> *coef;
    const int4 *units;       // (grid, first column | width << 16, first row | height << 16, k0 | k1 << 16)
    int ngrids, nunits;
    const T *src, *un;
    T *dst;
    T alpha, beta;
    int mode;                // MODE_STAGE or MODE_RESIDUAL
    int want_rate;
    const unsigned long long *rate_rd;
    unsigned long long *rate_wr, *rate_zero;
    T cfl_t, dt_fixed_t;
    unsigned *status;
    GridDev3 g0;             // the only grid's descriptor and constants
    GridCoef3<T> c0;
};

template <typename T>
struct Launchers3 {
    static cudaError_t stage(const StageArgs3<T> &a, int nscal, int threads, size_t smem, cudaStream_t s);
    static cudaError_t prepare(int nscal);   // lets the stage kernel take the shared memory it may ask for
    // Packed float64 host layout <-> state; the pack raises rate[g] (zeroed by the caller).
    static cudaError_t pack(const GridDev3 *grids, const GridCoef3<T> *coef, int g_lo, int g_hi, int nscal,
                            long long max_cells, const double *packed, T *U, unsigned long long *rate, cudaStream_t s);
    static cudaError_t unpack(const GridDev3 *grids, int g_lo, int g_hi, int nscal, long long max_cells, const T *U,
                              double *packed, cudaStream_t s);
    static cudaError_t totals(const GridDev3 *grids, int g, const T *U, int nv, double *partials, int nblocks,
                              cudaStream_t s);
};

}  // namespace roeam
