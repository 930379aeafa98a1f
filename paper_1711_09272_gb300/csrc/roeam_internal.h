// roeam_internal.h — device-side descriptors and launch entry points shared by the
// library's host code (roeam_api.cu) and its kernel translation units (roeam_k32.cu,
// roeam_k64.cu and their ablation-variant companions). Not part of the public ABI.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

namespace roeam {

constexpr int BC_PERIODIC = 0, BC_WALL = 1, BC_INFLOW = 2, BC_OUTFLOW = 3, BC_EXCHANGE = 4;

// Status bits raised by kernels (read back by the host at synchronising calls).
constexpr unsigned ST_NONPOSITIVE = 1u, ST_NONFINITE = 2u;
constexpr unsigned ST_BOUNDS = 4u;   // an index outside its buffer (bounds-checked debug builds only)

// Per-grid descriptor, resident in device memory, read-only in kernels.
struct GridDev {
    long long off;    // element offset of this grid's cell (0, 0) in the state buffers: cell (i, j)
                      // holds its four values (rho, rho u, rho v, rho E) at off + 4 (j pitch + i)
    long long plane;  // cells held (nj * pitch; (nj + 4) * pitch with an EXCHANGE side, which also
                      // keeps the ghost rows j = -2, -1, nj, nj+1)
    long long voff;   // element offset of this grid's vertex displacement planes (-1: Cartesian)
    long long soff;   // byte offset of this grid's solid mask (-1: none)
    long long poff;   // element offset of this grid in the packed host layout [4][nj][ni]
    int ni, nj, pitch, vpitch;
    int ntx, nty, tile_base, ntiles;
    int bc[4];        // W, E, S, N
    int limiter;      // 1 minmod, 2 van Leer (MUSCL kernels)
    int eps1, use_s1, xi_form;
    int scheme, dup_mode, ufix, xi_roe;   // ablation variants (0, 0, 1, 0: Roe-AM)
    double inflow[4]; // rho, u, v, p
    double gamma, m_ref, u_ref, eps2;
    double harten;    // classical Roe: eps_lambda of the entropy fix (0: none)
    double dx, dy;    // Cartesian spacings / reference-grid spacings of a curvilinear grid
    double nfluid;    // number of fluid cells
};

enum Mode { MODE_STAGE = 0, MODE_RESIDUAL = 1, MODE_NORM = 2 };

// Per-grid constants in the working precision, computed once on the host so that the
// FP32 kernels execute no FP64 arithmetic on their hot path.
template <typename T>
struct GridCoef {
    T g, gm1, gm1i, hgm1, mr2, rr_thr, eps2;   // gamma, gamma-1, 1/(gamma-1), (gamma-1)/2, M_ref^2, 1e-5 U_ref, eps2
    T dx, dy, V, Vi;                     // spacings (reference spacings if curvilinear), dx*dy, 1/(dx*dy)
    T idx, idy;                          // 1/dx, 1/dy (Cartesian)
    T inflow[4];                         // rho, u, v, p of INFLOW sides
    T harten;                            // classical Roe: eps_lambda (0: no entropy fix)
};

template <typename T>
struct StageArgs {
    const GridDev *grids;
    const GridCoef<T> *coef;
    const int4 *units;      // work units: (grid, column of lane 0, first row, end row)
    int ngrids;
    int tile_lo, tile_hi;   // work units [tile_lo, tile_hi) of the batch processed by this launch
    const T *src;           // U^(k): the state whose residual is evaluated (halo source)
    const T *un;            // U^n for the stage combination
    T *dst;                 // stage output, or the residual in MODE_RESIDUAL
    long long dst_shift;    // grid g's output starts at dst + (G.off - dst_shift) (0: the state layout)
    const T *vdx, *vdy;     // vertex displacement planes (curvilinear grids)
    const uint8_t *solid;   // solid masks
    T alpha, beta;          // dst = alpha * U^n + beta * (U^(k) + dt R(U^(k)))
    int mode;
    int want_rate;          // write each grid's max signal-speed rate of dst into rate_wr
    const unsigned long long *rate_rd;  // per-grid max rate of U^n (working-precision bits)
    unsigned long long *rate_wr;        // per-grid max rate of the stage output
    unsigned long long *rate_zero;      // per-grid slots to reset (the next step's rate_wr), may be null
    double cfl, dt_fixed;
    T cfl_t, dt_fixed_t;    // the same in the working precision
    unsigned *status;
    double *partials;       // MODE_NORM: gridDim.x * 8 (sum R^2 [4], max |R| [4])
    // Dynamic unit scheduling (null: static round robin): work[0] counts the units claimed past
    // each warp's first, work[1] the warps that have finished; the last warp to finish resets
    // both, so that the next launch on the handle's stream starts from zero.
    unsigned *work;
#ifdef ROEAM_DEBUG
    // buffer sizes (elements of src, un and dst, of each vertex plane buffer; bytes of
    // the solid masks), read by the bounds checks of debug builds
    long long n_state, n_un, n_dst, n_vert, n_solid;
#endif
};

// Work-unit shapes of the stage kernel: a warp sweeps a strip tx = 32 lanes wide (2H of
// them halo) over ty rows; nt threads per CTA. The autotuner picks among these.
// One warp per CTA: registers are then allocated warp by warp, so every 8 registers saved
// per thread buys another resident warp.
#ifndef STAGE_THREADS_DEF
#define STAGE_THREADS_DEF 32
#endif
constexpr int STAGE_THREADS = STAGE_THREADS_DEF;
// Resident CTAs per SM the compiler is asked to fit (register budget): 20 holds the FP32 Cartesian
// kernels to 96 registers, which they fit with no spill to speak of since the rows in flight and row
// j - 2 left the registers (512-grid batch, 8 steps: 16 warps per SM 8350 us, 20 warps 7927 us; 96-grid
// van Leer batch 2351 and 2226 us). The curvilinear FP32 variants are held to 128 registers (16 warps
// per SM; at 96 they spill 16 to 80 bytes, and the 4096^2 warped step takes 6957 us against 6514);
// FP64 and the ablation variants are left to the compiler.
#ifndef STAGE_MIN_BLOCKS_CART
#define STAGE_MIN_BLOCKS_CART 20
#endif
#ifndef STAGE_MIN_BLOCKS_CURV
#define STAGE_MIN_BLOCKS_CURV 16
#endif
template <typename T, bool MUSCL, bool CURV, bool ABL = false>
constexpr int stage_min_blocks()
{
    return (sizeof(T) != 4 || ABL) ? 1 : (!CURV ? STAGE_MIN_BLOCKS_CART : STAGE_MIN_BLOCKS_CURV);
}
// dyn: dynamic unit scheduling (warps claim units from a counter after
// their first; 0 = static round robin over the unit table).
struct TileCfg { int tx, ty, nt, dyn; };
constexpr int NUM_TILE_CFGS = 10;
constexpr TileCfg TILE_CFGS[NUM_TILE_CFGS] = {
    {32, 32, STAGE_THREADS, 1}, {32, 64, STAGE_THREADS, 1}, {32, 16, STAGE_THREADS, 1}, {32, 128, STAGE_THREADS, 1},
    {32, 256, STAGE_THREADS, 1}, {32, 32, STAGE_THREADS, 0}, {32, 64, STAGE_THREADS, 0}, {32, 16, STAGE_THREADS, 0},
    {32, 128, STAGE_THREADS, 0}, {32, 256, STAGE_THREADS, 0}};

// Stage-kernel families: no walls anywhere in the batch; some WALL side or solid cells; some
// grid uses an ablation variant of the flux (every face on the scalar path).
enum StageKind { KIND_PLAIN = 0, KIND_WALLS = 1, KIND_ABLATION = 2 };

// What a pack needs to take the time-step rate of the state it writes: the grids' coefficients,
// vertex displacements and solid masks, and the rate slots it raises with atomicMax.
template <typename T> struct RateOut {
    const GridCoef<T> *coef = nullptr;
    const T *vdx = nullptr, *vdy = nullptr;
    const uint8_t *solid = nullptr;
    unsigned long long *rate = nullptr;
    unsigned long long *rate_zero = nullptr;   // slots to reset (the next step's output), may be null
    int curv = 0;
};

template <typename T>
struct Launchers {
    // Fused face-flux / residual / stage kernel over tiles [tile_lo, tile_hi).
    static cudaError_t stage(const StageArgs<T> &a, int muscl, int curv, int kind, int nblocks, cudaStream_t s);
    // Largest resident CTAs per SM of a stage-kernel variant (for persistent launches).
    static int stage_occupancy(int muscl, int curv, int kind);
    // Packed float64 [4][nj][ni] per grid <-> the state's pitched working-precision cells.
    // (pack reads grid g at packed + G.poff - p_shift; the host-side layout in float64 or float;
    //  with ro it also writes the packed state's rate into ro->rate[g], zeroed by the caller)
    static cudaError_t pack(const GridDev *grids, int g_lo, int g_hi, int max_cells, const double *packed, T *U,
                            cudaStream_t s, long long p_shift = 0, const RateOut<T> *ro = nullptr);
    static cudaError_t pack(const GridDev *grids, int g_lo, int g_hi, int max_cells, const float *packed, T *U,
                            cudaStream_t s, long long p_shift = 0, const RateOut<T> *ro = nullptr);
    // (unpack reads grid g at U + G.off - u_shift and writes it at packed + G.poff - p_shift)
    static cudaError_t unpack(const GridDev *grids, int g_lo, int g_hi, int max_cells, const T *U, double *packed,
                              cudaStream_t s, long long u_shift = 0, long long p_shift = 0);
    static cudaError_t unpack(const GridDev *grids, int g_lo, int g_hi, int max_cells, const T *U, float *packed,
                              cudaStream_t s, long long u_shift = 0, long long p_shift = 0);
    // Two rows of a grid's state (from row r0) <-> rows, device memory laid out [4][2][ni].
    static cudaError_t rows(T *U, long long off, int pitch, int ni, int r0, T *rows, bool set, cudaStream_t s);
    // FP64 block partials of sum V*U over the fluid cells of one grid (gridDim.x * 4 doubles).
    static cudaError_t totals(const GridDev *grids, const GridCoef<T> *coef, int g, const T *U, const T *vdx,
                              const T *vdy, const uint8_t *solid, double *partials, int nblocks, int curv,
                              cudaStream_t s);
};

// ---- tile kernels (roeam_tile.cuh): a whole step per launch in FP32, a stage per launch in FP64
template <typename T> __host__ __device__ constexpr int tile_stages() { return sizeof(T) == 4 ? 3 : 1; }
template <typename T> __host__ __device__ constexpr int tile_threads() { return sizeof(T) == 4 ? 512 : 256; }
constexpr size_t TILE_SMEM_MAX = 226 * 1024;   // dynamic shared memory a tile may take (227 KB per CTA in all)

template <typename T>
struct TileArgs {
    GridDev g0;             // the only grid's descriptor and constants, and its rectangles: nx a row,
    GridCoef<T> c0;         // `wide` x `high` cells, the first `wider` columns and `higher` rows of them one more
    int nx, wide, wider, high, higher;
    const GridDev *grids;
    const GridCoef<T> *coef;
    const int4 *tiles;      // (grid, first column, first row, width | height << 16)
    int ngrids;
    const T *src, *un;      // U^(k) and U^n (STAGES = 3: both U^n)
    T *dst;
    const T *vdx, *vdy;
    const uint8_t *solid;
    T alpha, beta;          // STAGES = 1
    int residual;           // STAGES = 1: write the residual of `src` to `dst` instead of a stage's result,
    long long dst_shift;    // cell x of it at dst + x - dst_shift
    int want_rate;
    const unsigned long long *rate_rd;
    unsigned long long *rate_wr, *rate_zero;
    T cfl_t, dt_fixed_t;
    unsigned *status;
#ifdef ROEAM_DEBUG
    long long n_state, n_un, n_dst, n_vert, n_solid;   // buffer sizes, read by the bounds checks of debug builds
#endif
};

// Shared memory of a tile of W x R positions (the rectangle and its halo): quads of T per position
// (U, primitives, two fluxes, derived quantities or two slopes, U^n or U^(1) and U^(2)), the Eq. 97 ratios (one row
// more: the pair list's unused faces past the last row read it), vertices, column and row maps,
// flags.
template <typename T> inline size_t tile_bytes(int W, int R, bool muscl, bool curv, bool walls, int stages)
{
    const size_t P = (size_t)W * R;
    return sizeof(T) * (4 * P * (4 + (muscl ? 2 : 1) + (stages == 3 ? (walls ? 2 : 1) : 0)) + 2 * (P + W + 2) +
                        (curv ? 2 * (size_t)(W + 1) * (R + 1) : 0)) +
           sizeof(int) * 2 * (W + 1 + R + 1) + (walls ? (P + 15) / 16 * 16 : 0);
}

template <typename T>
struct TileLaunchers {
    static cudaError_t step(const TileArgs<T> &a, int muscl, int curv, int walls, int ntiles, int threads, size_t smem,
                            cudaStream_t s);
    static cudaError_t prepare(int muscl, int curv, int walls, bool one);   // (one: a single grid)
    // FP64 sums of squares [k] and maxima of magnitudes [4 + k] over grid idx of a residual R, one row of
    // eight per block.
    static cudaError_t norms(const GridDev *grids, int idx, const T *R, double *partials, int nblocks, cudaStream_t s);
};

// The ablation-variant stage kernels, instantiated in their own translation units.
template <typename T>
struct AblationLaunchers {
    static cudaError_t stage(const StageArgs<T> &a, int muscl, int curv, int nblocks, cudaStream_t s);
    static int stage_occupancy(int muscl, int curv);
};

// The kernels' reciprocal, rsqrt and sqrt on n device values (n rows of 6 doubles; test hook).
cudaError_t launch_math_check(int n, const double *x, double *out, cudaStream_t s);

// Sets the thread's roeam_last_error() message and returns `status` (host).
int record_error(int status, const char *msg);

// Fixed-order reduction of nblocks x 8 norm partials into out[8] (sum[4], max[4]).
cudaError_t launch_reduce_partials(const double *partials, int nblocks, int width, double *out, cudaStream_t s);

}  // namespace roeam
