// roeam_tile.cuh — sm_103a kernels of the Roe-AM step for grids that the warp strips of
// stage_kernel cannot fill the chip with, and for FP64.
//
// One CTA holds a rectangle of cells with its halo in shared memory and runs four phases per
// Runge-Kutta stage, a block barrier between them: primitives and derived quantities per cell
// (ghost cells from the boundary conditions), Eq. 97 ratios and limited slopes per cell, fluxes per
// face, update per cell. Every phase spreads its work over all threads, so a stage takes one flux
// evaluation's latency per few hundred faces instead of the strip's row after row.
//
// STAGES = 3 (FP32): the whole SSP-RK3 step in one launch. The CTA loads a halo of 3 H cells
// (H = 1 at first order, 2 with MUSCL) and updates a margin of 2 H, H and 0 cells around its
// rectangle in the three stages, recomputing what its neighbours also compute, so no CTA waits
// for another and U^(1), U^(2) never leave shared memory. What bounds a step is then latency and, on
// the larger grids, instruction issue: of 7 us for a 16 x 6 rectangle, 0.8 are descriptors and maps,
// 0.5 the load, and a stage takes 0.2 ratios, 0.7 fluxes, 0.5 update. The strips take 11 to 29 us a step
// on these grids whatever their size (three launches of a few serial row iterations each). Strips and
// tiles, us a step: 256^2 van Leer 19.0, 11.6, 400^2 corner 25.6, 18.4, 800 x 20 duct 18.1, 7.1 (7.9 with
// ghost cells in a phase of their own).
// STAGES = 1 (FP64): one stage per launch. FP64 kernels are bound by the FP64 pipe, so recomputed
// halos cost time; the phases evaluate each face once per CTA and keep all lanes busy where the
// strips of a small grid evaluated three rows of faces per two rows of cells. The fluxes take 75 % of
// a stage and run at the pipe's rate (133 operations per first-order face, about 190 reconstructed).
// Strips and tiles, us a step: 64^2 134, 32, 256^2 first order 267, 158, van Leer 483, 234, 1024^2 2604, 2224.
//
// In directions that are not periodic the halo ends H cells outside the grid; in periodic ones the
// halo cells are cells of the other side, which evolve like their originals.
#pragma once

#include "roeam_kernels.cuh"

namespace roeam {

// Bounds-checked debug builds: n elements at index i of a buffer of `size`, or ST_BOUNDS and no access.
#ifdef ROEAM_DEBUG
__device__ __forceinline__ bool tile_ok(long long i, int n, long long size, unsigned *status)
{
    if (i >= 0 && i + n <= size) return true;
    atomicOr(status, ST_BOUNDS);
    return false;
}
#define TILE_OK(i, n, size) tile_ok((i), (n), a.size, a.status)
#else
#define TILE_OK(i, n, size) true
#endif

template <bool ONE, typename T> __device__ __forceinline__ const GridDev &tile_grid(const TileArgs<T> &a, int g)
{
    if constexpr (ONE) return a.g0;
    else return a.grids[g];
}
template <bool ONE, typename T> __device__ __forceinline__ decltype(auto) tile_coef(const TileArgs<T> &a, int g)
{
    if constexpr (ONE) return (a.c0);
    else return GridCoef<T>(a.coef[g]);
}
template <bool B> struct Flag { static constexpr bool value = B; };

// ONE: a single grid. Its descriptor, its constants (FP32) and its rectangles are kernel arguments, so that
// the kernel does not begin with a chain of loads and holds none of them in registers: 256^2 Gresho
// vortex, 50 steps, 607 -> 577 us, 800 x 20 duct, 64 steps, 479 -> 462. (FP64 constants as operands from
// the constant bank: 64^2 vortex 688 -> 691, from registers 687.)
template <typename T, bool MUSCL, bool CURV, bool WALLS, int STAGES, bool ONE>
__global__ void __launch_bounds__(tile_threads<T>()) tile_kernel(const __grid_constant__ TileArgs<T> a)
{
    constexpr int H = MUSCL ? 2 : 1;
    constexpr int E = H * STAGES;
    constexpr bool PAIRS = sizeof(T) == 4;   // FP32 evaluates a cell's west and south faces as one packed pair
    pdl_trigger();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ T red[tile_threads<T>() / 32];

    int4 tile;
    if constexpr (ONE) {
        const int y = (int)blockIdx.x / a.nx, x = (int)blockIdx.x - y * a.nx;
        tile = make_int4(0, x * a.wide + min(x, a.wider), y * a.high + min(y, a.higher),
                         (a.wide + (x < a.wider)) | (a.high + (y < a.higher)) << 16);
    } else {
        tile = __ldg(a.tiles + blockIdx.x);
    }
    const int g = tile.x;
    const int x0 = tile.y, y0 = tile.z, w = tile.w & 0xffff, h = tile.w >> 16;
    const GridDev &G = tile_grid<ONE>(a, g);
    const GridCoef<T> &K = tile_coef<ONE && sizeof(T) == 4>(a, g);
    const int ni = G.ni, nj = G.nj, pitch = G.pitch;
    const int bcW = G.bc[0], bcE = G.bc[1], bcS = G.bc[2], bcN = G.bc[3];
    const bool perx = bcW == BC_PERIODIC, pery = bcS == BC_PERIODIC;
    const bool use_s1 = G.use_s1 != 0, vanleer = G.limiter == 2;
    const int eps1 = G.eps1, xi_form = G.xi_form;
    const int W = w + 2 * E, R = h + 2 * E, P = W * R;   // positions: column c is ix0 + c, row r is jy0 + r
    const int ix0 = x0 - E, jy0 = y0 - E;
    // ghost cells among the positions
    const bool edge = (!perx && (ix0 < 0 || ix0 + W > ni)) || (!pery && (jy0 < 0 || jy0 + R > nj));

    T *const U = reinterpret_cast<T *>(smem_raw);
    T *const A1 = U + 4 * P;
    T *const FX = A1 + 4 * P, *const FY = FX + 4 * P;
    T *const A2 = FY + 4 * P;                       // derived quantities, or x-slopes
    T *const SY = A2 + 4 * P;                       // y-slopes (MUSCL)
    T *const V = A2 + (MUSCL ? 8 : 4) * P;          // STAGES = 3: U^n; with walls U^(1) and U^(2), U staying U^n
    T *const PP = V + (STAGES == 3 ? (WALLS ? 8 : 4) : 0) * P;   // Eq. 97 ratios of the west and south faces
    T *const VV = PP + 2 * (P + W + 2);                       // vertex displacements (CURV): (W + 1) x (R + 1) pairs
    int *const CM = reinterpret_cast<int *>(VV + (CURV ? 2 * (W + 1) * (R + 1) : 0));   // columns, then rows: see below
    int *const RM = CM + 2 * (W + 1);
    uint8_t *const FL = reinterpret_cast<uint8_t *>(RM + 2 * (R + 1));
    const int tid = threadIdx.x, nt = blockDim.x;

    // The margins of the stages: stage s updates columns [lox, hix) and rows [loy, hiy) (clipped to
    // the grid in directions that are not periodic).
    auto margin = [&](int s, int &lox, int &hix, int &loy, int &hiy) {
        const int e = E - H * (s + 1);
        lox = perx ? E - e : max(E - e, -ix0); hix = perx ? E + w + e : min(E + w + e, ni - ix0);
        loy = pery ? E - e : max(E - e, -jy0); hiy = pery ? E + h + e : min(E + h + e, nj - jy0);
    };
    // Per column (and row): [0] the grid column its cells are loaded from (-1: none, more than H cells
    // outside the grid), or the vertex column; [1] the position its cells' values come from (its own but
    // for ghost cells) and their kind (resolve_index) in bits 16 and up. Divisions happen here once, not per position and phase: `recip` holds
    // 2^32 / n + 1 for the width n of every rectangle that a phase covers.
    __shared__ unsigned recip[3 * STAGES + 2];
    if (tid < 3 * STAGES + 2) {
        int n = tid == 3 * STAGES ? W + 1 : W;
        if (tid < 3 * STAGES) {
            int lox, hix, loy, hiy;
            margin(tid / 3, lox, hix, loy, hiy);
            n = hix - lox + 2 - tid % 3;   // ratios, face pairs (or west faces), cells
        }
        recip[tid] = 0xffffffffu / (unsigned)n + 1u;
    }
    for (int q = tid; q < W + 1 + R + 1; q += nt) {
        const bool col = q < W + 1;
        const int x = col ? q : q - (W + 1), v = (col ? ix0 : jy0) + x, n = col ? ni : nj, o = col ? ix0 : jy0;
        const bool per = col ? perx : pery;
        int src = v, from = x;
        if (per) { src = v % n; src = src < 0 ? src + n : src; }
        else if (v < 0 || v >= n) {
            int kind;
            src = resolve_index(v, n, col ? bcW : bcS, col ? bcE : bcN, kind);
            from = ((src - o) & 0xffff) | kind << 16;
            if (v < -H || v >= n + H) src = -1;
        }
        (col ? CM : RM)[2 * x] = src;
        (col ? CM : RM)[2 * x + 1] = from;
    }
    __syncthreads();

    // every position of the rectangle [c0, c1) x [r0, r1), spread over the threads; m = recip of its width
    auto over = [&](unsigned m, int c0, int c1, int r0, int r1, auto &&body) {
        const int wd = c1 - c0, n = wd * (r1 - r0);
#pragma unroll 1
        for (int idx = tid; idx < n; idx += nt) {
            const int q = wd == 1 ? idx : (int)__umulhi((unsigned)idx, m);   // idx / wd (idx wd < 2^32)
            body(c0 + idx - q * wd, r0 + q);
        }
    };

    // vertices do not depend on the launches before this one
    if constexpr (CURV)
        over(recip[3 * STAGES], 0, W + 1, 0, R + 1, [&](int c, int r) {
            // (a periodic seam's last vertex column repeats the first)
            int i = ix0 + c, j = jy0 + r;
            i = perx && (i < 0 || i > ni) ? CM[2 * c] : clampi(i, 0, ni);
            j = pery && (j < 0 || j > nj) ? RM[2 * r] : clampi(j, 0, nj);
            const long long b = G.voff + (long long)j * G.vpitch + i;
            if (TILE_OK(b, 1, n_vert)) {
                const unsigned d = (unsigned)__cvta_generic_to_shared(VV + 2 * (r * (W + 1) + c));
                copy_word(d, a.vdx + b);
                copy_word(d + (unsigned)sizeof(T), a.vdy + b);
            }
        });
    auto vtx = [&](int c, int r, T &x, T &y) { x = VV[2 * (r * (W + 1) + c)]; y = VV[2 * (r * (W + 1) + c) + 1]; };
    // unit normals and lengths of the west face and the south face of position (c, r)
    auto geom_x = [&](int c, int r, T &nx, T &ny, T &len) {
        if constexpr (CURV) {
            T xa, ya, xb, yb;
            vtx(c, r, xa, ya); vtx(c, r + 1, xb, yb);
            const T sx = K.dy + (yb - ya), sy = -(xb - xa);
            unit_normal(sx, sy, nx, ny, len);
        } else { nx = T(1); ny = T(0); len = T(2); }   // (the residual applies the Cartesian lengths)
    };
    auto geom_y = [&](int c, int r, T &nx, T &ny, T &len) {
        if constexpr (CURV) {
            T xa, ya, xb, yb;
            vtx(c, r, xa, ya); vtx(c + 1, r, xb, yb);
            const T sx = -(yb - ya), sy = K.dx + (xb - xa);
            unit_normal(sx, sy, nx, ny, len);
        } else { nx = T(0); ny = T(1); len = T(2); }
    };

    // everything from here on may depend on the launch before this one
    pdl_wait();
    if (a.rate_zero && blockIdx.x == 0)
        for (int q = tid; q < a.ngrids; q += nt) a.rate_zero[q] = 0ull;
    {
        const unsigned dst = (unsigned)__cvta_generic_to_shared(U);
        over(recip[3 * STAGES + 1], 0, W, 0, R, [&](int c, int r) {
            const int i = CM[2 * c], j = RM[2 * r];
            const long long x = G.off + 4 * ((long long)j * pitch + i);
            if ((i | j) >= 0 && TILE_OK(x, 4, n_state))
                copy_cell(dst + (unsigned)((r * W + c) * 4 * (int)sizeof(T)), a.src + x);
        });
        copies_commit();
    }
    if constexpr (WALLS) {
        const unsigned mw = recip[3 * STAGES + 1];
        const bool mask = G.soff >= 0;
#pragma unroll 4
        for (int at = tid; at < P; at += nt) {
            const int r = (int)__umulhi((unsigned)at, mw), c = at - r * W;
            const int i = CM[2 * c], j = RM[2 * r], kx = CM[2 * c + 1] >> 16, ky = RM[2 * r + 1] >> 16;
            uint8_t f = 0;
            const long long x = G.soff + (long long)j * ni + i;
            if (mask && (i | j) >= 0 && kx != 2 && ky != 2 && TILE_OK(x, 1, n_solid)) f = __ldg(a.solid + x) & 1;
            if ((kx == 1 || ky == 1) && kx != 2) f |= 2;
            FL[at] = f;
        }
    }
    // Primitives (and, at first order, the derived face quantities) of a cell from its state.
    auto prims = [&](const T raw[4], WC<T> &q) {
        const T ri = rcp(raw[0]);
        q.r = raw[0]; q.u = raw[1] * ri; q.v = raw[2] * ri;
        q.p = K.gm1 * vfnma(T(0.5) * raw[0], vfma(q.u, q.u, q.v * q.v), raw[3]);
    };
    auto put_cell = [&](int at, WC<T> &q) {
        const T a1[4] = {q.r, q.u, q.v, q.p};
        st_cell(A1 + 4 * at, a1);
        if constexpr (!MUSCL) {
            derive<T, false>(q, K);
            const T a2[4] = {q.c2, q.H, q.sr, q.Mq};
            st_cell(A2 + 4 * at, a2);
        }
    };
    auto inflow = [&](WC<T> &q) { q.r = K.inflow[0]; q.u = K.inflow[1]; q.v = K.inflow[2]; q.p = K.inflow[3]; };
    // Wall mirrors of the ghost cell at (c, r), whose values q are those of the cell at (cs, rs).
    auto mirror_ghost = [&](WC<T> &q, int c, int r, int cs, int kx, int ky) {
        const int i = ix0 + c, j = jy0 + r;
        // (the boundary face's row clamped to the grid: corner ghost cells, whose velocities are
        //  never used)
        if (ky == 1 && kx != 2) {
            T nx, ny, l;
            geom_y(cs, (j < 0 ? 0 : nj) - jy0, nx, ny, l);
            mirror_vel(q.u, q.v, nx, ny);
        }
        if (kx == 1) {
            T nx, ny, l;
            geom_x((i < 0 ? 0 : ni) - ix0, pery ? r : clampi(j, 0, nj - 1) - jy0, nx, ny, l);
            mirror_vel(q.u, q.v, nx, ny);
        }
    };
    const T rate = a.dt_fixed_t > T(0) ? T(1) : rate_at<T>(a.rate_rd + g);   // (used when the copies have landed)
    const T rxy = K.dy / K.dx, cy = T(0.5) * K.dx * K.Vi;   // Cartesian residual weights
    copies_wait<0>();
    // (each thread turns the cells that it copied itself into primitives: no barrier in between, but for
    //  the vertices that mirrors at curved walls need)
    if constexpr (CURV && WALLS) __syncthreads();
    over(recip[3 * STAGES + 1], 0, W, 0, R, [&](int c, int r) {
        if ((CM[2 * c] | RM[2 * r]) >= 0) {
            T raw[4];
            WC<T> q;
            ld_own(U + 4 * (r * W + c), raw);
            prims(raw, q);
            if (WALLS && edge) {
                const int cm = CM[2 * c + 1], kx = cm >> 16, ky = RM[2 * r + 1] >> 16;
                if (kx == 2 || ky == 2) inflow(q);
                if (kx | ky) mirror_ghost(q, c, r, cm & 0xffff, kx, ky);
            }
            put_cell(r * W + c, q);
        }
    });
    __syncthreads();

    // (divided here: next to its load the quotient waited for that, 256^2 Gresho vortex, 50 steps, 586 us against 569,
    //  64^2 FP64 vortex, 20 steps, 670 against 660)
    const T dt = a.dt_fixed_t > T(0) ? a.dt_fixed_t : a.cfl_t / rate;
    T my_rate = T(0);
#pragma unroll 1
    for (int s = 0; s < STAGES; ++s) {
        int lox, hix, loy, hiy;
        margin(s, lox, hix, loy, hiy);
        const unsigned *const m = recip + 3 * s;
        const T alpha = STAGES == 1 ? a.alpha : (s == 0 ? T(0) : (s == 1 ? T(0.75) : T(1.0 / 3.0)));
        const T beta = STAGES == 1 ? a.beta : (s == 0 ? T(1) : (s == 1 ? T(0.25) : T(2.0 / 3.0)));
        const bool last = s == STAGES - 1;

        // The ghost cells that a stage reads: H beyond its margin, where that leaves the grid on a side that is
        // not periodic; columns west and east (all rows), then rows south and north (0 to H of each).
        auto ghosts = [&](int s, int from, auto &&body) {
            int lx, hx, ly, hy;
            margin(s, lx, hx, ly, hy);
            const int gW = perx ? 0 : max(0, -ix0 - (lx - H)), gE = perx ? 0 : max(0, hx + H - (ni - ix0));
            const int gS = pery ? 0 : max(0, -jy0 - (ly - H)), gN = pery ? 0 : max(0, hy + H - (nj - jy0));
            const int rows = hy - ly + 2 * H, cl = lx - H + gW, cols = hx + H - gE - cl;
            const int nW = gW * rows, nE = nW + gE * rows, nS = nE + gS * cols, nN = nS + gN * cols;
#pragma unroll 1
            for (int k = from; k < nN; k += nt) {
                int c, r;
                if (k < nE) {
                    const int q = k < nW ? k : k - nW, two = (k < nW ? gW : gE) - 1;
                    c = (k < nW ? lx - H : hx + H - gE) + (two ? q & 1 : 0);
                    r = ly - H + (q >> two);
                } else {
                    const int q = k < nS ? k - nE : k - nS, d = q >= cols;
                    c = cl + q - (d ? cols : 0);
                    r = (k < nS ? ly - H : hy + H - gN) + d;
                }
                body(c, r, CM[2 * c + 1], RM[2 * r + 1]);
            }
        };
        if (!WALLS && edge) {
            ghosts(s, tid, [&](int c, int r, int cm, int rm) {
                WC<T> q;
                if (cm >> 16 == 2 || rm >> 16 == 2) inflow(q);
                else {
                    T raw[4];
                    ld_own(U + 4 * ((rm & 0xffff) * W + (cm & 0xffff)), raw);
                    prims(raw, q);
                }
                put_cell(r * W + c, q);
            });
            __syncthreads();
        }

        // ---- cells: Eq. 97 ratios of the west and south faces (1 at solid sides), limited slopes
        // (at first order the ratios of the outermost column's west and row's south faces read outside
        //  the stage's cells, but inside shared memory, and are not used)
        over(m[0], lox - 1, hix + 1, loy - 1, hiy + 1, [&](int c, int r) {
            const int at = r * W + c;
            T q[4], qw[4], qs[4];
            ld_own(A1 + 4 * at, q);
            ld_own(A1 + 4 * (at - 1), qw);
            ld_own(A1 + 4 * (at - W), qs);
            T Px = ratio_P(qw[0], qw[3], q[0], q[3]), Py = ratio_P(qs[0], qs[3], q[0], q[3]);
            int fl = 0, flw = 0, fls = 0;
            if constexpr (WALLS) {
                fl = FL[at] & 1; flw = FL[at - 1] & 1; fls = FL[at - W] & 1;
                if (fl | flw) Px = T(1);
                if (fl | fls) Py = T(1);
            }
            PP[2 * at] = Px;
            PP[2 * at + 1] = Py;
            if constexpr (MUSCL) {
                T qe[4], qn[4];
                ld_own(A1 + 4 * (at + 1), qe);
                ld_own(A1 + 4 * (at + W), qn);
                if constexpr (WALLS) {
                    // a solid stencil cell is replaced by the mirror of this cell about their face
                    const int fle = FL[at + 1] & 1, fln = FL[at + W] & 1;
                    if (flw | fls | fle | fln) {
                        T nx, ny, l;
                        if (flw) { for (int k = 0; k < 4; ++k) qw[k] = q[k]; geom_x(c, r, nx, ny, l); mirror_vel(qw[1], qw[2], nx, ny); }
                        if (fle) { for (int k = 0; k < 4; ++k) qe[k] = q[k]; geom_x(c + 1, r, nx, ny, l); mirror_vel(qe[1], qe[2], nx, ny); }
                        if (fls) { for (int k = 0; k < 4; ++k) qs[k] = q[k]; geom_y(c, r, nx, ny, l); mirror_vel(qs[1], qs[2], nx, ny); }
                        if (fln) { for (int k = 0; k < 4; ++k) qn[k] = q[k]; geom_y(c, r + 1, nx, ny, l); mirror_vel(qn[1], qn[2], nx, ny); }
                    }
                }
                // (FP32: half the slopes)
                T sx[4], sy[4];
                auto slopes = [&](auto limited) {
                    for (int k = 0; k < 4; ++k) {
                        if constexpr (PAIRS) {
                            const V2 B = mk2(q[k], q[k]), sl = limited(B - mk2(qw[k], qs[k]), mk2(qe[k], qn[k]) - B);
                            sx[k] = sl.v.x; sy[k] = sl.v.y;
                        } else {
                            sx[k] = limited(q[k] - qw[k], qe[k] - q[k]);
                            sy[k] = limited(q[k] - qs[k], qn[k] - q[k]);
                        }
                    }
                };
                if constexpr (PAIRS) {
                    if (vanleer) slopes([](V2 a, V2 b) { return half_vanleer(a, b); });
                    else slopes([](V2 a, V2 b) { return half_minmod(a, b); });
                } else {
                    slopes([&](T a, T b) { return limiter(vanleer, a, b); });
                }
                st_cell(A2 + 4 * at, sx);
                st_cell(SY + 4 * at, sy);
            }
        });
        __syncthreads();

        // ---- faces. `d` = 1: the west face of position (c, r), `d` = W: its south face.
        auto detector_min = [&](int at, int d) {
            // Eq. 96 in 2D: the face and the transverse faces of both its cells
            const int o = d == 1 ? 0 : 1, tr = d == 1 ? W : 1;
            const T *q = PP + 2 * at;
            return fmn3(fmn3(q[o], q[1 - o - 2 * d], q[1 - o - 2 * d + 2 * tr]), q[1 - o], q[1 - o + 2 * tr]);
        };
        // The two sides of a face in global primitives (MUSCL: reconstructed, else the cells), walls
        // taking the fluid side's first-order state and its mirror; false where no flux passes.
        auto sides = [&](int at, int d, T nx, T ny, T L[4], T Rr[4]) {
            ld_own(A1 + 4 * (at - d), L);
            ld_own(A1 + 4 * at, Rr);
            int fA = 0, fB = 0;
            if constexpr (WALLS) { fA = FL[at - d]; fB = FL[at]; }
            if constexpr (MUSCL) {
                if (!WALLS || (fA | fB) == 0) {
                    const T *S = d == 1 ? A2 : SY;
                    const T h = PAIRS ? T(1) : T(0.5);
                    T sA[4], sB[4], rL[4], rR[4];
                    ld_own(S + 4 * (at - d), sA);
                    ld_own(S + 4 * at, sB);
                    for (int k = 0; k < 4; ++k) { rL[k] = vfma(h, sA[k], L[k]); rR[k] = vfnma(h, sB[k], Rr[k]); }
                    // (FP32: positive by the limiters' bounds, the faces where it could fail being marginal_face's)
                    if (PAIRS || (rL[0] > T(0) && rL[3] > T(0) && rR[0] > T(0) && rR[3] > T(0)))
                        for (int k = 0; k < 4; ++k) { L[k] = rL[k]; Rr[k] = rR[k]; }
                }
            }
            if constexpr (WALLS) {
                if (fA | fB) {
                    if (fA & fB & 1) return false;
                    if (fA) { for (int k = 0; k < 4; ++k) L[k] = Rr[k]; mirror_vel(L[1], L[2], nx, ny); }
                    else { for (int k = 0; k < 4; ++k) Rr[k] = L[k]; mirror_vel(Rr[1], Rr[2], nx, ny); }
                }
            }
            return true;
        };
        // The whole evaluation of one face on its own (FP64; in FP32 the faces across a jump of 1e5
        // or more in density or pressure, whose positivity is decided in FP64): face_scalar.
        auto marginal_face = [&](int c, int r, int d, T s1, T F[4]) {
            const int at = r * W + c;
            Face<T> f;
            T l;
            auto cell = [&](int q, WC<T> &o) {
                T v[4];
                ld_own(A1 + 4 * q, v);
                o.r = v[0]; o.u = v[1]; o.v = v[2]; o.p = v[3];
                o.c2 = o.H = o.sr = o.Mq = T(0);
                o.fl = WALLS ? FL[q] : 0;
            };
            cell(at - d, f.A); cell(at, f.B);
            if constexpr (MUSCL) {
                cell(at - 2 * d, f.Am); cell(at + d, f.Bp);
                if (d == 1) { geom_x(c - 1, r, f.nAmx, f.nAmy, l); geom_x(c + 1, r, f.nBpx, f.nBpy, l); }
                else { geom_y(c, r - 1, f.nAmx, f.nAmy, l); geom_y(c, r + 1, f.nBpx, f.nBpy, l); }
            }
            if (d == 1) geom_x(c, r, f.nx, f.ny, f.len);
            else geom_y(c, r, f.nx, f.ny, f.len);
            f.s1 = s1;
            face_scalar<T, MUSCL>(f, K, eps1, xi_form, vanleer, F);
        };
        if constexpr (PAIRS) {
            over(m[1], lox, hix + 1, loy, hiy + 1, [&](int c, int r) {
                const int at = r * W + c;
                V2 s1 = mk2(1.f, 1.f);
                if (use_s1) s1 = detector_of(mk2(detector_min(at, 1), detector_min(at, W)));
                float Fx[4], Fy[4];
                if constexpr (MUSCL) {
                    const float eps = 1e-5f;
                    if (PP[2 * at] < eps || PP[2 * at + 1] < eps) {
                        marginal_face(c, r, 1, s1.v.x, Fx);
                        marginal_face(c, r, W, s1.v.y, Fy);
                        st_cell(FX + 4 * at, Fx);
                        st_cell(FY + 4 * at, Fy);
                        return;
                    }
                }
                Face<float> fx, fy;
                geom_x(c, r, fx.nx, fx.ny, fx.len);
                geom_y(c, r, fy.nx, fy.ny, fy.len);
                fx.s1 = s1.v.x; fy.s1 = s1.v.y;
                float Lx[4], Rx[4], Ly[4], Ry[4];
                const bool okx = sides(at, 1, fx.nx, fx.ny, Lx, Rx), oky = sides(at, W, fy.nx, fy.ny, Ly, Ry);
                V2 WL[4], WR[4];
                if constexpr (MUSCL) {
                    for (int k = 0; k < 4; ++k) {   // (Cartesian: the normal velocity first)
                        const int ky = CURV || k == 0 || k == 3 ? k : 3 - k;
                        WL[k] = mk2(Lx[k], Ly[ky]); WR[k] = mk2(Rx[k], Ry[ky]);
                    }
                } else {
                    auto put = [&](const float v[4], int q, WC<float> &o) {
                        float d4[4];
                        ld_own(A2 + 4 * q, d4);
                        o.r = v[0]; o.u = v[1]; o.v = v[2]; o.p = v[3];
                        o.c2 = d4[0]; o.H = d4[1]; o.sr = d4[2]; o.Mq = d4[3];
                    };
                    // (a wall face's mirrored side has the fluid cell's derived quantities)
                    int ax = at - 1, bx = at, ay = at - W, by = at;
                    if constexpr (WALLS) {
                        if (FL[ax]) ax = at; else if (FL[bx]) bx = at - 1;
                        if (FL[ay]) ay = at; else if (FL[by]) by = at - W;
                    }
                    put(Lx, ax, fx.A); put(Rx, bx, fx.B); put(Ly, ay, fy.A); put(Ry, by, fy.B);
                }
                faces_packed<MUSCL, CURV>(fx, fy, K, eps1, xi_form, WL, WR, Fx, Fy);
                if constexpr (WALLS) {
                    if (!okx) Fx[0] = Fx[1] = Fx[2] = Fx[3] = 0.f;
                    if (!oky) Fy[0] = Fy[1] = Fy[2] = Fy[3] = 0.f;
                }
                st_cell(FX + 4 * at, Fx);
                st_cell(FY + 4 * at, Fy);
            });
        } else {
            // west faces, then south faces, one list: every lane has a face
            const int wx = hix + 1 - lox, hx = hiy - loy, nx_ = wx * hx, wyy = hix - lox, ny_ = wyy * (hiy + 1 - loy);
            const unsigned mx = m[1], my = m[2];
            for (int idx = tid; idx < nx_ + ny_; idx += nt) {
                const bool isx = idx < nx_;
                const int k = isx ? idx : idx - nx_, wd = isx ? wx : wyy;
                const int q = wd == 1 ? k : (int)__umulhi((unsigned)k, isx ? mx : my);
                const int c = lox + k - q * wd, r = loy + q, at = r * W + c, d = isx ? 1 : W;
                T nx, ny, len;
                if (isx) geom_x(c, r, nx, ny, len); else geom_y(c, r, nx, ny, len);
                T L[4], Rr[4], F[4] = {T(0), T(0), T(0), T(0)};
                if (sides(at, d, nx, ny, L, Rr)) {
                    const T s1 = use_s1 ? detector_of(detector_min(at, d)) : T(1);
                    FS<T> sl, sr;
                    if constexpr (MUSCL) {
                        if constexpr (CURV) {
                            sl = side_rot(L[0], L[1], L[2], L[3], nx, ny, K);
                            sr = side_rot(Rr[0], Rr[1], Rr[2], Rr[3], nx, ny, K);
                        } else {
                            sl = side_from_prims(L[0], isx ? L[1] : L[2], isx ? L[2] : L[1], L[3], K);
                            sr = side_from_prims(Rr[0], isx ? Rr[1] : Rr[2], isx ? Rr[2] : Rr[1], Rr[3], K);
                        }
                    } else {
                        int qa = at - d, qb = at;
                        if constexpr (WALLS) { if (FL[qa]) qa = at; else if (FL[qb]) qb = at - d; }
                        T da[4], db[4];
                        ld_own(A2 + 4 * qa, da);
                        ld_own(A2 + 4 * qb, db);
                        if constexpr (CURV) {
                            sl = {L[0], vfma(nx, L[1], ny * L[2]), vfma(nx, L[2], -(ny * L[1])), L[3], da[0], da[1], da[2], da[3]};
                            sr = {Rr[0], vfma(nx, Rr[1], ny * Rr[2]), vfma(nx, Rr[2], -(ny * Rr[1])), Rr[3], db[0], db[1], db[2], db[3]};
                        } else {
                            sl = {L[0], isx ? L[1] : L[2], isx ? L[2] : L[1], L[3], da[0], da[1], da[2], da[3]};
                            sr = {Rr[0], isx ? Rr[1] : Rr[2], isx ? Rr[2] : Rr[1], Rr[3], db[0], db[1], db[2], db[3]};
                        }
                    }
                    T G2[4];
                    roeam_flux2(sl, sr, s1, K, eps1, xi_form, G2);
                    if constexpr (CURV) {
                        const T hl = T(0.5) * len, hx = hl * nx, hy = hl * ny;   // (as face_scalar)
                        F[0] = hl * G2[0];
                        F[1] = vfma(hx, G2[1], -(hy * G2[2]));
                        F[2] = vfma(hy, G2[1], hx * G2[2]);
                        F[3] = hl * G2[3];
                    } else {   // (twice the flux: the residual applies the half lengths)
                        F[0] = G2[0]; F[1] = isx ? G2[1] : G2[2]; F[2] = isx ? G2[2] : G2[1]; F[3] = G2[3];
                    }
                }
                st_cell((isx ? FX : FY) + 4 * at, F);
            }
        }
        __syncthreads();

        // ---- cells: R = D sc, then the stage combination. With walls also the ghost cells of the next stage,
        //      each from another update of its source cell: they need neither a phase of their own nor a
        //      barrier (0.4 us a stage on a curved duct), for which U^(k) must not be overwritten meanwhile.
        //      (Without walls ghost cells are cheap, and one buffer for U^(k) is 2 % faster.)
        T *const cur = !WALLS || s == 0 ? U : V + 4 * P * (s - 1), *const nxt = WALLS ? V + 4 * P * s : U;
        // (c, r): the cell; (gc, gr): where its values go, of kind (kx, ky)
        auto update = [&](auto is_ghost, int c, int r, int gc, int gr, int kx, int ky) {
            constexpr bool ghost = decltype(is_ghost)::value;
            const int at = r * W + c;
            T fw[4], fe[4], fs[4], fn[4], uk[4], un[4], out[4];
            ld_own(FX + 4 * at, fw);
            ld_own(FX + 4 * (at + 1), fe);
            ld_own(FY + 4 * at, fs);
            ld_own(FY + 4 * (at + W), fn);
            ld_own(cur + 4 * at, uk);
            const bool own = !ghost && c >= E && c < E + w && r >= E && r < E + h;   // (others also update halo cells)
            const long long x = G.off + 4 * ((long long)(jy0 + r) * pitch + (ix0 + c));
            if (STAGES == 1) {
                if (alpha != T(0) && TILE_OK(x, 4, n_un)) ld_own(a.un + x, un);
                else for (int k = 0; k < 4; ++k) un[k] = uk[k];
            } else if (WALLS) {
                ld_own(U + 4 * at, un);
            } else if (s == 0) {
                for (int k = 0; k < 4; ++k) un[k] = uk[k];
                st_cell(V + 4 * at, uk);
            } else {
                ld_own(V + 4 * at, un);
            }
            bool solid = false;
            if constexpr (WALLS) solid = FL[at] & 1;
            CellGeom<T> cg;
            if constexpr (CURV) {
                T x00, y00, x10, y10, x01, y01, x11, y11;
                vtx(c, r, x00, y00); vtx(c + 1, r, x10, y10); vtx(c, r + 1, x01, y01); vtx(c + 1, r + 1, x11, y11);
                cg = cell_geom(x00, x10, x01, x11, y00, y10, y01, y11, K.dx, K.dy);
            } else {
                cg.Xx = K.dy; cg.Xy = T(0); cg.Yx = T(0); cg.Yy = K.dx; cg.V = K.V;
            }
            const T sc = CURV ? rcp(cg.V) : cy;
            if (STAGES == 1 && a.residual) {
                for (int k = 0; k < 4; ++k) {
                    const T D = CURV ? (fw[k] - fe[k] + fs[k]) - fn[k] : vfma(fw[k] - fe[k], rxy, fs[k]) - fn[k];
                    out[k] = solid ? T(0) : D * sc;
                }
                if (TILE_OK(x - a.dst_shift, 4, n_dst)) st_cell(a.dst + (x - a.dst_shift), out);
                return;
            }
            for (int k = 0; k < 4; ++k) {
                T D = CURV ? (fw[k] - fe[k] + fs[k]) - fn[k] : vfma(fw[k] - fe[k], rxy, fs[k]) - fn[k];
                if (solid) D = T(0);
                const T upd = vfma(dt * sc, D, uk[k]);
                out[k] = vfma(alpha, un[k], beta * upd);
            }
            if (!last) {
                if (!ghost) st_cell(nxt + 4 * at, out);
                WC<T> q;
                prims(out, q);
                if constexpr (WALLS && ghost) mirror_ghost(q, gc, gr, c, kx, ky);
                put_cell(gr * W + gc, q);
            } else if (TILE_OK(x, 4, n_dst)) {
                st_cell(a.dst + x, out);
            }
            if (own && !solid) {
                if (last && a.want_rate) {
                    const CellPrims<T> cp = cell_prims(out[0], out[1], out[2], out[3], K);
                    if (!(out[0] > T(0)) || !(cp.p > T(0))) {
                        const bool fin = isfinite((double)out[0]) && isfinite((double)cp.p);
                        atomicOr(a.status, fin ? ST_NONPOSITIVE : ST_NONFINITE);
                    } else {
                        my_rate = vmax(my_rate, cell_rate<CURV>(cp, cg, K));
                    }
                } else {
                    const T e2 = T(2) * out[0] * out[3], m2 = vfma(out[1], out[1], out[2] * out[2]);
                    if (!(out[0] > T(0)) || !(e2 > m2)) {
                        const CellPrims<T> cp = cell_prims(out[0], out[1], out[2], out[3], K);
                        if (!(out[0] > T(0)) || !(cp.p > T(0))) {
                            const bool fin = isfinite((double)out[0]) && isfinite((double)cp.p);
                            atomicOr(a.status, fin ? ST_NONPOSITIVE : ST_NONFINITE);
                        }
                    }
                }
            }
        };
        over(m[2], lox, hix, loy, hiy, [&](int c, int r) { update(Flag<false>(), c, r, c, r, 0, 0); });
        if (WALLS && !last && edge)   // (the last threads are idle in the cells' last round)
            ghosts(s + 1, nt - 1 - tid, [&](int c, int r, int cm, int rm) {
                const int kx = cm >> 16, ky = rm >> 16;
                if (kx != 2 && ky != 2) update(Flag<true>(), cm & 0xffff, rm & 0xffff, c, r, kx, ky);   // (INFLOW: set at the start)
            });
        if (!last) __syncthreads();
    }
    if (a.want_rate) {
        my_rate = warp_rate_max(my_rate);
        if ((tid & 31) == 0) red[tid >> 5] = my_rate;
        __syncthreads();
        if (tid < 32) {
            my_rate = warp_rate_max(tid < nt / 32 ? red[tid] : T(0));
            if (tid == 0 && my_rate > T(0)) atomicMax(a.rate_wr + g, rate_bits(my_rate));
        }
    }
}

// Sums and maxima of a residual in a fixed order: warp shuffles, then the block's warps.
template <typename T>
__global__ void __launch_bounds__(256) norms_kernel(const GridDev *grids, int idx, const T *__restrict__ R, double *partials)
{
    __shared__ double wred[8][8];
    const GridDev &G = grids[idx];
    const unsigned ni = (unsigned)G.ni, n = ni * (unsigned)G.nj, pitch = (unsigned)G.pitch;
    const T *const base = R + G.off;
    double v[8] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
    for (unsigned q = blockIdx.x * 256u + threadIdx.x; q < n; q += gridDim.x * 256u) {
        const unsigned j = q / ni, i = q - j * ni;
        T r[4];
        ld_own(base + 4 * ((long long)j * pitch + i), r);
        for (int k = 0; k < 4; ++k) {
            const double x = (double)r[k];
            v[k] = fma(x, x, v[k]);
            v[4 + k] = fmax(v[4 + k], fabs(x));
        }
    }
    for (int o = 16; o > 0; o >>= 1)
        for (int k = 0; k < 8; ++k) {
            const double x = __shfl_xor_sync(0xffffffffu, v[k], o);
            v[k] = k < 4 ? v[k] + x : fmax(v[k], x);
        }
    if ((threadIdx.x & 31) == 0)
        for (int k = 0; k < 8; ++k) wred[threadIdx.x >> 5][k] = v[k];
    __syncthreads();
    if (threadIdx.x < 8) {
        double r = 0.0;
        for (int w = 0; w < 8; ++w) r = threadIdx.x < 4 ? r + wred[w][threadIdx.x] : fmax(r, wred[w][threadIdx.x]);
        partials[(size_t)blockIdx.x * 8 + threadIdx.x] = r;
    }
}

// ------------------------------------------------------------------ launchers
template <typename T, bool MUSCL, bool CURV, bool WALLS> struct TileVariant {
    static constexpr int STAGES = tile_stages<T>();
    static cudaError_t launch(const TileArgs<T> &a, int ntiles, int threads, size_t smem, cudaStream_t s)
    {
        return launch_pdl(a.ngrids == 1 ? tile_kernel<T, MUSCL, CURV, WALLS, STAGES, true> : tile_kernel<T, MUSCL, CURV, WALLS, STAGES, false>,
                          dim3((unsigned)ntiles), dim3((unsigned)threads), smem, s, a);
    }
    static cudaError_t prepare(bool one, size_t smem)
    {
        return cudaFuncSetAttribute(one ? tile_kernel<T, MUSCL, CURV, WALLS, STAGES, true> : tile_kernel<T, MUSCL, CURV, WALLS, STAGES, false>,
                                    cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    }
};

#define ROEAM_TILE_DISPATCH(CALL)                                                                              \
    if (muscl) return curv ? (walls ? TileVariant<T, true, true, true>::CALL : TileVariant<T, true, true, false>::CALL) \
                           : (walls ? TileVariant<T, true, false, true>::CALL : TileVariant<T, true, false, false>::CALL); \
    return curv ? (walls ? TileVariant<T, false, true, true>::CALL : TileVariant<T, false, true, false>::CALL) \
                : (walls ? TileVariant<T, false, false, true>::CALL : TileVariant<T, false, false, false>::CALL);

template <typename T>
cudaError_t TileLaunchers<T>::step(const TileArgs<T> &a, int muscl, int curv, int walls, int ntiles, int threads,
                                   size_t smem, cudaStream_t s)
{
    ROEAM_TILE_DISPATCH(launch(a, ntiles, threads, smem, s))
}

template <typename T>
cudaError_t TileLaunchers<T>::norms(const GridDev *grids, int idx, const T *R, double *partials, int nblocks, cudaStream_t s)
{
    norms_kernel<T><<<nblocks, 256, 0, s>>>(grids, idx, R, partials);
    return cudaGetLastError();
}

// Allows the kernel the most shared memory that a launch may ask for (the attribute belongs to the
// device, so every handle asks for the same).
template <typename T>
cudaError_t TileLaunchers<T>::prepare(int muscl, int curv, int walls, bool one)
{
    ROEAM_TILE_DISPATCH(prepare(one, TILE_SMEM_MAX))
}

}  // namespace roeam
