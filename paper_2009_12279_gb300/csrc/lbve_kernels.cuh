// lbve_kernels.cuh -- kernels of one time step of the coupled LB + Oldroyd-B method
// (Kuron et al., arXiv:2009.12279), templated on the PDF storage type.  Included by
// lbve_f64.cu (FP64 storage, FMA contraction off) and lbve_f32.cu (FP32/FP16/BF16
// storage with FP32 arithmetic), which instantiate them behind the launcher table of
// lbve_launch.h.
//
// Per step (split schedule):   k_momentum_exchange (links into tracked bodies)
//                              k_lb      : polymer force, moments, TRT collide, AA stream
//                              k_fv      : finite-volume stress update tau^t -> tau^{t+1}
// The fused schedule (k_fused) merges k_fv of step t with k_lb of step t+1.
#pragma once

#include <cstddef>
#include <type_traits>

#include "lbve_device.cuh"
#include "lbve_launch.h"

namespace lbve {

// 128-thread stream-collide blocks with a resident-block floor per SM, i.e. a register
// cap of 65536 / (128 x floor).  FP32 and 16-bit storage take 72 registers (7 blocks, no
// spills): measured on GB300 at 192^3, us, with 5 / 6 / 7 / 8 / 9 blocks: FP32 293 / 253 /
// 248 / 257 / 255; BF16 239 / 208 / 198 / 209 / 206; FP16 at 128^3 72 / - / 65 / 70 / 68.
// FP64, bound by its pipe from a few warps on, takes 128 (4 blocks, no spills).
template <class S>
constexpr int lb_min_blocks() {
    return sizeof(S) == 8 ? 4 : 7;
}
// 256-thread stress blocks, 3 resident per SM (64 registers, the variant builds 80; no spills)
#ifndef LBVE_FV_MIN_BLOCKS
#define LBVE_FV_MIN_BLOCKS 3
#endif
#ifndef LBVE_LBB_MIN_BLOCKS  // batched stream-collide (both parities in one kernel; the
#define LBVE_LBB_MIN_BLOCKS 7   // serving mix's pool step measured 1.201 ms at 7, 1.217 at 8)
#endif

// Division of a 32-bit dividend below 2^31 by a fixed divisor (T. Granlund and
// P. L. Montgomery, "Division by invariant integers using multiplication", 1994):
// q = (mulhi(m, n) + n) >> s with s = ceil(log2 d), m = floor(2^32 (2^s - d) / d) + 1.
struct FastDiv {
    unsigned m, s;
    __host__ __device__ static FastDiv of(unsigned d) {
        FastDiv f;
        f.s = 0;
        while ((1ull << f.s) < d) ++f.s;
        f.m = (unsigned)((((1ull << f.s) - d) << 32) / d + 1ull);
        return f;
    }
    __device__ __forceinline__ unsigned div(unsigned n) const { return (__umulhi(m, n) + n) >> s; }
};

template <class S>
struct KArgs {
    using R = typename Store<S>::R;
    Geo g;
    Phys<R> ph;
    S *f;
    const R *tau;     // stress at the time level read
    R *tau_out;       // stress at the next time level
    const R *u_in;    // velocity read by the stress update
    R *u_out;         // velocity written by the stream-collide
    const uint8_t *flag;
    const uint32_t *mask;
    const PartDev *parts;
    unsigned step;  // index of the step being performed (rounding keys of keyed stores)
    const unsigned *dstep;  // added to it (nullptr: nothing)
    unsigned *bad;  // instability flag (mapped host word) or nullptr
    int zlo, zhi;   // planes the step kernels compute
    unsigned key_base;  // added to the cell index in rounding keys (a z-slab: its global offset)
    unsigned lin;       // cells of the computed planes (per-cell kernels in memory order)
    FastDiv dnx, dny, dnz;  // division by nx, ny, nzc
    unsigned nzc;           // planes computed
    // per-direction / per-component bases (f + i np, tau + c np, u_out + k np, u_in + k np,
    // tau_out + c np), so that an address is one multiply-add of a 32-bit cell index; set
    // by link_dirs
    S *fq[Q];
    const R *tq[6];
    R *uq[3];
    const R *uiq[3];
    R *toq[6];
};

template <class S>
__host__ __device__ inline void link_dirs(KArgs<S> &a) {
    const size_t np = (size_t)a.g.np;
    for (int i = 0; i < Q; ++i) a.fq[i] = a.f + i * np;
    for (int c = 0; c < 6; ++c) a.tq[c] = a.tau + c * np;
    for (int k = 0; k < 3; ++k) a.uq[k] = a.u_out + k * np;
    for (int k = 0; k < 3; ++k) a.uiq[k] = a.u_in + k * np;
    for (int c = 0; c < 6; ++c) a.toq[c] = a.tau_out + c * np;
}

// Load f_i^t of cell r from its AA location for the given parity.
template <class S, int PAR>
__device__ __forceinline__ void load_pdfs(const KArgs<S> &a, const Cell &cl, unsigned r,
                                          typename Store<S>::R (&f)[Q]) {
    using R = typename Store<S>::R;
    const size_t np = (size_t)a.g.np;
    const R inv = a.ph.inv_scale;
#pragma unroll
    for (int i = 0; i < Q; ++i) {
        const S *p = PAR == 0 ? a.fq[i] + r : a.fq[copp(i)] + cl.idx(-cx(i), -cy(i), -cz(i));
        f[i] = Store<S>::ld(p, inv);
    }
}

// Product rounded by itself (FP64 is compiled without contraction).
__device__ __forceinline__ float mul1(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double mul1(double a, double b) { return a * b; }

// 6 w_i rho c_i . u_b of a link into the solid cell nb, whose velocity entries hold u_b.
template <class R>
__device__ __forceinline__ R moving_wall_term(R *const (&u)[3], unsigned nb, int i, R rho) {
    R cub = R(0);
    bool first = true;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const int c = cdir(i, k);
        if (c != 0) {
            const R ub = u[k][nb];
            if (first) {
                cub = c > 0 ? ub : -ub;
                first = false;
            } else {
                cub = c > 0 ? cub + ub : cub - ub;
            }
        }
    }
    const R w = i < 7 ? wgt<R>(1) : wgt<R>(7);
    return mul1(mul1(R(6) * w, rho), cub);
}
template <class R>
__device__ __noinline__ R moving_wall_call(R *u, size_t np, unsigned nb, int i, R rho) {
    R *const uq[3] = {u, u + np, u + 2 * np};
    return moving_wall_term<R>(uq, nb, i, rho);
}

// Step number of the rounding key.
template <class S>
__device__ __forceinline__ unsigned step_number(const KArgs<S> &a) {
    if constexpr (Store<S>::keyed) return a.dstep ? a.step + *a.dstep : a.step;
    return 0u;
}

// Store post-collision f*_i with AA addressing; links into solid cells bounce back with
// the moving-wall term of Eq. (ubb): f_-i(r, t+1) = f*_i(r) - 6 w_i rho c_i . u_b.
// Every f*_i also goes to its normal destination, unconditionally: when r + c_i is
// solid that slot belongs to the solid neighbour and is never read afterwards (even
// step: slot -i of r holds f_i(r + c_i)), or is the one this thread itself read before
// (odd step: slot i of r + c_i held the bounced population f_-i(r)).  The bounced value
// is an extra store for the links into solid cells only.
template <class S, int PAR, bool ROWS>
__device__ __forceinline__ void store_pdfs(const KArgs<S> &a, const Cell &cl, unsigned r, uint32_t mask,
                                           const typename Store<S>::R (&fs)[Q], typename Store<S>::R rho,
                                           unsigned step) {
    using R = typename Store<S>::R;
    const size_t np = (size_t)a.g.np;
    auto wall_term = [&](unsigned nb, int i) -> R {
        if constexpr (ROWS) return moving_wall_call<R>(a.uq[0], np, nb, i, rho);
        return moving_wall_term<R>(a.uq, nb, i, rho);
    };
    const R sc = a.ph.scale;
    const bool moving = mask & MASK_MOVING;  // else every solid neighbour is a resting no-slip wall
    if constexpr (Store<S>::keyed) {
        // 16-bit storage: the pairs (i, -i) round together (stochastically, see Store); a
        // bounce from a resting wall stores the very bits of the normal store (one of the
        // two copies is never read), a moving-wall bounce rounds its own value
        if constexpr (!ROWS) step = step_number(a);
        const uint32_t h = fmix32((r + a.key_base) ^ (step * 0x9E3779B9u));
        const uint32_t d0 = Store<S>::round2(fs[0], fs[0], sc, pair_bits(h, 0));
        Store<S>::store16(a.fq[0] + r, d0);
        if (!__any_sync(__activemask(), moving)) {
            // no lane of the warp next to a moving boundary: every bounce is a predicated
            // store of the normal store's bits
#pragma unroll
            for (int i = 1; i < Q; i += 2) {
                const uint32_t d = Store<S>::round2(fs[i], fs[i + 1], sc, pair_bits(h, (i + 1) >> 1));
#pragma unroll
                for (int q = 0; q < 2; ++q) {
                    const int j = i + q;
                    const uint32_t bits = q == 0 ? d >> 16 : d;
                    const unsigned nb = cl.idx(cx(j), cy(j), cz(j));
                    Store<S>::store16(PAR == 0 ? a.fq[copp(j)] + r : a.fq[j] + nb, bits);
                    if (nb_solid(mask, j)) Store<S>::store16(PAR == 0 ? a.fq[j] + nb : a.fq[copp(j)] + r, bits);
                }
            }
            return;
        }
#pragma unroll
        for (int i = 1; i < Q; i += 2) {
            const uint32_t d = Store<S>::round2(fs[i], fs[i + 1], sc, pair_bits(h, (i + 1) >> 1));
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                const int j = i + q;
                const uint32_t bits = q == 0 ? d >> 16 : d;
                const unsigned nb = cl.idx(cx(j), cy(j), cz(j));
                Store<S>::store16(PAR == 0 ? a.fq[copp(j)] + r : a.fq[j] + nb, bits);
                if (!nb_solid(mask, j)) continue;
                S *dst = PAR == 0 ? a.fq[j] + nb : a.fq[copp(j)] + r;
                const R X = moving ? wall_term(nb, j) : R(0);
                // a boundary at rest (X exactly zero) bounces the normal store's bits
                Store<S>::store16(dst, X == R(0) ? bits
                                                 : Store<S>::round2(fs[j] - X, fs[j] - X, sc, pair_bits(h, Q + j)));
            }
        }
        return;
    }
    Store<S>::st(a.fq[0] + r, fs[0], sc);
    if (!__any_sync(__activemask(), moving)) {
        // no lane of the warp next to a moving boundary: bounce-back is a predicated store
#pragma unroll
        for (int i = 1; i < Q; ++i) {
            const unsigned nb = cl.idx(cx(i), cy(i), cz(i));
            Store<S>::st(PAR == 0 ? a.fq[copp(i)] + r : a.fq[i] + nb, fs[i], sc);
            if (nb_solid(mask, i)) Store<S>::st(PAR == 0 ? a.fq[i] + nb : a.fq[copp(i)] + r, fs[i], sc);
        }
        return;
    }
#pragma unroll
    for (int i = 1; i < Q; ++i) {
        const unsigned nb = cl.idx(cx(i), cy(i), cz(i));
        Store<S>::st(PAR == 0 ? a.fq[copp(i)] + r : a.fq[i] + nb, fs[i], sc);
        if (nb_solid(mask, i)) {
            const R X = moving ? wall_term(nb, i) : R(0);
            Store<S>::st(PAR == 0 ? a.fq[i] + nb : a.fq[copp(i)] + r, fs[i] - X, sc);
        }
    }
}

// LB half of the step for one fluid cell, given its own stress tr and an accessor tn for
// its face neighbours' stress (tau^t): F = g + F^p, moments, u^t written out, TRT
// collision with forcing, AA streaming with bounce-back.  ROWS: the row pipeline's build.  Its
// 16 warps on an SM feel the instruction fetch of the rare moving-boundary stores and the
// step number's load in every cell, so it calls the wall term and passes step_number(a) in
// (512^3: BF16 3.67 -> 3.54 ms, FP16 3.86 -> 3.64; the per-cell kernels would spill).
template <class S, int PAR, bool FENE, bool ROWS, class TauNb>
__device__ __forceinline__ void lb_core_f(const KArgs<S> &a, const Cell &cl, unsigned r, uint32_t mask,
                                          const typename Store<S>::R (&tr)[6], const TauNb &tn,
                                          typename Store<S>::R (&f)[Q], unsigned step = 0) {
    using R = typename Store<S>::R;
    constexpr bool SH = Store<S>::shifted;
    R Fp[3], F[3], u[3], rho, drho;
    if constexpr (FENE)
        polymer_force_core_fene<R>(tr, mask, tn, a.ph, Fp);
    else
        polymer_force_core<R>(tr, mask, tn, Fp);
#pragma unroll
    for (int k = 0; k < 3; ++k) F[k] = a.ph.g[k] + Fp[k];
    moments<R, SH>(f, F, a.ph.rho0, rho, drho, u);
    const size_t np = (size_t)a.g.np;
#pragma unroll
    for (int k = 0; k < 3; ++k) a.uq[k][r] = u[k];
    const bool bad = collide<R, SH>(f, rho, drho, u, F, a.ph);
    store_pdfs<S, PAR, ROWS>(a, cl, r, mask, f, rho, step);
    // instability (rho <= 0, |u| at or above the lattice sound speed, or a NaN): a rare
    // store to the host-mapped flag
    if (bad && a.bad != nullptr) *(volatile unsigned *)a.bad = 1u;
}
template <class S, int PAR, class TauNb>
__device__ __forceinline__ void lb_core(const KArgs<S> &a, const Cell &cl, unsigned r, uint32_t mask,
                                        const typename Store<S>::R (&tr)[6], const TauNb &tn) {
    typename Store<S>::R f[Q];
    load_pdfs<S, PAR>(a, cl, r, f);
    lb_core_f<S, PAR, false, false>(a, cl, r, mask, tr, tn, f);
}

// Velocity / stress accessors of the face neighbours in global memory
// (kernel parameters: per-component bases, one multiply-add per address).
template <class S>
struct GlobalNb {
    using R = typename Store<S>::R;
    const KArgs<S> &a;
    const Cell &cl;
    __device__ __forceinline__ unsigned at(int l) const {
        const int k = l >> 1, s = (l & 1) ? -1 : 1;
        return cl.idx(k == 0 ? s : 0, k == 1 ? s : 0, k == 2 ? s : 0);
    }
    __device__ __forceinline__ R u(int l, int j) const { return a.uiq[j][at(l)]; }
    __device__ __forceinline__ R tau(int l, int c) const { return a.tq[c][at(l)]; }
};

// Cell of a thread of the per-cell kernels: blocks of x-y tiles (blockDim (bx, by), grid
// (nx/bx, ny/by, nz)), or, where tiles would leave lanes idle (83 cells on 64-wide blocks:
// 65 % of the lanes used), the cells of the computed planes in memory order (LIN: a.lin of
// them, one-dimensional grid; a build of its own, the choice at run time spilled registers
// in the stream-collide).
template <class S, bool LIN>
__device__ __forceinline__ bool cell_of_thread(const KArgs<S> &a, int &x, int &y, int &z) {
    if constexpr (LIN) {
        const unsigned r = blockIdx.x * blockDim.x + threadIdx.x;
        if (r >= a.lin) return false;
        const unsigned row = a.dnx.div(r), pl = a.dny.div(row);
        x = (int)(r - row * (unsigned)a.g.nx);
        y = (int)(row - pl * (unsigned)a.g.ny);
        z = (int)pl + a.zlo;
        return true;
    }
    x = blockIdx.x * blockDim.x + threadIdx.x;
    // chunks of rows, each swept in z (see cell_launch)
    const unsigned chunk = a.dnz.div(blockIdx.z);
    y = (chunk * gridDim.y + blockIdx.y) * blockDim.y + threadIdx.y;
    z = (int)(blockIdx.z - chunk * a.nzc) + a.zlo;
    return x < a.g.nx && y < a.g.ny;
}

// Stream-collide of the fluid cell (x, y, z) with the stress stencil read from global memory.
template <class S, int PAR, bool FENE = false>
__device__ __forceinline__ void lb_cell_at(const KArgs<S> &a, int x, int y, int z) {
    using R = typename Store<S>::R;
    const Cell cl(a.g, x, y, z);
    const unsigned r = cl.self();
    // the PDF and stress loads go out together with the mask (valid addresses for any
    // cell), not one DRAM round trip after it
    R f[Q], tr[6];
    load_pdfs<S, PAR>(a, cl, r, f);
#pragma unroll
    for (int c = 0; c < 6; ++c) tr[c] = a.tq[c][r];
    const uint32_t m = a.mask[r];
    if constexpr (Store<S>::shifted) step_next();
    if (m & 1u) return;
    auto tn = [&](int l, int c) -> R {
        const int k = l >> 1, s = (l & 1) ? -1 : 1;
        return a.tq[c][cl.idx(k == 0 ? s : 0, k == 1 ? s : 0, k == 2 ? s : 0)];
    };
    lb_core_f<S, PAR, FENE, false>(a, cl, r, m, tr, tn, f);
}

// FENE: the stress arrays hold FENE-P conformation tensors (see polymer_force_core_fene)
template <class S, int PAR, bool FENE, bool LIN>
__global__ void __launch_bounds__(128, lb_min_blocks<S>()) k_lb(KArgs<S> a) {
    step_wait();
    int x, y, z;
    if (!cell_of_thread<S, LIN>(a, x, y, z)) return;
    lb_cell_at<S, PAR, FENE>(a, x, y, z);
}

// Stress update of the cell (x, y, z) with the stencil read from global memory.
template <class S, bool VAR>
__device__ __forceinline__ void fv_cell_at(const KArgs<S> &a, int x, int y, int z) {
    using R = typename Store<S>::R;
    constexpr bool SH = Store<S>::shifted;
    const Cell cl(a.g, x, y, z);
    const unsigned r = cl.self();
    R tr[6], ur[3], out[6];
#pragma unroll
    for (int c = 0; c < 6; ++c) tr[c] = a.tq[c][r];
#pragma unroll
    for (int j = 0; j < 3; ++j) ur[j] = a.uiq[j][r];
    const uint32_t m = a.mask[r];
    if constexpr (Store<S>::shifted) step_next();
    if (m & 1u) {
#pragma unroll
        for (int c = 0; c < 6; ++c) out[c] = R(0);
    } else {
        const GlobalNb<S> nb{a, cl};
        fv_core<R, SH, VAR>(a.ph, tr, ur, m, nb, out);
    }
#pragma unroll
    for (int c = 0; c < 6; ++c) a.toq[c][r] = out[c];
}

// Per-cell stress update, for grids whose z-marching columns would not fill the chip (and
// all FP64 ones).  Bound by latency there (one round of loads, then the arithmetic), so it
// is split as finely as it goes: one cell per thread, 128-thread blocks, the neighbours'
// values through L1 (a 32^3 grid: 256 blocks in 7.7 us, where 8 columns took 20.3).  72
// registers: FENE-P 100 x 84 x 60 at 5 / 6 / 7 / 8 blocks per SM 20.4 / 19.2 / 18.7 / 18.2 us,
// Oldroyd-B 15.7 / 14.2 / 14.1 / 14.7.
template <class S, bool VAR, bool LIN>
__global__ void __launch_bounds__(128, sizeof(S) == 8 ? 5 : 7) k_fv_cells(KArgs<S> a) {
    step_wait();
    int x, y, z;
    if (!cell_of_thread<S, LIN>(a, x, y, z)) return;
    fv_cell_at<S, VAR>(a, x, y, z);
}

// Neighbour masks of the cells in a box (whole grid: lo = 0, ext = n) from the flags.
// A neighbour outside a closed side counts as solid.
__device__ __forceinline__ uint32_t cell_mask(const Geo &g, const uint8_t *__restrict__ flag, int x, int y, int z) {
    const Cell cl(g, x, y, z);
    uint32_t m = flag[cl.self()] != FLAG_FLUID ? 1u : 0u;
#pragma unroll
    for (int i = 1; i < Q; ++i) {
        const bool out = (!g.per[0] && (x + cx(i) < 0 || x + cx(i) >= g.nx)) ||
                         (!g.per[1] && (y + cy(i) < 0 || y + cy(i) >= g.ny)) ||
                         (!g.per[2] && (z + cz(i) < 0 || z + cz(i) >= g.nz));
        const int fl = out ? FLAG_NOSLIP : flag[cl.idx(cx(i), cy(i), cz(i))];
        if (fl != FLAG_FLUID) m |= 1u << i;
        if (fl != FLAG_FLUID && fl != FLAG_NOSLIP) m |= MASK_MOVING;
    }
    return m;
}

// What the step kernels read at solid cells: the boundary velocity in the velocity field
// (both buffers of the fused schedule's ping-pong, u0 and u1), so that bounce-back and the
// velocity gradient need no flag and no FP64 evaluation per link and face, and zero stress
// (the stress update multiplies it by the zero coefficient of a solid face).
template <class S>
__device__ __forceinline__ void set_solid_velocity(const KArgs<S> &a, int x, int y, int z, unsigned r,
                                                   typename Store<S>::R *u0, typename Store<S>::R *u1) {
    using R = typename Store<S>::R;
    R ub[3];
    boundary_velocity<R>(a.g, a.ph, a.parts, a.flag[r], x, y, z, ub);
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        u0[j * (size_t)a.g.np + r] = ub[j];
        u1[j * (size_t)a.g.np + r] = ub[j];
    }
}

// Neighbour masks of the cells of a box (periodically wrapped), and what its solid cells
// hold: boundary velocity, and zero stress in both stress buffers.
template <class S>
__global__ void k_build_mask(KArgs<S> a, uint32_t *__restrict__ mask, int lx, int ly, int lz, int ex, int ey, int ez,
                             typename Store<S>::R *__restrict__ tau0, typename Store<S>::R *__restrict__ tau1,
                             typename Store<S>::R *u0, typename Store<S>::R *u1) {
    using R = typename Store<S>::R;
    const Geo &g = a.g;
    const long long cells = (long long)ex * ey * ez;
    for (long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x; k < cells;
         k += (long long)gridDim.x * blockDim.x) {
        const int ix = (int)(k % ex), iy = (int)((k / ex) % ey), iz = (int)(k / ((long long)ex * ey));
        const int x = ((lx + ix) % g.nx + g.nx) % g.nx;
        const int y = ((ly + iy) % g.ny + g.ny) % g.ny;
        const int z = ((lz + iz) % g.nz + g.nz) % g.nz;
        const unsigned r = (unsigned)x + (unsigned)g.nx * ((unsigned)y + (unsigned)g.ny * (unsigned)z);
        const uint32_t m = cell_mask(g, a.flag, x, y, z);
        mask[r] = m;
        if (m & 1u) {
#pragma unroll
            for (int c = 0; c < 6; ++c) {
                tau0[c * (size_t)g.np + r] = R(0);
                tau1[c * (size_t)g.np + r] = R(0);
            }
            set_solid_velocity<S>(a, x, y, z, r, u0, u1);
        }
    }
}

// ---------------------------------------------------------------------------------
// fused schedule: one kernel per step t does the stress update of step t-1 (tau^t from
// tau^{t-1}, u^{t-1}) and the LB half of step t, marching along z through an x-y tile.
// tau^{t-1} and u^{t-1} planes are staged in shared memory with cp.async (two planes
// ahead), tau^t is kept for three planes so the polymer force of plane z reads its
// face neighbours from shared memory, and only the tile's own cells are written out.
// ---------------------------------------------------------------------------------
constexpr int FT_X = 32, FT_Y = 8;
constexpr int H2X = FT_X + 4, H2Y = FT_Y + 4, NH2 = H2X * H2Y;  // staged inputs
constexpr int H1X = FT_X + 2, H1Y = FT_Y + 2, NH1 = H1X * H1Y;  // tau^t and masks

template <class R>
struct FusedSmem {
    R in_tau[3][6][NH2];
    R in_u[3][3][NH2];
    R tnew[3][6][NH1];
    uint32_t mask[4][NH1];
};

struct FusedWork {
    int tiles_x, tiles_y, zchunk, nzchunks;
};

__device__ __forceinline__ void cp_async4(void *dst, const void *src) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(d), "l"(src));
}
__device__ __forceinline__ void cp_async8(void *dst, const void *src) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(d), "l"(src));
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;\n" ::: "memory"); }

template <class R>
__device__ __forceinline__ void cp_async_real(R *dst, const R *src) {
    if constexpr (sizeof(R) == 8)
        cp_async8(dst, src);
    else
        cp_async4(dst, src);
}
// Copy of one real that reads n (sizeof(R) or 0) bytes and zero-fills the rest: n = 0
// writes a zero without reading src (which must still be a valid address).
// 16-byte copy that reads n (16 or 0) bytes: both addresses 16-byte aligned
__device__ __forceinline__ void cp_async16_zfill(void *dst, const void *src, unsigned n) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(d), "l"(src), "r"(n));
}
template <class R>
__device__ __forceinline__ void cp_async_real_zfill(R *dst, const R *src, unsigned n) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    if constexpr (sizeof(R) == 8)
        asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;\n" ::"r"(d), "l"(src), "r"(n));
    else
        asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;\n" ::"r"(d), "l"(src), "r"(n));
}

// wrapped coordinate along a side, or -1 outside a closed side
__device__ __forceinline__ int side_coord(int q, int n, int per) {
    if (q >= 0 && q < n) return q;
    if (!per) return -1;
    return ((q % n) + n) % n;
}

__device__ __forceinline__ int ring3(int z) { return ((z % 3) + 3) % 3; }
__device__ __forceinline__ int ring4(int z) { return ((z % 4) + 4) % 4; }

// Smem neighbour accessor of the fused stress update (the staged planes zz-1, zz, zz+1).
template <class S>
struct SmemNb {
    using R = typename Store<S>::R;
    const FusedSmem<R> &sm;
    int sc, sd, su, c2;
    __device__ __forceinline__ int slot(int l) const { return l == 4 ? su : (l == 5 ? sd : sc); }
    __device__ __forceinline__ int cell(int l) const {
        return l == 0 ? c2 + 1 : l == 1 ? c2 - 1 : l == 2 ? c2 + H2X : l == 3 ? c2 - H2X : c2;
    }
    __device__ __forceinline__ R u(int l, int j) const { return sm.in_u[slot(l)][j][cell(l)]; }
    __device__ __forceinline__ R tau(int l, int c) const { return sm.in_tau[slot(l)][c][cell(l)]; }
};

template <class S, int PAR>
__global__ void __launch_bounds__(FT_X * FT_Y, sizeof(typename Store<S>::R) == 8 ? 1 : 3) k_fused(KArgs<S> a, FusedWork w) {
    using R = typename Store<S>::R;
    constexpr bool SH = Store<S>::shifted;
    constexpr int NT = FT_X * FT_Y;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    FusedSmem<R> &sm = *reinterpret_cast<FusedSmem<R> *>(smem_raw);
    const int tid = threadIdx.x;
    const int item = blockIdx.x;
    const int tx = item % w.tiles_x;
    const int ty = (item / w.tiles_x) % w.tiles_y;
    const int zc = item / (w.tiles_x * w.tiles_y);
    const int x0 = tx * FT_X, y0 = ty * FT_Y;
    const int z0 = zc * w.zchunk;
    const int z1 = min(a.g.nz, z0 + w.zchunk);
    const size_t np = (size_t)a.g.np;
    const unsigned nx = (unsigned)a.g.nx, nxy = (unsigned)a.g.nx * (unsigned)a.g.ny;

    // in-plane offsets of the cells this thread stages (H2: tid, tid + NT; H1: the same)
    // and of its own stress-update cells; -1 marks a cell outside a closed side
    int off2[2], off1[2];
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        const int k2 = tid + q * NT;
        off2[q] = -1;
        if (k2 < NH2) {
            const int xg = side_coord(x0 - 2 + k2 % H2X, a.g.nx, a.g.per[0]);
            const int yg = side_coord(y0 - 2 + k2 / H2X, a.g.ny, a.g.per[1]);
            if (xg >= 0 && yg >= 0) off2[q] = xg + (int)nx * yg;
        }
        const int k1 = tid + q * NT;
        off1[q] = -1;
        if (k1 < NH1) {
            const int xg = side_coord(x0 - 1 + k1 % H1X, a.g.nx, a.g.per[0]);
            const int yg = side_coord(y0 - 1 + k1 / H1X, a.g.ny, a.g.per[1]);
            if (xg >= 0 && yg >= 0) off1[q] = xg + (int)nx * yg;
        }
    }

    // stage tau^{t-1}, u^{t-1} (H2 region) and neighbour masks (H1 region) of plane zz
    auto stage = [&](int zz) {
        const int zg = side_coord(zz, a.g.nz, a.g.per[2]);
        const int s3 = ring3(zz), s4 = ring4(zz);
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const int k2 = tid + q * NT;
            if (k2 < NH2) {
                if (off2[q] < 0 || zg < 0) {
#pragma unroll
                    for (int c = 0; c < 6; ++c) sm.in_tau[s3][c][k2] = R(0);
#pragma unroll
                    for (int j = 0; j < 3; ++j) sm.in_u[s3][j][k2] = R(0);
                } else {
                    const unsigned r = (unsigned)off2[q] + nxy * (unsigned)zg;
#pragma unroll
                    for (int c = 0; c < 6; ++c) cp_async_real<R>(&sm.in_tau[s3][c][k2], a.tau + c * np + r);
#pragma unroll
                    for (int j = 0; j < 3; ++j) cp_async_real<R>(&sm.in_u[s3][j][k2], a.u_in + j * np + r);
                }
            }
            const int k1 = tid + q * NT;
            if (k1 < NH1) {
                if (off1[q] < 0 || zg < 0)
                    sm.mask[s4][k1] = 0xffffffffu;
                else
                    cp_async4(&sm.mask[s4][k1], a.mask + ((unsigned)off1[q] + nxy * (unsigned)zg));
            }
        }
        cp_async_commit();
    };

    const int ti = tid % FT_X, tj = tid / FT_X;
    const int x = x0 + ti, y = y0 + tj;
    const int kc = (ti + 1) + (tj + 1) * H1X;  // the thread's own cell in H1 coordinates
    const bool own_xy = x < a.g.nx && y < a.g.ny;

#pragma unroll 1
    for (int zz = z0 - 2; zz <= z0; ++zz) stage(zz);

    // plane zf: stress update tau^t (H1 region), then stream-collide of plane zf - 1
#pragma unroll 1
    for (int zf = z0 - 1; zf <= z1; ++zf) {
        cp_async_wait_all();
        __syncthreads();
        {
            const int sc = ring3(zf), sd = ring3(zf - 1), su = ring3(zf + 1), s4 = ring4(zf);
            const int zg = side_coord(zf, a.g.nz, a.g.per[2]);
            const bool own_plane = zf >= z0 && zf < z1;
#pragma unroll 1
            for (int k = tid; k < NH1; k += NT) {
                const int hi = k % H1X, hj = k / H1X;
                const uint32_t m = sm.mask[s4][k];
                R out[6];
                if (m & 1u) {
#pragma unroll
                    for (int c = 0; c < 6; ++c) out[c] = R(0);
                } else {
                    const int c2 = (hi + 1) + (hj + 1) * H2X;
                    R tr[6], ur[3];
#pragma unroll
                    for (int c = 0; c < 6; ++c) tr[c] = sm.in_tau[sc][c][c2];
#pragma unroll
                    for (int j = 0; j < 3; ++j) ur[j] = sm.in_u[sc][j][c2];
                    const SmemNb<S> nb{sm, sc, sd, su, c2};
                    fv_core<R, SH, true>(a.ph, tr, ur, m, nb, out);
                }
#pragma unroll
                for (int c = 0; c < 6; ++c) sm.tnew[sc][c][k] = out[c];
                if (own_plane && hi >= 1 && hi <= FT_X && hj >= 1 && hj <= FT_Y) {
                    const int xo = x0 + hi - 1, yo = y0 + hj - 1;
                    if (xo < a.g.nx && yo < a.g.ny) {
                        const unsigned r = (unsigned)xo + nx * (unsigned)yo + nxy * (unsigned)zf;
#pragma unroll
                        for (int c = 0; c < 6; ++c) a.tau_out[c * np + r] = out[c];
                    }
                }
            }
        }
        __syncthreads();
        if (zf + 2 <= z1 + 1) stage(zf + 2);
        const int z = zf - 1;
        if (z >= z0 && own_xy) {
            const uint32_t m = sm.mask[ring4(z)][kc];
            if (!(m & 1u)) {
                const int sc = ring3(z), sd = ring3(z - 1), su = ring3(z + 1);
                R tr[6];
#pragma unroll
                for (int c = 0; c < 6; ++c) tr[c] = sm.tnew[sc][c][kc];
                auto tn = [&](int l, int c) -> R {
                    const int slot = l == 4 ? su : (l == 5 ? sd : sc);
                    const int cell = l == 0 ? kc + 1 : l == 1 ? kc - 1 : l == 2 ? kc + H1X : l == 3 ? kc - H1X : kc;
                    return sm.tnew[slot][c][cell];
                };
                const Cell cl(a.g, x, y, z);
                lb_core<S, PAR>(a, cl, cl.self(), m, tr, tn);
            }
        }
    }
    cp_async_wait_all();
}

// ---------------------------------------------------------------------------------
// stress update, z-marching: a block owns a 32 x 8 column of cells and walks a chunk of
// z-planes; tau^t and u^t of the planes z-1 .. z+2 (with a one-cell x-y halo) sit in a
// four-plane shared-memory ring filled with cp.async one plane ahead, so every stencil
// read of the update comes from shared memory.
// ---------------------------------------------------------------------------------
// Stress tiles: 256 threads over TX x (256 / TX) cells; the single-solve kernel uses
// 32 x 8, the batched kernel picks 16 x 16, 32 x 8 or 64 x 4 per solve.  A staged halo
// row holds the tile's TX cells from column XO on; W16 rows are widened to whole aligned
// 16-byte chunks (4 cells on each side) so that they are staged by 16-byte copies.
constexpr int FV_NT = 256;
constexpr int FV_X = 32, FV_Y = FV_NT / FV_X;
template <int TX, bool W16 = false>
struct FvTile {
    static constexpr int TY = FV_NT / TX;
    static constexpr int XO = W16 ? 4 : 1;
    static constexpr int HX = TX + 2 * XO, HN = HX * (TY + 2);  // halo row, halo cells
};
constexpr int FVH_X = FV_X + 2, FVH_Y = FV_Y + 2, FVH_N = FVH_X * FVH_Y;

// planes fetched beyond z + 1 while plane z is updated; the ring holds z - 1, z, z + 1
// and those
#ifndef LBVE_FV_AHEAD
#define LBVE_FV_AHEAD 1
#endif
constexpr int FV_RING = LBVE_FV_AHEAD + 3;
// ring slot of plane z (z >= -1); a power-of-two ring takes the low bits (two's complement)
__device__ __forceinline__ int fv_slot(int z) {
    if constexpr ((FV_RING & (FV_RING - 1)) == 0) return z & (FV_RING - 1);
    return ((z % FV_RING) + FV_RING) % FV_RING;
}

template <class R, int NH = FVH_N>
struct FvSmem {
    R tau[FV_RING][6][NH];
    R u[FV_RING][3][NH];
};

template <class S, int HX, int NH>
struct FvSmemNb {
    using R = typename Store<S>::R;
    const FvSmem<R, NH> &sm;
    int sc, sd, su, c;
    __device__ __forceinline__ int slot(int l) const { return l == 4 ? su : (l == 5 ? sd : sc); }
    __device__ __forceinline__ int cell(int l) const {
        return l == 0 ? c + 1 : l == 1 ? c - 1 : l == 2 ? c + HX : l == 3 ? c - HX : c;
    }
    __device__ __forceinline__ R u(int l, int j) const { return sm.u[slot(l)][j][cell(l)]; }
    __device__ __forceinline__ R tau(int l, int cc) const { return sm.tau[slot(l)][cc][cell(l)]; }
};

// Stress update of work item `item` (TX x TY tile, z-chunk) of one solve; VAR compiles in
// the optional finite-volume variants, ZR the restriction to planes [zlo, zhi) of a
// z-slab (a separate build: the plain one keeps its register budget).  W16 stages the
// planes by 16-byte copies: 4-byte reals, nx a multiple of 4 and 16-byte aligned stress
// and velocity arrays (the launcher checks); the result is the same either way.  PB:
// the arguments are kernel parameters, so the per-component bases (tq, uiq, toq) are
// operands for free; the batched kernel (arguments in shared memory) forms base + c np.
template <class S, int TX, bool VAR, bool ZR = false, bool W16 = false, bool PB = false>
__device__ __forceinline__ void fv_tile(const KArgs<S> &a, FvSmem<typename Store<S>::R, FvTile<TX, W16>::HN> &sm,
                                        int item, int zchunk) {
    using R = typename Store<S>::R;
    constexpr bool SH = Store<S>::shifted;
    using T = FvTile<TX, W16>;
    constexpr int NT = FV_NT, TY = T::TY, FVH_X = T::HX, FVH_N = T::HN, XO = T::XO;
    static_assert(!W16 || sizeof(R) == 4, "16-byte staging of 4-byte reals");
    static_assert(FVH_N <= 2 * NT, "two halo cells per thread at most");
    const int tid = threadIdx.x;
    const int tiles_x = (a.g.nx + TX - 1) / TX, tiles_y = (a.g.ny + TY - 1) / TY;
    const int tx = item % tiles_x, ty = (item / tiles_x) % tiles_y, zc = item / (tiles_x * tiles_y);
    const int x0 = tx * TX, y0 = ty * TY;
    const int z0 = ZR ? a.zlo + zc * zchunk : zc * zchunk;
    const int z1 = ZR ? min(a.zhi, z0 + zchunk) : min(a.g.nz, z0 + zchunk);
    const size_t np = (size_t)a.g.np;
    const unsigned nx = (unsigned)a.g.nx, nxy = (unsigned)a.g.nx * (unsigned)a.g.ny;
    auto tau_in = [&](int c) -> const R * {
        if constexpr (PB) return a.tq[c];
        return a.tau + c * np;
    };
    auto u_in = [&](int j) -> const R * {
        if constexpr (PB) return a.uiq[j];
        return a.u_in + j * np;
    };
    auto tau_out = [&](int c) -> R * {
        if constexpr (PB) return a.toq[c];
        return a.tau_out + c * np;
    };
    // 4-byte staging: halo cells tid and tid + NT of each plane (plane offsets, -1 beyond
    // a closed side); 16-byte staging: one aligned 4-cell chunk of a halo row per thread
    // (threads below CH: stress components 0..4; CH .. 2 CH - 1: component 5 and u)
    constexpr int CPR = FVH_X / 4, CH = CPR * (TY + 2);
    static_assert(!W16 || 2 * CH <= NT, "two threads per 16-byte chunk position at most");
    int off[2] = {-1, -1};
    int dpos = 0;
    const int half = W16 ? tid / CH : 0;
    if constexpr (W16) {
        if (half < 2) {
            const int p = tid - half * CH, row = p / CPR, cq = p - row * CPR;
            dpos = row * FVH_X + 4 * cq;
            const int xg = side_coord(x0 - XO + 4 * cq, a.g.nx, a.g.per[0]);
            const int yg = side_coord(y0 - 1 + row, a.g.ny, a.g.per[1]);
            if (xg >= 0 && yg >= 0) off[0] = xg + (int)nx * yg;
        }
    } else {
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const int k = tid + q * NT;
            if (k < FVH_N) {
                const int xg = side_coord(x0 - 1 + k % FVH_X, a.g.nx, a.g.per[0]);
                const int yg = side_coord(y0 - 1 + k / FVH_X, a.g.ny, a.g.per[1]);
                if (xg >= 0 && yg >= 0) off[q] = xg + (int)nx * yg;
            }
        }
    }
    static_assert(W16 || FVH_N > NT, "the first halo cell of every thread exists");
    auto stage = [&](int zz) {
        const int zg = side_coord(zz, a.g.nz, a.g.per[2]);
        const int s4 = fv_slot(zz);
        if constexpr (W16) {
            if (half < 2) {
                const bool in = off[0] >= 0 && zg >= 0;
                const unsigned r = in ? (unsigned)off[0] + nxy * (unsigned)zg : 0u;
                const unsigned n = in ? 16u : 0u;
                if (half == 0) {
#pragma unroll
                    for (int c = 0; c < 5; ++c) cp_async16_zfill(&sm.tau[s4][c][dpos], tau_in(c) + r, n);
                } else {
                    cp_async16_zfill(&sm.tau[s4][5][dpos], tau_in(5) + r, n);
#pragma unroll
                    for (int j = 0; j < 3; ++j) cp_async16_zfill(&sm.u[s4][j][dpos], u_in(j) + r, n);
                }
            }
        } else {
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                const int k = tid + q * NT;
                if (q > 0 && k >= FVH_N) continue;
                // a halo cell beyond a closed side is zero-filled by the copy itself
                const bool in = off[q] >= 0 && zg >= 0;
                const unsigned r = in ? (unsigned)off[q] + nxy * (unsigned)zg : 0u;
                const unsigned n = in ? (unsigned)sizeof(R) : 0u;
#pragma unroll
                for (int c = 0; c < 6; ++c) cp_async_real_zfill<R>(&sm.tau[s4][c][k], tau_in(c) + r, n);
#pragma unroll
                for (int j = 0; j < 3; ++j) cp_async_real_zfill<R>(&sm.u[s4][j][k], u_in(j) + r, n);
            }
        }
        cp_async_commit();
    };
    const int ti = tid % TX, tj = tid / TX;
    const int x = x0 + ti, y = y0 + tj;
    const int kc = (ti + XO) + (tj + 1) * FVH_X;
    const bool own = x < a.g.nx && y < a.g.ny;
#pragma unroll
    for (int q = -1; q <= LBVE_FV_AHEAD; ++q) stage(z0 + q);
    // the mask of the next plane is fetched one plane ahead
    uint32_t m_next = own ? a.mask[(unsigned)x + nx * (unsigned)y + nxy * (unsigned)z0] : 1u;
#pragma unroll 1
    for (int z = z0; z < z1; ++z) {
        const uint32_t m = m_next;
        if (own && z + 1 < z1) m_next = a.mask[(unsigned)x + nx * (unsigned)y + nxy * (unsigned)(z + 1)];
        // planes up to z + 1 have landed; behind the barrier plane z - 1 is done with in the
        // whole block, so plane z + 1 + AHEAD may take the slot of plane z - 2 and arrives
        // while plane z is updated: one barrier per plane
        cp_async_wait_all();
        __syncthreads();
        if (z + 1 + LBVE_FV_AHEAD <= z1) stage(z + 1 + LBVE_FV_AHEAD);
        if (z + 1 == z1) step_next();
        if (own) {
            const unsigned r = (unsigned)x + nx * (unsigned)y + nxy * (unsigned)z;
            R out[6];
            if (m & 1u) {
#pragma unroll
                for (int c = 0; c < 6; ++c) out[c] = R(0);
            } else {
                const int sc = fv_slot(z), sd = fv_slot(z - 1), su = fv_slot(z + 1);
                R tr[6], ur[3];
#pragma unroll
                for (int c = 0; c < 6; ++c) tr[c] = sm.tau[sc][c][kc];
#pragma unroll
                for (int j = 0; j < 3; ++j) ur[j] = sm.u[sc][j][kc];
                const FvSmemNb<S, FVH_X, FVH_N> nb{sm, sc, sd, su, kc};
                fv_core<R, SH, VAR>(a.ph, tr, ur, m, nb, out);
            }
#pragma unroll
            for (int c = 0; c < 6; ++c) tau_out(c)[r] = out[c];
        }
    }
}

template <class S, bool VAR, bool ZR = false, bool W16 = false>
__global__ void __launch_bounds__(FV_X * FV_Y, LBVE_FV_MIN_BLOCKS) k_fv_tiled(KArgs<S> a, int zchunk) {
    using R = typename Store<S>::R;
    step_wait();
    extern __shared__ __align__(16) unsigned char fv_smem_raw[];
    using Sm = FvSmem<R, FvTile<FV_X, W16>::HN>;
    Sm &sm = *reinterpret_cast<Sm *>(fv_smem_raw);
    fv_tile<S, FV_X, VAR, ZR, W16, true>(a, sm, blockIdx.x, zchunk);
}

// ---------------------------------------------------------------------------------
// Two-cell stress update (the shifted modes' plain build: flux and source on, no
// variant).  As k_fv_tiled, a block marches a column through a z-chunk with the tau and u
// planes (one-cell halo in y, four cells in x: whole 16-byte chunks) staged in a
// four-plane shared-memory ring one plane ahead; the column is 64 x 8 cells and each of
// the 256 threads updates the cells x, x + 1 of one row in the two lanes of fv_core_sh
// (paired FP32 instructions), so the results are bitwise those of k_fv_tiled.
// ---------------------------------------------------------------------------------
constexpr int FP_TX = 64, FP_TY = 8, FP_NT = 256;
constexpr int FP_XO = 4, FP_HX = FP_TX + 2 * FP_XO, FP_HY = FP_TY + 2, FP_HN = FP_HX * FP_HY;
constexpr int FP_CPR = FP_HX / 4, FP_CH = FP_CPR * FP_HY;  // 16-byte chunks per halo row, per plane
struct FvPairSmem {
    float tau[FV_RING][6][FP_HN];
    float u[FV_RING][3][FP_HN];
};

template <class S, bool ZR>
__global__ void __launch_bounds__(FP_NT, 2) k_fv_pair(KArgs<S> a, int zchunk) {
    static_assert(Store<S>::shifted, "two-cell stress update: FP32 stress");
    step_wait();
    extern __shared__ __align__(16) unsigned char fp_smem_raw[];
    FvPairSmem &sm = *reinterpret_cast<FvPairSmem *>(fp_smem_raw);
    const int tid = threadIdx.x;
    const int nx = a.g.nx, ny = a.g.ny;
    const int tiles_x = (nx + FP_TX - 1) / FP_TX, tiles_y = (ny + FP_TY - 1) / FP_TY;
    const int item = blockIdx.x;
    const int tx = item % tiles_x, ty = (item / tiles_x) % tiles_y, zc = item / (tiles_x * tiles_y);
    const int x0 = tx * FP_TX, y0 = ty * FP_TY;
    const int z0 = ZR ? a.zlo + zc * zchunk : zc * zchunk;
    const int z1 = ZR ? min(a.zhi, z0 + zchunk) : min(a.g.nz, z0 + zchunk);
    const unsigned nxu = (unsigned)nx, nxy = (unsigned)nx * (unsigned)ny;
    // staging: chunk positions tid and tid + FP_NT of 2 FP_CH (the first FP_CH carry tau
    // components 0..4, the others component 5 and u); -1 beyond a closed side
    int off[2], dpos[2], half[2];
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        const int p = tid + q * FP_NT;
        half[q] = p < 2 * FP_CH ? p / FP_CH : 2;
        off[q] = -1;
        dpos[q] = 0;
        if (half[q] < 2) {
            const int pp = p - half[q] * FP_CH, row = pp / FP_CPR, cq = pp - row * FP_CPR;
            dpos[q] = row * FP_HX + 4 * cq;
            const int xg = side_coord(x0 - FP_XO + 4 * cq, nx, a.g.per[0]);
            const int yg = side_coord(y0 - 1 + row, ny, a.g.per[1]);
            if (xg >= 0 && yg >= 0) off[q] = xg + nx * yg;
        }
    }
    auto stage = [&](int zz) {
        const int zg = side_coord(zz, a.g.nz, a.g.per[2]);
        const int s4 = fv_slot(zz);
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            if (half[q] >= 2) continue;
            const bool in = off[q] >= 0 && zg >= 0;
            const unsigned r = in ? (unsigned)off[q] + nxy * (unsigned)zg : 0u;
            const unsigned n = in ? 16u : 0u;
            if (half[q] == 0) {
#pragma unroll
                for (int c = 0; c < 5; ++c) cp_async16_zfill(&sm.tau[s4][c][dpos[q]], a.tq[c] + r, n);
            } else {
                cp_async16_zfill(&sm.tau[s4][5][dpos[q]], a.tq[5] + r, n);
#pragma unroll
                for (int j = 0; j < 3; ++j) cp_async16_zfill(&sm.u[s4][j][dpos[q]], a.uiq[j] + r, n);
            }
        }
        cp_async_commit();
    };
    const int ti = tid % (FP_TX / 2), tj = tid / (FP_TX / 2);
    const int x = x0 + 2 * ti, y = y0 + tj;
    const int kc = (2 * ti + FP_XO) + (tj + 1) * FP_HX;
    const bool own = x < nx && y < ny;  // nx is a multiple of 4: x + 1 < nx too
#pragma unroll
    for (int q = -1; q <= LBVE_FV_AHEAD; ++q) stage(z0 + q);
    auto mask2 = [&](int zz) { return *reinterpret_cast<const uint2 *>(a.mask + ((unsigned)x + nxu * (unsigned)y + nxy * (unsigned)zz)); };
    uint2 m_next = own ? mask2(z0) : make_uint2(1u, 1u);
#pragma unroll 1
    for (int z = z0; z < z1; ++z) {
        const uint2 m = m_next;
        if (own && z + 1 < z1) m_next = mask2(z + 1);
        // one barrier per plane, as in fv_tile
        cp_async_wait_all();
        __syncthreads();
        if (z + 1 + LBVE_FV_AHEAD <= z1) stage(z + 1 + LBVE_FV_AHEAD);
        if (z + 1 == z1) step_next();
        if (own) {
            const unsigned r = (unsigned)x + nxu * (unsigned)y + nxy * (unsigned)z;
            const bool fa = !(m.x & 1u), fb = !(m.y & 1u);
            float2 out[6];
            if (fa || fb) {
                const int sc = fv_slot(z), sd = fv_slot(z - 1), su = fv_slot(z + 1);
                auto ld2 = [](const float *p) { return *reinterpret_cast<const float2 *>(p); };
                float2 tr[6], ur[3];
#pragma unroll
                for (int c = 0; c < 6; ++c) tr[c] = ld2(&sm.tau[sc][c][kc]);
#pragma unroll
                for (int j = 0; j < 3; ++j) ur[j] = ld2(&sm.u[sc][j][kc]);
                struct Nb {
                    const FvPairSmem &sm;
                    const float2 (&tr)[6];
                    const float2 (&ur)[3];
                    int sc, sd, su, kc;
                    __device__ __forceinline__ float2 val(const float (*pl)[FP_HN], int l, int q, float2 own2,
                                                          const float (*pd)[FP_HN], const float (*pu)[FP_HN]) const {
                        switch (l) {
                            case 0: return make_float2(own2.y, pl[q][kc + 2]);
                            case 1: return make_float2(pl[q][kc - 1], own2.x);
                            case 2: return *reinterpret_cast<const float2 *>(&pl[q][kc + FP_HX]);
                            case 3: return *reinterpret_cast<const float2 *>(&pl[q][kc - FP_HX]);
                            case 4: return *reinterpret_cast<const float2 *>(&pu[q][kc]);
                            default: return *reinterpret_cast<const float2 *>(&pd[q][kc]);
                        }
                    }
                    __device__ __forceinline__ float2 u(int l, int k) const {
                        return val(sm.u[sc], l, k, ur[k], sm.u[sd], sm.u[su]);
                    }
                    __device__ __forceinline__ float2 tau(int l, int c) const {
                        return val(sm.tau[sc], l, c, tr[c], sm.tau[sd], sm.tau[su]);
                    }
                };
                const Nb nb{sm, tr, ur, sc, sd, su, kc};
                fv_core_sh<float2, uint2, false>(a.ph, tr, ur, m, nb, out);
#pragma unroll
                for (int c = 0; c < 6; ++c) out[c] = make_float2(fa ? out[c].x : 0.0f, fb ? out[c].y : 0.0f);
            } else {
#pragma unroll
                for (int c = 0; c < 6; ++c) out[c] = make_float2(0.0f, 0.0f);
            }
#pragma unroll
            for (int c = 0; c < 6; ++c) *reinterpret_cast<float2 *>(a.toq[c] + r) = out[c];
        }
    }
}

// ---------------------------------------------------------------------------------
// batched schedule: the resident solves of a pool advance together.  Each kernel is a
// persistent grid over a packed list of work items (solve, block); a block reads the
// solve's descriptor into shared memory and runs the same per-cell code as the
// single-solve kernels, so every cell's arithmetic is the same alone and in the mix.
// ---------------------------------------------------------------------------------
constexpr int BLB_X = 32, BLB_Y = 4;  // cells per stream-collide work item

template <class S>
struct BatchEntry {
    KArgs<S> a[2];   // arguments for even / odd steps k of a launch sequence (k odd swaps
                     // the stress / velocity ping-pong), pointers linked on the host
    int parity0;     // AA parity at k = 0
    int lb_first, lb_items;
    int fv_first, fv_items, fv_zchunk;
    int lb_tx;       // stream-collide tile: lb_tx x (128 / lb_tx) cells (16, 32, 64, 128)
    int fv_tx;       // stress tile: fv_tx x (256 / fv_tx) cells (16, 32, 64; 32 for FP64)
};

// Stress tile widths the batched kernels support for real type R (FP64: 32 x 8 only,
// which keeps 2 blocks per SM).
template <class R>
struct FvBatchTiles {
    static constexpr bool wide = sizeof(R) == 4;
    __host__ __device__ static bool ok(int tx) { return tx == 32 || (wide && (tx == 16 || tx == 64)); }
};

// the entry whose [first, first + items) range holds work item `it` (binary search)
template <class S>
__device__ __forceinline__ int batch_find(const BatchEntry<S> *__restrict__ e, int n, int it, bool fv) {
    int lo = 0, hi = n - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        const int first = fv ? e[mid].fv_first : e[mid].lb_first;
        if (first <= it)
            lo = mid;
        else
            hi = mid - 1;
    }
    return lo;
}

// Cooperative copy of a solve's arguments for step k into shared memory (all threads).
// The step index word gets `dstep` added: the steps the pool has taken since the
// arguments were built.
template <class S>
__device__ __forceinline__ void batch_load(KArgs<S> &sa, const BatchEntry<S> &e, int k, unsigned dstep, int tid,
                                           int nt) {
    static_assert(sizeof(KArgs<S>) % 4 == 0, "argument block copied as words");
    static_assert(offsetof(KArgs<S>, step) % 4 == 0, "step index is one word");
    constexpr int ws = (int)(offsetof(KArgs<S>, step) / 4);
    const unsigned *src = reinterpret_cast<const unsigned *>(&e.a[k & 1]);
    unsigned *dst = reinterpret_cast<unsigned *>(&sa);
    for (int w = tid; w < (int)(sizeof(KArgs<S>) / 4); w += nt) dst[w] = w == ws ? src[w] + dstep : src[w];
}

// Stream-collide over solves that all take AA parity PAR at this step (the pool keeps its
// members in two lists by parity and launches one kernel per list and step).
template <class S, int PAR>
__global__ void __launch_bounds__(BLB_X * BLB_Y, LBVE_LBB_MIN_BLOCKS) k_lb_batched(const BatchEntry<S> *__restrict__ e,
                                                                                 int nsolves, int total, int k,
                                                                                 const unsigned *__restrict__ dstep) {
    __shared__ KArgs<S> sa;
    const int tid = threadIdx.x;  // 1-D blocks of BLB_X * BLB_Y threads
    // items blockIdx.x, + gridDim.x, ...: the resident blocks sweep neighbouring tiles
    // together (halos shared through L2); a block's items only increase, so its solve
    // advances by a forward scan
    if ((int)blockIdx.x >= total) return;
    const unsigned ds = *dstep;
    int sv = batch_find<S>(e, nsolves, blockIdx.x, false), end = -1, first = 0, lx = 5;
    for (int it = blockIdx.x; it < total; it += gridDim.x) {
        if (it >= end) {
            while (it >= e[sv].lb_first + e[sv].lb_items) ++sv;
            first = e[sv].lb_first;
            end = first + e[sv].lb_items;
            lx = __ffs(e[sv].lb_tx) - 1;  // log2 of the tile width
            __syncthreads();  // every thread is done with the previous solve's arguments
            batch_load<S>(sa, e[sv], k, ds, tid, BLB_X * BLB_Y);
            __syncthreads();
        }
        const int local = it - first;
        const int tw = 1 << lx, th = (BLB_X * BLB_Y) >> lx;
        const int tiles_x = (sa.g.nx + tw - 1) >> lx, tiles_y = (sa.g.ny + th - 1) / th;
        const int bx = local % tiles_x, by = (local / tiles_x) % tiles_y, z = local / (tiles_x * tiles_y);
        const int x = (bx << lx) + (tid & (tw - 1)), y = by * th + (tid >> lx);
        if (x < sa.g.nx && y < sa.g.ny) lb_cell_at<S, PAR>(sa, x, y, z);
    }
}

// Batched stress update over the solves whose stress tile is TX wide (the pool launches
// one of these per tile width present; fv_first counts within that group).  VAR when a
// solve of the group uses a finite-volume variant (the others compute as without it).
template <class S, int TX, bool VAR>
__global__ void __launch_bounds__(FV_NT, sizeof(typename Store<S>::R) == 8 ? 2 : LBVE_FV_MIN_BLOCKS) k_fv_batched(
    const BatchEntry<S> *__restrict__ e, int nsolves, int total, int k) {
    using R = typename Store<S>::R;
    extern __shared__ __align__(16) unsigned char fv_smem_raw[];
    FvSmem<R, FvTile<TX>::HN> &sm = *reinterpret_cast<FvSmem<R, FvTile<TX>::HN> *>(fv_smem_raw);
    __shared__ KArgs<S> sa;
    if ((int)blockIdx.x >= total) return;
    int sv = batch_find<S>(e, nsolves, blockIdx.x, true), end = -1, first = 0, zchunk = 1;
    for (int it = blockIdx.x; it < total; it += gridDim.x) {
        if (it >= end) {
            while (it >= e[sv].fv_first + e[sv].fv_items) ++sv;
            first = e[sv].fv_first;
            end = first + e[sv].fv_items;
            zchunk = e[sv].fv_zchunk;
            __syncthreads();
            batch_load<S>(sa, e[sv], k, 0u, threadIdx.x, FV_NT);  // the stress update uses no step index
            __syncthreads();
        }
        fv_tile<S, TX, VAR>(sa, sm, it - first, zchunk);
        __syncthreads();
    }
}

// Residual of one solve: sums over fluid cells of |u - u_snap|^2 and |u|^2 (FP64,
// fixed-shape block partials), then u_snap = u.
template <class S>
__global__ void __launch_bounds__(256) k_residual(Geo g, const uint32_t *__restrict__ mask,
                                                  const typename Store<S>::R *__restrict__ u,
                                                  typename Store<S>::R *__restrict__ usnap, double *__restrict__ partial) {
    const size_t np = (size_t)g.np;
    double d2 = 0.0, u2 = 0.0;
    for (long long r = (long long)blockIdx.x * blockDim.x + threadIdx.x; r < g.n; r += (long long)gridDim.x * blockDim.x) {
        if (mask[r] & 1u) continue;
        for (int j = 0; j < 3; ++j) {
            const double v = (double)u[j * np + r], w = (double)usnap[j * np + r];
            d2 += (v - w) * (v - w);
            u2 += v * v;
            usnap[j * np + r] = u[j * np + r];
        }
    }
    __shared__ double sh[2][256];
    sh[0][threadIdx.x] = d2;
    sh[1][threadIdx.x] = u2;
    __syncthreads();
    for (int s = 128; s > 0; s >>= 1) {
        if ((int)threadIdx.x < s) {
            sh[0][threadIdx.x] += sh[0][threadIdx.x + s];
            sh[1][threadIdx.x] += sh[1][threadIdx.x + s];
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        partial[2 * blockIdx.x] = sh[0][0];
        partial[2 * blockIdx.x + 1] = sh[1][0];
    }
}

// ---------------------------------------------------------------------------------
// momentum exchange (Sec. "Moving boundaries"): for every link (fluid cell r,
// direction i into a tracked solid cell) the force c_i (2 f*_i - 6 w_i rho c_i.u_b) and
// its torque about the owning particle.  Runs before k_lb on the same f^t and repeats
// the cell's collision, so f*_i is exactly the value k_lb streams.
// ---------------------------------------------------------------------------------
// Momentum-exchange contribution of one link (code = r << 5 | i) into contrib[8].
template <class S, int PAR>
__device__ __forceinline__ void me_link(const KArgs<S> &a, long long code, double *o) {
    using R = typename Store<S>::R;
    constexpr bool SH = Store<S>::shifted;
    const int i = (int)(code & 31);
    const unsigned r = (unsigned)(code >> 5);
    const int x = (int)(r % a.g.nx), y = (int)((r / a.g.nx) % a.g.ny), z = (int)(r / ((unsigned)a.g.nx * a.g.ny));
    const Cell cl(a.g, x, y, z);
    R f[Q];
    load_pdfs<S, PAR>(a, cl, r, f);
    R Fp[3], F[3], u[3], rho, drho;
    polymer_force<R>(a.g, a.ph, cl, r, a.mask[r], a.tau, Fp);
#pragma unroll
    for (int k = 0; k < 3; ++k) F[k] = a.ph.g[k] + Fp[k];
    moments<R, SH>(f, F, a.ph.rho0, rho, drho, u);
    collide<R, SH>(f, rho, drho, u, F, a.ph);
    // f*_i (a full population: the stored deviation plus w_i rho0 in shifted modes)
    R fsi = R(0);
    int ci[3] = {0, 0, 0};
#pragma unroll
    for (int k = 1; k < Q; ++k)
        if (k == i) {
            fsi = f[k];
            ci[0] = cx(k);
            ci[1] = cy(k);
            ci[2] = cz(k);
        }
    const int xb = cl.X(ci[0]), yb = cl.Y(ci[1]), zb = cl.Z(ci[2]);
    const unsigned nb = (unsigned)xb + (unsigned)a.g.nx * ((unsigned)yb + (unsigned)a.g.ny * (unsigned)zb);
    const int fl = a.flag[nb];
    R ub[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) ub[k] = a.uq[k][nb];
    R cub = R(0);
    {
        bool first = true;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            if (ci[k] != 0) {
                if (first) {
                    cub = ci[k] > 0 ? ub[k] : -ub[k];
                    first = false;
                } else {
                    cub = ci[k] > 0 ? cub + ub[k] : cub - ub[k];
                }
            }
        }
    }
    const R wi = i < 7 ? wgt<R>(1) : wgt<R>(7);
    const R X = R(6) * wi * rho * cub;
    double m;
    if constexpr (SH)
        m = 2.0 * ((double)fsi + (double)(i < 7 ? wgt<double>(1) : wgt<double>(7)) * (double)a.ph.rho0) - (double)X;
    else
        m = 2.0 * fsi - X;
    const double Fl[3] = {ci[0] * m, ci[1] * m, ci[2] * m};
    double T[3] = {0.0, 0.0, 0.0};
    if (fl >= FLAG_PART0 && fl < FLAG_PART0 + MAX_PART) {
        const PartDev &P = a.parts[fl - FLAG_PART0];
        double q[3] = {(double)xb, (double)yb, (double)zb}, d[3];
        int nn[3] = {a.g.nx, a.g.ny, a.g.nz};
        for (int k = 0; k < 3; ++k) {
            d[k] = q[k] - P.X[k];
            if (a.g.per[k]) d[k] = min_image_1d(d[k], nn[k]);
        }
        T[0] = d[1] * Fl[2] - d[2] * Fl[1];
        T[1] = d[2] * Fl[0] - d[0] * Fl[2];
        T[2] = d[0] * Fl[1] - d[1] * Fl[0];
    }
    o[0] = Fl[0];
    o[1] = Fl[1];
    o[2] = Fl[2];
    o[3] = T[0];
    o[4] = T[1];
    o[5] = T[2];
    o[6] = (double)fl;
}

// Momentum exchange over link segments (one segment per tracked body, blockIdx.y):
// link l of segment b is links[seg_begin[b] + l] for l < seg_count[b].
template <class S, int PAR>
__global__ void __launch_bounds__(128) k_momentum_exchange(KArgs<S> a, const long long *links,
                                                           const int *__restrict__ seg_begin, const int *seg_count,
                                                           double *contrib) {
    step_wait();
    const int b = blockIdx.y;
    const int l = blockIdx.x * blockDim.x + threadIdx.x;
    if (l >= seg_count[b]) return;
    const long long at = (long long)seg_begin[b] + l;
    me_link<S, PAR>(a, links[at], contrib + at * 8);
}

// Same with the links of a block summed inside the block (fixed tree order): one partial
// of 6 doubles (stride 8) per (body, block) at part[(b * gridDim.x + block) * 8].  The
// final per-body sum then reads ceil(count / 128) partials instead of every link.
template <class S, int PAR>
__global__ void __launch_bounds__(128) k_momentum_exchange_part(KArgs<S> a, const long long *links,
                                                                const int *__restrict__ seg_begin,
                                                                const int *seg_count, double *part) {
    step_wait();
    step_next();
    const int b = blockIdx.y;
    const int cnt = seg_count[b];
    if ((int)blockIdx.x * 128 >= cnt) return;  // the whole block is past this body's links
    const int l = blockIdx.x * 128 + threadIdx.x;
    double o[8] = {0, 0, 0, 0, 0, 0, 0, 0};
    if (l < cnt) me_link<S, PAR>(a, links[(long long)seg_begin[b] + l], o);
    __shared__ double sh[6][128];
#pragma unroll
    for (int k = 0; k < 6; ++k) sh[k][threadIdx.x] = o[k];
    __syncthreads();
    // a warp per component: halves added until one value is left
    const int lane = (int)threadIdx.x & 31;
#pragma unroll 1
    for (int k = (int)threadIdx.x >> 5; k < 6; k += 4) {
        double v = (sh[k][lane] + sh[k][lane + 64]) + (sh[k][lane + 32] + sh[k][lane + 96]);
#pragma unroll
        for (int s = 16; s > 0; s >>= 1) v += __shfl_down_sync(0xffffffffu, v, s);
        if (lane == 0) part[((long long)b * gridDim.x + blockIdx.x) * 8 + k] = v;
    }
}

// ---------------------------------------------------------------------------------
// initialisation, read-back and reductions
// ---------------------------------------------------------------------------------

// f = f^eq(rho, u) of Eq. (lb-equilibrium) in the even-step layout; tau copied.  Works on
// the cells r0 .. r0+count-1; the inputs hold those cells with leading dimension ld.
template <class S>
__global__ void k_init(KArgs<S> a, const double *__restrict__ rho_in, const double *__restrict__ u_in,
                       const double *__restrict__ tau_in, typename Store<S>::R *__restrict__ tau_dst, long long r0,
                       long long count, long long ld) {
    using R = typename Store<S>::R;
    const long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= count) return;
    const long long r = r0 + k;
    const double rho = rho_in ? rho_in[k] : (double)a.ph.rho_ref;
    double u[3] = {0.0, 0.0, 0.0};
    if (u_in)
        for (int j = 0; j < 3; ++j) u[j] = u_in[j * ld + k];
    const double usq = u[0] * u[0] + u[1] * u[1] + u[2] * u[2];
#pragma unroll
    for (int i = 0; i < Q; ++i) {
        const double cu = (double)cx(i) * u[0] + (double)cy(i) * u[1] + (double)cz(i) * u[2];
        double v;
        if constexpr (!Store<S>::shifted) {
            v = wgt<double>(i) * rho * (1.0 + 3.0 * cu + 4.5 * cu * cu - 1.5 * usq);
        } else {
            // deviation from w_i rho0, evaluated without forming f_i first
            v = wgt<double>(i) * ((rho - (double)a.ph.rho0) + rho * (3.0 * cu + 4.5 * cu * cu - 1.5 * usq));
        }
        Store<S>::st(a.f + (long long)i * a.g.np + r, (R)v, a.ph.scale);
    }
    double t6[6];
    const bool solid = a.mask[r] & 1u;  // a solid cell carries no stress
    for (int c = 0; c < 6; ++c) t6[c] = (tau_in && !solid) ? tau_in[c * ld + k] : 0.0;
    if (a.ph.fene && !solid) {
        // FENE-P: the conformation of the given stress, A = (I + lambda tau / eta_p) / f with
        // f = 1 + (3 + lambda tr tau / eta_p) / L^2
        const double lam = (double)a.ph.lam, eta_p = (double)a.ph.eta_p;
        const double s = 3.0 + lam * (t6[0] + t6[1] + t6[2]) / eta_p;
        const double f = 1.0 + s / (double)a.ph.fene_L2;
        for (int c = 0; c < 6; ++c) t6[c] = ((c < 3 ? 1.0 : 0.0) + lam * t6[c] / eta_p) / f;
    }
    for (int c = 0; c < 6; ++c) tau_dst[c * a.g.np + r] = (R)t6[c];
}

// rho, physical u and tau of the a.lin cells from plane a.zlo on, 0 in non-fluid cells;
// FP64 outputs indexed from the first of them with leading dimension ld.
template <class S, int PAR, bool LIN>
__global__ void __launch_bounds__(128) k_read(KArgs<S> a, double *__restrict__ rho_out, double *__restrict__ u_out,
                                              double *__restrict__ tau_out, long long ld) {
    using R = typename Store<S>::R;
    constexpr bool SH = Store<S>::shifted;
    step_wait();
    int x, y, z;
    if (!cell_of_thread<S, LIN>(a, x, y, z)) return;
    const Cell cl(a.g, x, y, z);
    const unsigned r = cl.self();
    const long long k = (long long)r - (long long)a.zlo * a.g.nx * a.g.ny;
    // the loads go out together with the mask, as in the stream-collide
    R f[Q], tr[6];
    load_pdfs<S, PAR>(a, cl, r, f);
#pragma unroll
    for (int c = 0; c < 6; ++c) tr[c] = a.tq[c][r];
    const uint32_t m = a.mask[r];
    if (m & 1u) {
        if (rho_out) rho_out[k] = 0.0;
        for (int j = 0; j < 3; ++j)
            if (u_out) u_out[j * ld + k] = 0.0;
        for (int c = 0; c < 6; ++c)
            if (tau_out) tau_out[c * ld + k] = 0.0;
        return;
    }
    auto tn = [&](int l, int c) -> R {
        const int q = l >> 1, s = (l & 1) ? -1 : 1;
        return a.tq[c][cl.idx(q == 0 ? s : 0, q == 1 ? s : 0, q == 2 ? s : 0)];
    };
    R Fp[3], F[3], u[3], rho, drho;
    if (a.ph.fene)
        polymer_force_core_fene<R>(tr, m, tn, a.ph, Fp);
    else
        polymer_force_core<R>(tr, m, tn, Fp);
#pragma unroll
    for (int j = 0; j < 3; ++j) F[j] = a.ph.g[j] + Fp[j];
    moments<R, SH>(f, F, a.ph.rho0, rho, drho, u);
    if (rho_out) rho_out[k] = SH ? (double)a.ph.rho0 + (double)drho : (double)rho;
    if (u_out)
#pragma unroll
        for (int j = 0; j < 3; ++j) u_out[j * ld + k] = (double)u[j];
    if (tau_out)
#pragma unroll
        for (int c = 0; c < 6; ++c) tau_out[c * ld + k] = (double)stored_to_stress<R>(a.ph, tr, c);
}

// PDFs of every cell to / from unshifted FP64 in the plain (pre-collision) layout.
template <class S, int PAR>
__global__ void k_pdfs_io(KArgs<S> a, double *__restrict__ io, int write) {
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    if (x >= a.g.nx) return;
    const Cell cl(a.g, x, blockIdx.y, blockIdx.z);
    const unsigned r = cl.self();
    const long long np = a.g.np, n = a.g.n;
#pragma unroll
    for (int i = 0; i < Q; ++i) {
        S *p = PAR == 0 ? a.f + (long long)i * np + r : a.f + (long long)copp(i) * np + cl.idx(-cx(i), -cy(i), -cz(i));
        const double base = Store<S>::shifted ? wgt<double>(i) * (double)a.ph.rho0 : 0.0;
        if (write) {
            Store<S>::st(p, (typename Store<S>::R)(io[i * n + r] - base), a.ph.scale);
        } else {
            io[i * n + r] = base + (double)Store<S>::ld(p, a.ph.inv_scale);
        }
    }
}

// Probe listed cells: 19 unshifted PDFs, rho, physical u, tau (29 doubles per cell).
template <class S, int PAR>
__global__ void k_probe(KArgs<S> a, const long long *__restrict__ cells, int count, double *__restrict__ out) {
    using R = typename Store<S>::R;
    constexpr bool SH = Store<S>::shifted;
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= count) return;
    const unsigned r = (unsigned)cells[k];
    const int x = (int)(r % a.g.nx), y = (int)((r / a.g.nx) % a.g.ny), z = (int)(r / ((unsigned)a.g.nx * a.g.ny));
    const Cell cl(a.g, x, y, z);
    R f[Q];
    load_pdfs<S, PAR>(a, cl, r, f);
    double *o = out + (long long)k * 29;
    for (int i = 0; i < Q; ++i) o[i] = (double)f[i] + (SH ? wgt<double>(i) * (double)a.ph.rho0 : 0.0);
    for (int j = 19; j < 29; ++j) o[j] = 0.0;
    if (a.flag[r] != FLAG_FLUID) return;
    R Fp[3], F[3], u[3], rho, drho;
    polymer_force<R>(a.g, a.ph, cl, r, a.mask[r], a.tau, Fp);
    for (int j = 0; j < 3; ++j) F[j] = a.ph.g[j] + Fp[j];
    moments<R, SH>(f, F, a.ph.rho0, rho, drho, u);
    o[19] = SH ? (double)a.ph.rho0 + (double)drho : (double)rho;
    for (int j = 0; j < 3; ++j) o[20 + j] = (double)u[j];
    R t6[6];
    for (int c = 0; c < 6; ++c) t6[c] = a.tau[c * a.g.np + r];
    for (int c = 0; c < 6; ++c) o[23 + c] = (double)stored_to_stress<R>(a.ph, t6, c);
}

// Per-block FP64 partial sums over fluid cells: mass, momentum, count, bad-value flag.
template <class S, int PAR>
__global__ void __launch_bounds__(256) k_reduce(KArgs<S> a, double *__restrict__ partial) {
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    double v[6] = {0, 0, 0, 0, 0, 0};
    if (x < a.g.nx) {
        const Cell cl(a.g, x, blockIdx.y, blockIdx.z);
        const unsigned r = cl.self();
        if (a.flag[r] == FLAG_FLUID && (int)blockIdx.z >= a.zlo && (int)blockIdx.z < a.zhi) {
            typename Store<S>::R f[Q];
            load_pdfs<S, PAR>(a, cl, r, f);
            for (int i = 0; i < Q; ++i) {
                const double fi = (double)f[i] + (Store<S>::shifted ? wgt<double>(i) * (double)a.ph.rho0 : 0.0);
                v[0] += fi;
                v[1] += cx(i) * fi;
                v[2] += cy(i) * fi;
                v[3] += cz(i) * fi;
                if (!isfinite(fi)) v[5] = 1.0;
            }
            v[4] = 1.0;
            if (!(v[0] > 0.0)) v[5] = 1.0;
        }
    }
    __shared__ double sh[6][256];
    for (int k = 0; k < 6; ++k) sh[k][threadIdx.x] = v[k];
    __syncthreads();
    for (int s = blockDim.x / 2; s > 0; s >>= 1) {
        if ((int)threadIdx.x < s)
            for (int k = 0; k < 6; ++k)
                sh[k][threadIdx.x] = k == 5 ? fmax(sh[k][threadIdx.x], sh[k][threadIdx.x + s])
                                            : sh[k][threadIdx.x] + sh[k][threadIdx.x + s];
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        const long long b = blockIdx.x + (long long)gridDim.x * (blockIdx.y + (long long)gridDim.y * blockIdx.z);
        for (int k = 0; k < 6; ++k) partial[b * 6 + k] = sh[k][0];
    }
}

// ---------------------------------------------------------------------------------
// z-slab decomposition: halo exchange between the slabs of one domain.  A slab computes
// planes [zlo, zhi) and holds one ghost plane on each side (zlo - 1, zhi) mirroring the
// neighbouring slab's boundary plane (its flags included).  Per step:
//   after the stream-collide: u of the boundary planes -> the neighbours' ghost planes,
//     and the 5 PDFs per cell that cross each face (below);
//   after the stress update: tau of the boundary planes -> the neighbours' ghost planes.
// The PDFs follow the in-place (AA) pattern.  D+ / D- are the directions with c_z = +1 /
// -1 (5 each).  After an even step a fluid cell's slot -i holds its f*_i, which the next
// odd step reads from the cell above (-i in D-, i moving up) or below: the boundary
// plane's slots D- (high side) / D+ (low side) go into the neighbour's ghost plane, for
// fluid ghost cells (a solid ghost cell's slots hold this slab's own bounced values).
// After an odd step a fluid cell has written f*_i into slot i of r + c_i, in the ghost
// plane for i crossing the face: the ghost plane's slots D+ (high side) / D- (low side)
// go into the neighbour's boundary plane, where the source cell r - c_i is fluid (else
// the slot holds that cell's own bounced value).
// ---------------------------------------------------------------------------------
__host__ __device__ constexpr int dir_zp(int k) { return k == 0 ? 5 : k == 1 ? 11 : k == 2 ? 14 : k == 3 ? 15 : 18; }
__host__ __device__ constexpr int dir_zm(int k) { return k == 0 ? 6 : k == 1 ? 12 : k == 2 ? 13 : k == 3 ? 16 : 17; }

__host__ __device__ constexpr int halo_values(int what) { return what == 0 ? 5 : (what == 1 ? 3 : 6); }

// plane and slot set of a PDF pack (side: 0 low, 1 high; parity of the last stream-collide)
__device__ __forceinline__ void halo_f_pack_plan(int side, int parity, int zlo, int zhi, int &z, bool &up) {
    if (parity == 0) {
        z = side ? zhi - 1 : zlo;
        up = side == 0;  // low side sends D+, high side D-
    } else {
        z = side ? zhi : zlo - 1;
        up = side == 1;  // from the ghost planes: high sends D+, low D-
    }
}

template <class S>
__global__ void k_halo_pack(KArgs<S> a, int what, int side, int parity, void *__restrict__ buf) {
    using R = typename Store<S>::R;
    const int x = blockIdx.x * blockDim.x + threadIdx.x, y = blockIdx.y;
    if (x >= a.g.nx) return;
    const long long plane = (long long)a.g.nx * a.g.ny, p = x + (long long)a.g.nx * y;
    const size_t np = (size_t)a.g.np;
    if (what == 0) {
        int z;
        bool up;
        halo_f_pack_plan(side, parity, a.zlo, a.zhi, z, up);
        const unsigned r = (unsigned)(p + plane * z);
        S *o = (S *)buf;
#pragma unroll
        for (int k = 0; k < 5; ++k) o[k * plane + p] = a.f[(up ? dir_zp(k) : dir_zm(k)) * np + r];
    } else {
        const int z = side ? a.zhi - 1 : a.zlo;
        const unsigned r = (unsigned)(p + plane * z);
        R *o = (R *)buf;
        if (what == 1)
            for (int j = 0; j < 3; ++j) o[j * plane + p] = a.u_out[j * np + r];
        else
            for (int c = 0; c < 6; ++c) o[c * plane + p] = a.tau[c * np + r];
    }
}

template <class S>
__global__ void k_halo_unpack(KArgs<S> a, int what, int side, int parity, const void *__restrict__ buf) {
    using R = typename Store<S>::R;
    const int x = blockIdx.x * blockDim.x + threadIdx.x, y = blockIdx.y;
    if (x >= a.g.nx) return;
    const long long plane = (long long)a.g.nx * a.g.ny, p = x + (long long)a.g.nx * y;
    const size_t np = (size_t)a.g.np;
    if (what == 0) {
        const S *in = (const S *)buf;
        if (parity == 0) {
            // into the ghost plane, for fluid ghost cells; the low side receives the lower
            // slab's D-, the high side the upper slab's D+
            const int z = side ? a.zhi : a.zlo - 1;
            const unsigned r = (unsigned)(p + plane * z);
            if (a.flag[r] != FLAG_FLUID) return;
#pragma unroll
            for (int k = 0; k < 5; ++k) a.f[(side ? dir_zp(k) : dir_zm(k)) * np + r] = in[k * plane + p];
        } else {
            // into the boundary plane, where the source cell r - c_i (in the ghost plane) is
            // fluid: the low side receives D+ (moving up from the lower slab), the high
            // side D- (moving down from the upper slab)
            const int z = side ? a.zhi - 1 : a.zlo;
            const unsigned r = (unsigned)(p + plane * z);
            const Cell cl(a.g, x, y, z);
            if (a.flag[r] != FLAG_FLUID) return;
#pragma unroll
            for (int k = 0; k < 5; ++k) {
                const int i = side ? dir_zm(k) : dir_zp(k);
                const int sx = -cx(i), sy = -cy(i);
                const int xs = x + sx, ys = y + sy;
                if ((xs < 0 || xs >= a.g.nx) && !a.g.per[0]) continue;
                if ((ys < 0 || ys >= a.g.ny) && !a.g.per[1]) continue;
                if (a.flag[cl.idx(sx, sy, -cz(i))] != FLAG_FLUID) continue;
                a.f[i * np + r] = in[k * plane + p];
            }
        }
    } else {
        const int z = side ? a.zhi : a.zlo - 1;
        const unsigned r = (unsigned)(p + plane * z);
        const R *in = (const R *)buf;
        if (what == 1)
            for (int j = 0; j < 3; ++j) a.u_out[j * np + r] = in[j * plane + p];
        else
            for (int c = 0; c < 6; ++c) const_cast<R *>(a.tau)[c * np + r] = in[c * plane + p];
    }
}

} // namespace lbve
