// lbve_particles.cuh -- moving rigid spheres (Kuron et al., arXiv:2009.12279, Sec. "Moving
// boundaries"): placement, and the particle phase of a step -- body sums, symplectic
// Euler, re-voxelisation with fill/drain, boundary links -- as one kernel on a
// thread-block cluster per solve.
#pragma once

#include <cooperative_groups.h>

#include "lbve_kernels.cuh"

namespace lbve {

struct BBox {
    int lo[3], ext[3];
    __host__ __device__ long long cells() const { return (long long)ext[0] * ext[1] * ext[2]; }
};

// One side of a particle's box: cells within R + margin of the centre coordinate X (the
// whole side where a periodic one would wrap onto itself; clamped to the domain along a
// closed one).
__host__ __device__ inline void bbox_side(int n, int per, double X, double R, int margin, int &lo, int &ext) {
    lo = (int)floor(X - R) - margin;
    int hi = (int)ceil(X + R) + margin;
    if (!per) {
        lo = lo < 0 ? 0 : lo;
        hi = hi > n - 1 ? n - 1 : hi;
    }
    ext = hi - lo + 1;
    if (ext > n) {
        lo = 0;
        ext = n;
    }
    if (ext < 0) ext = 0;
}
__host__ __device__ inline BBox particle_bbox(const Geo &g, const double X[3], double R, int margin) {
    BBox b;
    const int nn[3] = {g.nx, g.ny, g.nz};
    for (int k = 0; k < 3; ++k) bbox_side(nn[k], g.per[k], X[k], R, margin, b.lo[k], b.ext[k]);
    return b;
}

// A particle's box as the phase walks it: the lower corner wrapped into the domain once, so
// that a cell's coordinate and a cell's place in the box are each one conditional
// correction away.
struct BoxWalk {
    int lo[3], ext[3], cells;
};
__device__ __forceinline__ BoxWalk box_walk(const Geo &g, const BBox &b) {
    BoxWalk w;
    const int nn[3] = {g.nx, g.ny, g.nz};
    for (int k = 0; k < 3; ++k) {
        w.lo[k] = ((b.lo[k] % nn[k]) + nn[k]) % nn[k];
        w.ext[k] = b.ext[k];
    }
    w.cells = (int)b.cells();
    return w;
}
// coordinates of cell k of the box
__device__ __forceinline__ void box_cell(const Geo &g, const BoxWalk &w, int k, int &x, int &y, int &z) {
    const unsigned row = (unsigned)k / (unsigned)w.ext[0], pl = row / (unsigned)w.ext[1];
    x = w.lo[0] + k - (int)row * w.ext[0];
    y = w.lo[1] + (int)row - (int)pl * w.ext[1];
    z = w.lo[2] + (int)pl;
    if (x >= g.nx) x -= g.nx;
    if (y >= g.ny) y -= g.ny;
    if (z >= g.nz) z -= g.nz;
}
__device__ __forceinline__ unsigned cell_index(const Geo &g, int x, int y, int z) {
    return (unsigned)x + (unsigned)g.nx * ((unsigned)y + (unsigned)g.ny * (unsigned)z);
}
// place of the cell (x, y, z) in the box, or -1
__device__ __forceinline__ int box_index(const Geo &g, const BoxWalk &w, int x, int y, int z) {
    int dx = x - w.lo[0], dy = y - w.lo[1], dz = z - w.lo[2];
    if (g.per[0] && dx < 0) dx += g.nx;
    if (g.per[1] && dy < 0) dy += g.ny;
    if (g.per[2] && dz < 0) dz += g.nz;
    if (dx < 0 || dy < 0 || dz < 0 || dx >= w.ext[0] || dy >= w.ext[1] || dz >= w.ext[2]) return -1;
    return dx + w.ext[0] * (dy + w.ext[1] * dz);
}
// (x, y, z) + s e_ax (ax < 3), wrapped; false beyond a closed side
__device__ __forceinline__ bool step_cell(const Geo &g, int l, int &x, int &y, int &z) {
    const int ax = l >> 1, s = (l & 1) ? -1 : 1;
    int &q = ax == 0 ? x : (ax == 1 ? y : z);
    const int n = ax == 0 ? g.nx : (ax == 1 ? g.ny : g.nz);
    q += s;
    if (q >= 0 && q < n) return true;
    if (!g.per[ax]) return false;
    q = q < 0 ? n - 1 : 0;
    return true;
}

__device__ __forceinline__ void min_image(const Geo &g, const double X[3], int x, int y, int z, double d[3]) {
    const double q[3] = {(double)x, (double)y, (double)z};
    const int nn[3] = {g.nx, g.ny, g.nz};
    for (int k = 0; k < 3; ++k) {
        d[k] = q[k] - X[k];
        if (g.per[k]) d[k] = min_image_1d(d[k], nn[k]);
    }
}

// Sphere test |r - X|^2 <= R^2 (minimum image), decided as in FP64 but almost always
// computed in FP32: FP64 issues at a small fraction of the FP32 rate here, and every cell
// of a particle's box is tested each step.  The centre is split into its nearest integer
// and a remainder |X_f| <= 1/2, so r - X has an exact integer part: in the box, where
// |r_k - X_k| <= D = R + 5, the remainder's rounding (2^-26) and the subtraction's
// (2^-24 D) leave each component within 2^-23 D, and the sum of squares, with its own
// roundings and that of R^2, within 2^-18 D^2 of the FP64 value.  Only in that shell (a
// few cells in ten thousand) does the FP64 test decide.  (Working on the coordinates
// themselves needs a shell thousands of times wider, and nearly every warp at the surface
// then ran the FP64 branch: 33 us per step for an R = 8 sphere in one block.)
struct SphereFilter {
    int Xi[3];
    float Xf[3], R2, tol;
    float deep2;  // squared distance below which every neighbour lies inside, too
};
// The box and (sf != nullptr) the filter of a particle, a side per lane of one warp (FP64
// latencies side by side): into shared memory.
__device__ __forceinline__ void prepare_box(const Geo &g, const PartDev &P, int margin, BoxWalk &w, SphereFilter *sf) {
    const int lane = (int)threadIdx.x & 31;
    int ext = 1;
    if (lane < 3) {
        const int n = lane == 0 ? g.nx : (lane == 1 ? g.ny : g.nz), per = g.per[lane];
        const double X = P.X[lane];
        int lo;
        bbox_side(n, per, X, P.R, margin, lo, ext);
        w.lo[lane] = ((lo % n) + n) % n;
        w.ext[lane] = ext;
        if (sf) {
            const double c = rint(X);
            sf->Xf[lane] = (float)(X - c);
            const int i = (int)c;
            sf->Xi[lane] = per ? ((i % n) + n) % n : i;
        }
    } else if (lane == 3 && sf) {
        const double D = P.R + 5.0;
        sf->R2 = (float)(P.R * P.R);
        sf->tol = (float)(D * D * 0x1p-18);
        const float deep = fmaxf((float)P.R - 1.5f, 0.0f);
        sf->deep2 = deep * deep;
    }
    const int e1 = __shfl_sync(0xffffffffu, ext, 1), e2 = __shfl_sync(0xffffffffu, ext, 2);
    if (lane == 0) w.cells = ext * e1 * e2;
}
__device__ __forceinline__ bool inside_sphere(const Geo &g, const PartDev &P, const SphereFilter &f, int x, int y,
                                              int z, float &d2) {
    const int q[3] = {x, y, z}, nn[3] = {g.nx, g.ny, g.nz};
    d2 = 0.0f;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        int i = q[k] - f.Xi[k];
        if (g.per[k]) {
            if (2 * i > nn[k]) i -= nn[k];
            if (2 * i < -nn[k]) i += nn[k];
        }
        const float dk = (float)i - f.Xf[k];
        d2 += dk * dk;
    }
    if (d2 < f.R2 - f.tol) return true;
    if (d2 > f.R2 + f.tol) return false;
    double d[3];
    min_image(g, P.X, x, y, z, d);
    return d[0] * d[0] + d[1] * d[1] + d[2] * d[2] <= P.R * P.R;
}

// Initial placement: covered fluid cells become particle cells, their stress is zeroed.
template <class S>
__global__ void k_voxelise(KArgs<S> a, PartDev *__restrict__ parts, int p, uint8_t *__restrict__ flag,
                           typename Store<S>::R *__restrict__ tau0, typename Store<S>::R *__restrict__ tau1) {
    using R = typename Store<S>::R;
    const PartDev &P = parts[p];
    const BBox b = particle_bbox(a.g, P.X, P.R, 1);
    const BoxWalk w = box_walk(a.g, b);
    for (long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x; k < b.cells(); k += (long long)gridDim.x * blockDim.x) {
        int x, y, z;
        box_cell(a.g, w, (int)k, x, y, z);
        const long long r = cell_index(a.g, x, y, z);
        if (flag[r] != FLAG_FLUID) continue;
        double d[3];
        min_image(a.g, P.X, x, y, z, d);
        if (d[0] * d[0] + d[1] * d[1] + d[2] * d[2] <= P.R * P.R) {
            flag[r] = (uint8_t)(FLAG_PART0 + p);
            for (int c = 0; c < 6; ++c) {
                tau0[c * a.g.np + r] = R(0);
                tau1[c * a.g.np + r] = R(0);
            }
        }
    }
}

// ---------------------------------------------------------------------------------
// particle phase: a cluster of PC thread blocks per solve
// ---------------------------------------------------------------------------------
constexpr int PC = 8, PT = 512, PW = PT / 32;  // blocks per cluster, threads and warps per block

// A solve's particle phase (single solve: a kernel parameter; pool: one entry per member).
template <class S>
struct PartEntry {
    KArgs<S> a[2];   // for even / odd steps k of a launch sequence (the stress ping-pong
                     // after the step's swap), pointers linked on the host
    int parity0;     // AA parity fill/drain works in at k = 0
    int nparts, first_seg;
    PartDev *parts;
    uint8_t *flag;
    uint32_t *mask;
    uint8_t *kind, *nf;
    double *delta, *diag;
    int *conv;
    long long *links;
    const int *seg_begin;
    int *seg_count;
    const int *capacity;
    // momentum-exchange partials of the solve's bodies to sum first (nullptr: already summed)
    const double *sums;
    int sum_stride, nbody;  // partials per body, bodies
    const int *seg_flag;
    double *body_F;
};

// Block-wide exclusive prefix sum of v in thread order; total: the block's sum.
__device__ __forceinline__ int block_scan(int v, int *wsum, int &total) {
    const int lane = (int)threadIdx.x & 31, warp = (int)threadIdx.x >> 5;
    int incl = 0;
    if (__ballot_sync(0xffffffffu, v != 0)) {
        incl = v;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int t = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += t;
        }
    }
    __syncthreads();  // wsum is free
    if (lane == 31) wsum[warp] = incl;
    __syncthreads();
    int before = 0;
    total = 0;
#pragma unroll
    for (int w = 0; w < PW; ++w) {
        const int t = wsum[w];
        if (w < warp) before += t;
        total += t;
    }
    return before + incl - v;
}

// Every block of the cluster learns every block's count (two alternating buffers: a block
// can be at most one exchange ahead of another).
struct ClusterCounts {
    int n[2][PC];
};
__device__ __forceinline__ void cluster_exchange(cooperative_groups::cluster_group &cl, ClusterCounts &c, int buf,
                                                 int mine, int &before, int &total) {
    const int rank = (int)cl.block_rank();
    if (threadIdx.x < PC) cl.map_shared_rank(&c, threadIdx.x)->n[buf][rank] = mine;
    cl.sync();
    before = total = 0;
#pragma unroll
    for (int b = 0; b < PC; ++b) {
        const int t = c.n[buf][b];
        if (b < rank) before += t;
        total += t;
    }
}

// Boundary links of particle p: every (fluid cell r, direction i) with r + c_i covered by
// it, in cell order then direction order.  The blocks of the cluster take consecutive
// ranges of the box; counts first, then the links at their places.  The neighbour masks
// tell the few cells that have a moving neighbour, so the others cost one load.
__device__ __forceinline__ void particle_links(cooperative_groups::cluster_group &cl, const Geo &g, const PartDev &P,
                                               int p, const uint8_t *flag, const uint32_t *mask, long long *links,
                                               const int *seg_begin, int *seg_count, int seg, int cap,
                                               ClusterCounts &counts, int &buf, int *wsum) {
    __shared__ BoxWalk w;
    __syncthreads();
    if (threadIdx.x < 32) prepare_box(g, P, 2, w, nullptr);
    __syncthreads();
    const int rank = (int)cl.block_rank();
    const int per = (w.cells + PC - 1) / PC, lo = min(w.cells, per * rank), hi = min(w.cells, lo + per);
    auto dirs = [&](int k, unsigned &r) -> unsigned {
        int x, y, z;
        box_cell(g, w, k, x, y, z);
        r = cell_index(g, x, y, z);
        const uint32_t m = mask[r];
        if ((m & 1u) || !(m & MASK_MOVING)) return 0u;
        const Cell c(g, x, y, z);
        unsigned d = 0;
        // set bits, six at a time: their flag loads go out together
#pragma unroll 1
        for (uint32_t s = m & 0x7fffeu; s;) {
            int i[6], f[6];
#pragma unroll
            for (int n = 0; n < 6; ++n) {
                i[n] = s ? __ffs(s) - 1 : 0;  // 0: the cell itself, which is fluid
                f[n] = flag[c.idx(cx(i[n]), cy(i[n]), cz(i[n]))];
                s &= s - 1u;
            }
#pragma unroll
            for (int n = 0; n < 6; ++n)
                if (f[n] == FLAG_PART0 + p) d |= 1u << i[n];
        }
        return d;
    };
    // directions of the first KEEP cells of the range, for the second pass
    constexpr int KEEP = 4 * PT;
    __shared__ unsigned keep[KEEP];
    int mine = 0;
#pragma unroll 1
    for (int k = lo + (int)threadIdx.x; k < hi; k += PT) {
        unsigned r;
        const unsigned m = dirs(k, r);
        if (k - lo < KEEP) keep[k - lo] = m;
        mine += __popc(m);
    }
    int total_block;
    block_scan(mine, wsum, total_block);
    int base, total;
    cluster_exchange(cl, counts, buf, total_block, base, total);
    buf ^= 1;
    long long *out = links + seg_begin[seg];
    if (total_block > 0)
#pragma unroll 1
        for (int k0 = lo; k0 < hi; k0 += PT) {
            const int k = k0 + (int)threadIdx.x;
            unsigned r = 0, m = 0;
            if (k < hi) {
                if (k - lo >= KEEP) {
                    m = dirs(k, r);
                } else if ((m = keep[k - lo]) != 0u) {
                    int x, y, z;
                    box_cell(g, w, k, x, y, z);
                    r = cell_index(g, x, y, z);
                }
            }
            int n;
            int pos = base + block_scan(__popc(m), wsum, n);
#pragma unroll 1
            for (; m; m &= m - 1) {
                if (pos < cap) out[pos] = ((long long)r << 5) | (__ffs(m) - 1);
                ++pos;
            }
            base += n;
        }
    if (rank == 0 && threadIdx.x == 0) seg_count[seg] = total < cap ? total : cap;
}

// Links of the particles marked as changed (set-up and restore).
template <class S>
__global__ void __cluster_dims__(PC, 1, 1) __launch_bounds__(PT)
    k_particle_links(Geo g, const PartDev *parts, const uint8_t *flag, const uint32_t *mask, long long *links,
                     const int *seg_begin, int *seg_count, int first_seg, const int *capacity) {
    cooperative_groups::cluster_group cl = cooperative_groups::this_cluster();
    __shared__ ClusterCounts counts;
    __shared__ int wsum[PW];
    int buf = 0;
    const int p = (int)blockIdx.x / PC;
    cl.sync();  // every block of the cluster is running before its shared memory is written
    if (parts[p].changed)
        particle_links(cl, g, parts[p], p, flag, mask, links, seg_begin, seg_count, first_seg + p, capacity[p], counts,
                       buf, wsum);
    cl.sync();  // no block leaves while another may still write to its shared memory
}

// Fill/drain of the listed converted cells of particle p (first block of the cluster).
// kind: 0 other, 1 fluid before and after, 2 destroyed (fluid -> particle), 3 created
// (particle -> fluid).  All stress moves use the pre-conversion stress:
//   destroyed d: each of its N_f stable D3Q7 neighbours gains tau(d)/N_f;
//   created c:   tau(c) = sum of its stable neighbours' tau / (N_f + 1), each of
//                them gives up tau(c)/N_f;
// the deleted / created momentum goes to the particle as an impulse at the cell.
// The work follows the list (a few cells per step), not the box.  It runs once per launch,
// so its time is that of dependent loads and of fetching the code: a warp works on one cell
// (or pair, or mask) with its neighbours, components or directions in the lanes, loads side
// by side, code rolled up (straight-line code for one thread per cell took 67 us for a
// single converted cell, where this takes 27 with the masks).
constexpr int FD_CHUNK = 64, FD_GATHER = 8;  // converted cells per impulse chunk; warps that gather densities
template <class R>
struct FillDrainSmem {
    double pm[FD_CHUNK][6];             // momentum and lever arm of a chunk of converted cells
    R f[FD_GATHER][(Q - 1) * Q + 2];    // PDFs of a created cell's neighbours, per warp
};
template <class S, int PAR>
__device__ __forceinline__ void fill_drain(const PartEntry<S> &E, const KArgs<S> &a, PartDev &P, int p,
                                           const BoxWalk &w, int nconv, FillDrainSmem<typename Store<S>::R> &sm) {
    using R = typename Store<S>::R;
    constexpr bool SH = Store<S>::shifted;
    constexpr unsigned ALL = 0xffffffffu;
    const long long np = a.g.np;
    const int nc = w.cells, tid = (int)threadIdx.x, lane = tid & 31, warp = tid >> 5;
    R *tau = const_cast<R *>(a.tau);
    uint8_t *kind = E.kind, *nf_arr = E.nf, *flag = E.flag;
    double *delta = E.delta;
    const int *conv = E.conv;
    auto kind_of = [&](int x, int y, int z) -> int {
        const int k = box_index(a.g, w, x, y, z);
        if (k >= 0) return kind[k];
        return flag[cell_index(a.g, x, y, z)] == FLAG_FLUID ? 1 : 0;
    };
    // stored location of population i of the cell, in the layout PAR reads
    auto slot = [&](const Cell &c, int i) -> S * {
        return PAR == 0 ? a.f + (long long)i * np + c.self()
                        : a.f + (long long)copp(i) * np + c.idx(-cx(i), -cy(i), -cz(i));
    };
    auto outside = [&](int x, int y, int z, int i) -> bool {
        return (!a.g.per[0] && (x + cx(i) < 0 || x + cx(i) >= a.g.nx)) ||
               (!a.g.per[1] && (y + cy(i) < 0 || y + cy(i) >= a.g.ny)) ||
               (!a.g.per[2] && (z + cz(i) < 0 || z + cz(i) >= a.g.nz));
    };
    // B: N_f of converted cells, new stress of created cells.  Lane l: face l; then lane c:
    // component c, summed in face order.
#pragma unroll 1
    for (int q = warp; q < nconv; q += PW) {
        const int k = conv[q];
        int x, y, z;
        box_cell(a.g, w, k, x, y, z);
        bool stable = false;
        unsigned nb = 0;
        if (lane < 6 && step_cell(a.g, lane, x, y, z)) {
            stable = kind_of(x, y, z) == 1;
            nb = cell_index(a.g, x, y, z);
        }
        const unsigned sb = __ballot_sync(ALL, stable);
        const int nf = __popc(sb), c = lane < 6 ? lane : 0;
        double t[6], sum = 0.0;
#pragma unroll
        for (int l = 0; l < 6; ++l) {
            const unsigned n = __shfl_sync(ALL, nb, l);
            t[l] = (sb >> l) & 1u ? (double)tau[c * np + n] : 0.0;
        }
#pragma unroll
        for (int l = 0; l < 6; ++l)
            if ((sb >> l) & 1u) sum += t[l];
        if (lane == 0) nf_arr[k] = (uint8_t)nf;
        if (lane < 6 && kind[k] == 3) delta[(long long)c * nc + k] = sum / (double)(nf + 1);
    }
    __syncthreads();
    // C: stress gathered by each stable cell from its converted D3Q7 neighbours, face by
    // face.  Pair e = (converted cell, face) stands for the stable cell on that face when
    // the converted cell is the first one in that cell's face order.  First pass: the gains,
    // kept in delta; second pass: added (all gains are formed from the stress before).
#pragma unroll 1
    for (int pass = 0; pass < 2; ++pass) {
#pragma unroll 1
        for (int e = warp; e < 6 * nconv; e += PW) {
            const int q = e / 6, l = e - 6 * q;
            int x, y, z;
            box_cell(a.g, w, conv[q], x, y, z);
            if (!step_cell(a.g, l, x, y, z)) continue;
            const int ks = box_index(a.g, w, x, y, z);
            if (ks < 0 || kind[ks] != 1) continue;
            const unsigned r = cell_index(a.g, x, y, z);
            int kb = -1, kk = 0;
            unsigned nb = 0;
            if (lane < 6 && step_cell(a.g, lane, x, y, z)) {
                kb = box_index(a.g, w, x, y, z);
                kk = kb >= 0 ? kind[kb] : 0;
                nb = cell_index(a.g, x, y, z);
            }
            const unsigned cb = __ballot_sync(ALL, kk >= 2);
            if (__shfl_sync(ALL, kb, __ffs(cb) - 1) != conv[q]) continue;
            const int c = lane < 6 ? lane : 0;
            if (pass == 1) {
                if (lane < 6) tau[c * np + r] = (R)((double)tau[c * np + r] + delta[(long long)c * nc + ks]);
                continue;
            }
            double acc = 0.0;
#pragma unroll 1
            for (unsigned m = cb; m; m &= m - 1u) {
                const int f = __ffs(m) - 1, kf = __shfl_sync(ALL, kb, f);
                const unsigned n = __shfl_sync(ALL, nb, f);
                const bool gone = __shfl_sync(ALL, kk, f) == 2;
                const double v = gone ? (double)tau[c * np + n] : delta[(long long)c * nc + kf];
                const double t = v / (double)nf_arr[kf];
                acc = gone ? acc + t : acc - t;
            }
            if (lane < 6) delta[(long long)c * nc + ks] = acc;
        }
        __syncthreads();
    }
    // D: impulses and the populations of created cells, a warp per converted cell: the
    // momentum of a destroyed cell's deleted populations, or f^eq(rho_bar, u_b) written to
    // a created cell with its momentum.  A created cell reads only stable cells' populations
    // and writes only its own, so the cells are independent.  Thread 0 then adds the
    // momenta to the impulse in the sequential order of the method: destroyed cells in cell
    // order, then created cells in cell order.  Sums over directions run in direction order.
    double dP[3] = {0, 0, 0}, dL[3] = {0, 0, 0};
    const int i = lane < Q ? lane : 0;  // lane i: population or direction i
#pragma unroll 1
    for (int pass = 0; pass < 2; ++pass) {
        const int want = pass == 0 ? 2 : 3, warps = pass == 0 ? PW : FD_GATHER;
#pragma unroll 1
        for (int q0 = 0; q0 < nconv; q0 += FD_CHUNK) {
            const int m = min(FD_CHUNK, nconv - q0);
#pragma unroll 1
            for (int j = warp; j < m && warp < warps; j += warps) {
                const int k = conv[q0 + j];
                if (kind[k] != want) continue;
                int x, y, z;
                box_cell(a.g, w, k, x, y, z);
                const Cell cl(a.g, x, y, z);
                double d[3], fi;
                min_image(a.g, P.X, x, y, z, d);
                if (want == 2) {
                    fi = (double)Store<S>::ld(slot(cl, i), a.ph.inv_scale) +
                         (SH ? wgt<double>(i) * (double)a.ph.rho0 : 0.0);
                } else {
                    // density of the neighbour r + c_i if it is stable
                    const int xq = cl.X(cx(i)), yq = cl.Y(cy(i)), zq = cl.Z(cz(i));
                    const bool stable = lane >= 1 && lane < Q && !outside(x, y, z, i) && kind_of(xq, yq, zq) == 1;
                    const unsigned sb = __ballot_sync(ALL, stable);
                    R *sf = sm.f[warp];
#pragma unroll 4
                    for (int t = lane; t < (Q - 1) * Q; t += 32) {
                        const int h = 1 + t / Q, pop = t - (h - 1) * Q;
                        const Cell cn(a.g, cl.X(cx(h)), cl.Y(cy(h)), cl.Z(cz(h)));
                        sf[t] = (sb >> h) & 1u ? Store<S>::ld(slot(cn, pop), a.ph.inv_scale) : R(0);
                    }
                    __syncwarp();
                    double rn = 0.0;
                    if (stable)
#pragma unroll 1
                        for (int pop = 0; pop < Q; ++pop)
                            rn += (double)sf[(lane - 1) * Q + pop] + (SH ? wgt<double>(pop) * (double)a.ph.rho0 : 0.0);
                    __syncwarp();
                    double rsum = 0.0;
#pragma unroll 1
                    for (int h = 1; h < Q; ++h) {
                        const double t = __shfl_sync(ALL, rn, h);
                        if ((sb >> h) & 1u) rsum += t;
                    }
                    const int cnt = __popc(sb);
                    const double rho_bar = cnt > 0 ? rsum / (double)cnt : (double)a.ph.rho_ref;
                    double ub[3];
                    const double wxd[3] = {P.w[1] * d[2] - P.w[2] * d[1], P.w[2] * d[0] - P.w[0] * d[2],
                                           P.w[0] * d[1] - P.w[1] * d[0]};
                    for (int c3 = 0; c3 < 3; ++c3) ub[c3] = P.v[c3] + wxd[c3];
                    const double usq = ub[0] * ub[0] + ub[1] * ub[1] + ub[2] * ub[2];
                    const double cu = cx(i) * ub[0] + cy(i) * ub[1] + cz(i) * ub[2];
                    fi = wgt<double>(i) * rho_bar * (1.0 + 3.0 * cu + 4.5 * cu * cu - 1.5 * usq);
                    if (lane < Q) {
                        const double v = SH ? fi - wgt<double>(i) * (double)a.ph.rho0 : fi;
                        Store<S>::st(slot(cl, i), (R)v, a.ph.scale);
                    }
                }
                double Pm = 0.0;  // lanes 0..2: the momentum's components
#pragma unroll 1
                for (int h = 0; h < Q; ++h) {
                    const double t = __shfl_sync(ALL, fi, h);
                    Pm += t * (double)cdir(h, lane % 3);
                }
                if (lane < 3) sm.pm[j][lane] = Pm;
                if (lane == 0)
                    for (int c3 = 0; c3 < 3; ++c3) sm.pm[j][3 + c3] = d[c3];
            }
            __syncthreads();
            if (tid == 0) {
#pragma unroll 1
                for (int t = 0; t < m; ++t) {
                    const int k = conv[q0 + t];
                    if (kind[k] != want) continue;
                    const double *Pm = sm.pm[t], *d = sm.pm[t] + 3;
                    const double s = want == 2 ? 1.0 : -1.0;  // x + s y: exactly x + y or x - y
                    dP[0] += s * Pm[0];
                    dP[1] += s * Pm[1];
                    dP[2] += s * Pm[2];
                    dL[0] += s * (d[1] * Pm[2] - d[2] * Pm[1]);
                    dL[1] += s * (d[2] * Pm[0] - d[0] * Pm[2]);
                    dL[2] += s * (d[0] * Pm[1] - d[1] * Pm[0]);
                    if (want == 2 && nf_arr[k] == 0) {
                        int x, y, z;
                        box_cell(a.g, w, k, x, y, z);
                        const unsigned r = cell_index(a.g, x, y, z);
                        for (int c = 0; c < 6; ++c) E.diag[c] += (double)tau[c * np + r];
                    }
                    E.diag[want == 2 ? 6 : 7] += 1.0;
                }
            }
            __syncthreads();
        }
    }
    if (tid == 0)
        for (int c3 = 0; c3 < 3; ++c3) {
            P.dP[c3] = dP[c3];
            P.dL[c3] = dL[c3];
        }
    // E: the converted cells' stress and flags
#pragma unroll 1
    for (int q = tid; q < nconv; q += PT) {
        const int k = conv[q];
        int x, y, z;
        box_cell(a.g, w, k, x, y, z);
        const unsigned r = cell_index(a.g, x, y, z);
        const bool made = kind[k] == 3;
        for (int c = 0; c < 6; ++c) tau[c * np + r] = made ? (R)delta[(long long)c * nc + k] : R(0);
        flag[r] = (uint8_t)(made ? FLAG_FLUID : FLAG_PART0 + p);
        nf_arr[k] = 0;
    }
    __syncthreads();
    // F: neighbour masks of the converted cells and their neighbours (the only cells whose
    // masks change; a cell reached twice gets the same value twice): a warp per mask, lane i
    // looking in direction i (see cell_mask)
#pragma unroll 1
    for (int e = warp; e < nconv * Q; e += PW) {
        const int q = e / Q, h = e - q * Q;
        int x, y, z;
        box_cell(a.g, w, conv[q], x, y, z);
        if (outside(x, y, z, h)) continue;
        const Cell c0(a.g, x, y, z);
        const Cell c1(a.g, c0.X(cx(h)), c0.Y(cy(h)), c0.Z(cz(h)));
        int fl = FLAG_FLUID;
        if (lane < Q)
            fl = outside(c1.x, c1.y, c1.z, lane) ? FLAG_NOSLIP : flag[c1.idx(cx(lane), cy(lane), cz(lane))];
        uint32_t m = __ballot_sync(ALL, fl != FLAG_FLUID);
        if (__ballot_sync(ALL, lane > 0 && fl != FLAG_FLUID && fl != FLAG_NOSLIP)) m |= MASK_MOVING;
        if (lane == 0) E.mask[c1.self()] = m;
    }
    if (tid < 3) {
        if (tid == 0) P.changed = 1;
        P.v[tid] += P.dP[tid] / P.m;
        P.w[tid] += P.dL[tid] / P.I;
    }
    __syncthreads();
}

// The particles in `changed` and those that overlap or nearly touch one of them.  A cell that
// a particle leaves inside another (spheres may overlap) has neighbours deep in that other
// one, whose surface velocities are not kept up to date; it lies within R + 1 of the centre
// it was left by, so the pairs closer than R_p + R_q + 1 + sqrt(2) matter.  FP32 with a cell
// to spare; a lane per changed particle.  A call of its own, for solves with several spheres: in
// line it cost those with one 0.7 us of fetched code per step.
static __device__ __noinline__ unsigned long long with_touching(const Geo &g, const PartDev *parts, int nparts,
                                                                unsigned long long changed) {
    unsigned long long out = changed;
    const int nn[3] = {g.nx, g.ny, g.nz};
#pragma unroll 1
    for (int p = 0; p < nparts; ++p) {
        if ((changed >> p) & 1ull) continue;
        bool near = false;
#pragma unroll 1
        for (int q = (int)threadIdx.x & 31; q < nparts; q += 32) {
            if (!((changed >> q) & 1ull)) continue;
            float d2 = 0.0f;
            for (int k = 0; k < 3; ++k) {
                float d = (float)parts[p].X[k] - (float)parts[q].X[k];
                if (g.per[k]) d -= (float)nn[k] * rintf(d / (float)nn[k]);
                d2 += d * d;
            }
            const float reach = (float)parts[p].R + (float)parts[q].R + 3.5f;
            near |= d2 <= reach * reach;
        }
        if (__any_sync(0xffffffffu, near)) out |= 1ull << p;
    }
    return out;
}

// Particle phase of one step for one solve per cluster: sums of the momentum-exchange
// partials (reduced modes), symplectic Euler, fill/drain of the cells the spheres now cover
// or have left (the particles one after another), links of the particles whose cells
// converted, and the boundary velocities of the cells they cover (set_solid_velocity).
// Every cell of a particle's box is classified each step and few convert, so
// the bounds are latency and the FP64 pipe: the cluster spreads the classification and the
// link list over PC x PT threads and as many SMs, FP64 work runs in single threads or in
// lanes side by side, and the conversions work on a list.  An R = 8 sphere takes 18 us per
// step without conversions (11 of them the classification with the surface velocities) and
// 66 with one converted cell (16 of them the links); three kernels of one block each took
// 40 and about 300.
// One cluster per solve: entries[blockIdx.x / PC], or `one` when entries is nullptr.
template <class S>
__global__ void __cluster_dims__(PC, 1, 1) __launch_bounds__(PT)
    k_particle_phase(const PartEntry<S> *__restrict__ entries, const __grid_constant__ PartEntry<S> one, int k) {
    step_wait();
    step_next();  // its few blocks leave the device to the next kernel's anyway
    cooperative_groups::cluster_group cl = cooperative_groups::this_cluster();
    const PartEntry<S> &E = entries ? entries[blockIdx.x / PC] : one;
    const KArgs<S> &a = E.a[k & 1];
    const int rank = (int)cl.block_rank(), tid = (int)threadIdx.x, lane = tid & 31, warp = tid >> 5;
    __shared__ ClusterCounts counts;
    __shared__ int wsum[PW], s_mine;
    __shared__ BoxWalk w;
    __shared__ SphereFilter sf;
    __shared__ FillDrainSmem<typename Store<S>::R> sm;
    int buf = 0;
    if (rank == 0) {
        if (E.sums) {
            // as k_body_partials: component c of body b over partials lane, lane + 32, ...
            for (int it = warp; it < 6 * E.nbody; it += PW) {
                const int b = it / 6, c = it - 6 * b;
                const int n = (E.seg_count[b] + 127) / 128;
                double acc = 0.0;
                for (int j = lane; j < n; j += 32) acc += E.sums[((long long)b * E.sum_stride + j) * 8 + c];
                for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
                if (lane == 0) {
                    const int fl = E.seg_flag[b];
                    if (c < 3) E.body_F[fl * 3 + c] = acc;
                    if (fl >= FLAG_PART0 && fl < FLAG_PART0 + MAX_PART)
                        (c < 3 ? E.parts[fl - FLAG_PART0].Fme[c] : E.parts[fl - FLAG_PART0].Tme[c - 3]) = acc;
                }
            }
            __syncthreads();
        }
        // symplectic Euler (FP64): velocities with this step's momentum-exchange force and
        // torque and the external ones, then the position with the new velocity
        for (int t = tid; t < 3 * E.nparts; t += PT) {
            PartDev &P = E.parts[t / 3];
            const int c = t % 3;
            P.v[c] += (P.Fme[c] + P.Fext[c]) / P.m;
            P.w[c] += (P.Tme[c] + P.Text[c]) / P.I;
            P.X[c] += P.v[c];
        }
    }
    cl.sync();
    unsigned long long changed = 0;
    for (int p = 0; p < E.nparts; ++p) {
        PartDev &P = E.parts[p];
        __syncthreads();
        if (warp == 0) prepare_box(a.g, P, 3, w, &sf);
        if (tid == 0) s_mine = 0;
        __syncthreads();
        // A: classify a consecutive range of the box
        const int per = (w.cells + PC - 1) / PC, lo = min(w.cells, per * rank), hi = min(w.cells, lo + per);
        int mine = 0;
#pragma unroll 1
        for (int q = lo + tid; q < hi; q += PT) {
            int x, y, z;
            box_cell(a.g, w, q, x, y, z);
            const unsigned r = cell_index(a.g, x, y, z);
            const int old = E.flag[r];
            int kd = 0;
            if (old == FLAG_FLUID || old == FLAG_PART0 + p) {
                float d2;
                const bool inside = inside_sphere(a.g, P, sf, x, y, z, d2);
                kd = old == FLAG_FLUID ? (inside ? 2 : 1) : (inside ? 0 : 3);
                // the surface velocity of a cell the sphere keeps (again below when
                // conversions change the sphere's velocity or free a cell inside it).  A cell
                // deeper than sqrt(2) below the surface has no fluid neighbour to read it.
                if (kd == 0 && d2 >= sf.deep2) set_solid_velocity<S>(a, x, y, z, r, a.u_out, a.u_out);
            }
            E.kind[q] = (uint8_t)kd;
            mine += kd >= 2 ? 1 : 0;
        }
        if (mine) atomicAdd(&s_mine, mine);
        __syncthreads();
        int before, nconv;
        cluster_exchange(cl, counts, buf, s_mine, before, nconv);
        buf ^= 1;
        if (nconv == 0) {
            // nothing converts: no impulse, flags and links stay as they are
            if (rank == 0 && tid == 0) {
                for (int c3 = 0; c3 < 3; ++c3) P.dP[c3] = P.dL[c3] = 0.0;
                P.changed = 0;
            }
            continue;
        }
        changed |= 1ull << p;
        // A': the converted cells listed in cell order
        if (s_mine > 0)
            for (int q0 = lo; q0 < hi; q0 += PT) {
                const int q = q0 + tid, is = q < hi && E.kind[q] >= 2 ? 1 : 0;
                int n;
                const int pos = before + block_scan(is, wsum, n);
                if (is) E.conv[pos] = q;
                before += n;
            }
        cl.sync();
        if (rank == 0) {
            if (((E.parity0 + k) & 1) == 0)
                fill_drain<S, 0>(E, a, P, p, w, nconv, sm);
            else
                fill_drain<S, 1>(E, a, P, p, w, nconv, sm);
        }
        cl.sync();
    }
    // surface velocities of the spheres whose velocity or neighbourhood the conversions changed
    const unsigned long long redo = changed && E.nparts > 1 ? with_touching(a.g, E.parts, E.nparts, changed) : changed;
    for (int p = E.nparts - 1; p >= 0; --p) {
        if (!((redo >> p) & 1ull)) continue;
        if (p + 1 < E.nparts) {  // the box of the last particle is still there
            __syncthreads();
            if (warp == 0) prepare_box(a.g, E.parts[p], 3, w, nullptr);
            __syncthreads();
        }
#pragma unroll 1
        for (int q = rank * PT + tid; q < w.cells; q += PC * PT) {
            int x, y, z;
            box_cell(a.g, w, q, x, y, z);
            const unsigned r = cell_index(a.g, x, y, z);
            if (E.flag[r] == FLAG_PART0 + p && (E.mask[r] & 0x7fffeu) != 0x7fffeu)
                set_solid_velocity<S>(a, x, y, z, r, a.u_out, a.u_out);
        }
    }
    for (int p = 0; p < E.nparts; ++p)
        if ((changed >> p) & 1ull)
            particle_links(cl, a.g, E.parts[p], p, E.flag, E.mask, E.links, E.seg_begin, E.seg_count, E.first_seg + p,
                           E.capacity[p], counts, buf, wsum);
    cl.sync();  // no block leaves while another may still write to its shared memory
}

} // namespace lbve
