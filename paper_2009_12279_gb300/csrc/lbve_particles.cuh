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

// Cells within R + margin of the particle centre (whole domain along a periodic side
// the box would wrap onto itself; clamped to the domain along a closed side).
__host__ __device__ inline BBox particle_bbox(const Geo &g, const double X[3], double R, int margin) {
    BBox b;
    const int nn[3] = {g.nx, g.ny, g.nz};
    for (int k = 0; k < 3; ++k) {
        int lo = (int)floor(X[k] - R) - margin;
        int hi = (int)ceil(X[k] + R) + margin;
        if (!g.per[k]) {
            lo = lo < 0 ? 0 : lo;
            hi = hi > nn[k] - 1 ? nn[k] - 1 : hi;
        }
        int ext = hi - lo + 1;
        if (ext > nn[k]) {
            lo = 0;
            ext = nn[k];
        }
        if (ext < 0) ext = 0;
        b.lo[k] = lo;
        b.ext[k] = ext;
    }
    return b;
}

__host__ __device__ inline int bbox_capacity_side(double R, int margin) { return 2 * (int)ceil(R) + 2 * margin + 3; }

// A particle's box as the phase walks it: the lower corner wrapped into the domain once, so
// that a cell's coordinate and a cell's place in the box are each one conditional
// correction away.
struct BoxWalk {
    int lo[3], ext[3];
    FastDiv dx, dy;
    int cells;
};
__device__ __forceinline__ BoxWalk box_walk(const Geo &g, const BBox &b) {
    BoxWalk w;
    const int nn[3] = {g.nx, g.ny, g.nz};
    for (int k = 0; k < 3; ++k) {
        w.lo[k] = ((b.lo[k] % nn[k]) + nn[k]) % nn[k];
        w.ext[k] = b.ext[k];
    }
    w.cells = (int)b.cells();
    w.dx = FastDiv::of((unsigned)(b.ext[0] > 0 ? b.ext[0] : 1));
    w.dy = FastDiv::of((unsigned)(b.ext[1] > 0 ? b.ext[1] : 1));
    return w;
}
// coordinates of cell k of the box
__device__ __forceinline__ void box_cell(const Geo &g, const BoxWalk &w, int k, int &x, int &y, int &z) {
    const unsigned row = w.dx.div((unsigned)k), pl = w.dy.div(row);
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
// then ran the FP64 branch: 33 us per step for an R = 8 sphere, now part of 5.)
struct SphereFilter {
    int Xi[3];
    float Xf[3], R2, tol;
};
__device__ __forceinline__ SphereFilter sphere_filter(const Geo &g, const PartDev &P) {
    SphereFilter f;
    const int nn[3] = {g.nx, g.ny, g.nz};
    for (int k = 0; k < 3; ++k) {
        const double c = rint(P.X[k]);
        f.Xf[k] = (float)(P.X[k] - c);
        f.Xi[k] = (int)c;
        if (g.per[k]) f.Xi[k] = ((f.Xi[k] % nn[k]) + nn[k]) % nn[k];
    }
    const double D = P.R + 5.0;
    f.R2 = (float)(P.R * P.R);
    f.tol = (float)(D * D * 0x1p-18);
    return f;
}
__device__ __forceinline__ bool inside_sphere(const Geo &g, const PartDev &P, const SphereFilter &f, int x, int y,
                                              int z) {
    const int q[3] = {x, y, z}, nn[3] = {g.nx, g.ny, g.nz};
    float d2 = 0.0f;
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
// ranges of the box; counts first, then the links at their places.
template <class S>
__device__ __forceinline__ void particle_links(cooperative_groups::cluster_group &cl, const Geo &g, const PartDev &P,
                                               int p, const uint8_t *flag, long long *links, const int *seg_begin,
                                               int *seg_count, int seg, int cap, ClusterCounts &counts, int &buf,
                                               int *wsum) {
    __shared__ BoxWalk w;
    __syncthreads();
    if (threadIdx.x == 0) w = box_walk(g, particle_bbox(g, P.X, P.R, 2));
    __syncthreads();
    const int rank = (int)cl.block_rank();
    const int per = (w.cells + PC - 1) / PC, lo = min(w.cells, per * rank), hi = min(w.cells, lo + per);
    auto dirs = [&](int k, unsigned &r) -> unsigned {
        int x, y, z;
        box_cell(g, w, k, x, y, z);
        r = cell_index(g, x, y, z);
        unsigned m = 0;
        if (flag[r] != FLAG_FLUID) return 0u;
        const Cell c(g, x, y, z);
#pragma unroll
        for (int i = 1; i < Q; ++i) {
            const bool out = (!g.per[0] && (x + cx(i) < 0 || x + cx(i) >= g.nx)) ||
                             (!g.per[1] && (y + cy(i) < 0 || y + cy(i) >= g.ny)) ||
                             (!g.per[2] && (z + cz(i) < 0 || z + cz(i) >= g.nz));
            if (!out && flag[c.idx(cx(i), cy(i), cz(i))] == FLAG_PART0 + p) m |= 1u << i;
        }
        return m;
    };
    int mine = 0;
    for (int k = lo + (int)threadIdx.x; k < hi; k += PT) {
        unsigned r;
        mine += __popc(dirs(k, r));
    }
    int total_block;
    block_scan(mine, wsum, total_block);
    int base, total;
    cluster_exchange(cl, counts, buf, total_block, base, total);
    buf ^= 1;
    long long *out = links + seg_begin[seg];
    if (total_block > 0)
        for (int k0 = lo; k0 < hi; k0 += PT) {
            const int k = k0 + (int)threadIdx.x;
            unsigned r = 0, m = 0;
            if (k < hi) m = dirs(k, r);
            int n;
            int pos = base + block_scan(__popc(m), wsum, n);
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
    k_particle_links(Geo g, const PartDev *parts, const uint8_t *flag, long long *links, const int *seg_begin,
                     int *seg_count, int first_seg, const int *capacity) {
    cooperative_groups::cluster_group cl = cooperative_groups::this_cluster();
    __shared__ ClusterCounts counts;
    __shared__ int wsum[PW];
    int buf = 0;
    const int p = (int)blockIdx.x / PC;
    cl.sync();  // every block of the cluster is running before its shared memory is written
    if (parts[p].changed)
        particle_links<S>(cl, g, parts[p], p, flag, links, seg_begin, seg_count, first_seg + p, capacity[p], counts, buf,
                          wsum);
    cl.sync();  // no block leaves while another may still write to its shared memory
}

// Fill/drain of the listed converted cells of particle p (first block of the cluster).
// kind: 0 other, 1 fluid before and after, 2 destroyed (fluid -> particle), 3 created
// (particle -> fluid).  All stress moves use the pre-conversion stress:
//   destroyed d: each of its N_f stable D3Q7 neighbours gains tau(d)/N_f;
//   created c:   tau(c) = sum of its stable neighbours' tau / (N_f + 1), each of
//                them gives up tau(c)/N_f;
// the deleted / created momentum goes to the particle as an impulse at the cell.
// The work follows the list (a few cells per step), not the box.
template <class S, int PAR>
__device__ __forceinline__ void fill_drain(const PartEntry<S> &E, const KArgs<S> &a, PartDev &P, int p,
                                           const BoxWalk &w, int nconv, double (*s_pm)[6]) {
    using R = typename Store<S>::R;
    constexpr bool SH = Store<S>::shifted;
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
    // B: N_f of converted cells, new stress of created cells
    for (int q = tid; q < nconv; q += PT) {
        const int k = conv[q], kd = kind[k];
        int x, y, z, kn[6];
        box_cell(a.g, w, k, x, y, z);
        unsigned nb[6];
#pragma unroll
        for (int l = 0; l < 6; ++l) {
            int xq = x, yq = y, zq = z;
            kn[l] = step_cell(a.g, l, xq, yq, zq) ? kind_of(xq, yq, zq) : 0;
            nb[l] = cell_index(a.g, xq, yq, zq);
        }
        int nf = 0;
        double sum[6] = {0, 0, 0, 0, 0, 0};
#pragma unroll
        for (int l = 0; l < 6; ++l)
            if (kn[l] == 1) {
                nf++;
                for (int c = 0; c < 6; ++c) sum[c] += (double)tau[c * np + nb[l]];
            }
        nf_arr[k] = (uint8_t)nf;
        if (kd == 3)
            for (int c = 0; c < 6; ++c) delta[(long long)c * nc + k] = sum[c] / (double)(nf + 1);
    }
    __syncthreads();
    // C: stress gathered by each stable cell from its converted D3Q7 neighbours, face by
    // face.  Pair e = (converted cell, face) stands for the stable cell on that face when
    // the converted cell is the first one in that cell's face order; returns its place in
    // the box, or -1.
    auto owned = [&](int e, int &x, int &y, int &z, int (&kb)[6], int (&kk)[6]) -> int {
        const int q = e / 6, l = e - 6 * q;
        box_cell(a.g, w, conv[q], x, y, z);
        if (!step_cell(a.g, l, x, y, z)) return -1;
        const int ks = box_index(a.g, w, x, y, z);
        if (ks < 0 || kind[ks] != 1) return -1;
        int first = -1;
#pragma unroll
        for (int m = 0; m < 6; ++m) {
            int xq = x, yq = y, zq = z;
            kb[m] = step_cell(a.g, m, xq, yq, zq) ? box_index(a.g, w, xq, yq, zq) : -1;
            kk[m] = kb[m] >= 0 ? kind[kb[m]] : 0;
            if (kk[m] < 2) kb[m] = -1;
            if (first < 0 && kb[m] >= 0) first = kb[m];
        }
        return first == conv[q] ? ks : -1;
    };
    for (int e = tid; e < 6 * nconv; e += PT) {
        int x, y, z, kb[6], kk[6];
        const int ks = owned(e, x, y, z, kb, kk);
        if (ks < 0) continue;
        double acc[6] = {0, 0, 0, 0, 0, 0};
#pragma unroll
        for (int m = 0; m < 6; ++m) {
            if (kb[m] < 0) continue;
            const double nf = (double)nf_arr[kb[m]];
            if (kk[m] == 2) {
                int xq = x, yq = y, zq = z;
                step_cell(a.g, m, xq, yq, zq);
                const unsigned nb = cell_index(a.g, xq, yq, zq);
                for (int c = 0; c < 6; ++c) acc[c] += (double)tau[c * np + nb] / nf;
            } else {
                for (int c = 0; c < 6; ++c) acc[c] -= delta[(long long)c * nc + kb[m]] / nf;
            }
        }
        for (int c = 0; c < 6; ++c) delta[(long long)c * nc + ks] = acc[c];
    }
    // D: impulses and the populations of created cells, a warp per converted cell: the
    // momentum of a destroyed cell's deleted populations, or f^eq(rho_bar, u_b) written to
    // a created cell with its momentum.  A created cell reads only stable cells' populations
    // and writes only its own, so the cells are independent.  Thread 0 then adds the
    // momenta to the impulse in the sequential order of the method: destroyed cells in cell
    // order, then created cells in cell order.  Sums over directions run in direction order
    // (shuffles hand every lane the terms).
    double dP[3] = {0, 0, 0}, dL[3] = {0, 0, 0};
    for (int pass = 0; pass < 2; ++pass) {
        const int want = pass == 0 ? 2 : 3;
        for (int q0 = 0; q0 < nconv; q0 += PT) {
            const int m = min(PT, nconv - q0);
            for (int j = warp; j < m; j += PW) {
                const int k = conv[q0 + j];
                if (kind[k] != want) continue;
                int x, y, z;
                box_cell(a.g, w, k, x, y, z);
                const unsigned r = cell_index(a.g, x, y, z);
                const Cell cl(a.g, x, y, z);
                double d[3], fi = 0.0;
                min_image(a.g, P.X, x, y, z, d);
                if (want == 2) {
                    // lane i: population i
#pragma unroll
                    for (int i = 0; i < Q; ++i)
                        if (lane == i) {
                            const S *src = PAR == 0 ? a.f + (long long)i * np + r
                                                    : a.f + (long long)copp(i) * np + cl.idx(-cx(i), -cy(i), -cz(i));
                            fi = (double)Store<S>::ld(src, a.ph.inv_scale) + (SH ? wgt<double>(i) * (double)a.ph.rho0 : 0.0);
                        }
                } else {
                    // lane i: density of the neighbour r + c_i if it is stable
                    double rn = 0.0;
                    bool stable = false;
                    int xq = x, yq = y, zq = z;
                    if (lane >= 1 && lane < Q) {
                        const int dx = cx(lane), dy = cy(lane), dz = cz(lane);
                        const bool out = (!a.g.per[0] && (x + dx < 0 || x + dx >= a.g.nx)) ||
                                         (!a.g.per[1] && (y + dy < 0 || y + dy >= a.g.ny)) ||
                                         (!a.g.per[2] && (z + dz < 0 || z + dz >= a.g.nz));
                        if (!out) {
                            xq = cl.X(dx);
                            yq = cl.Y(dy);
                            zq = cl.Z(dz);
                            stable = kind_of(xq, yq, zq) == 1;
                        }
                    }
                    if (stable) {
                        const Cell cn(a.g, xq, yq, zq);
                        R fn[Q];
                        load_pdfs<S, PAR>(a, cn, cn.self(), fn);
                        for (int i = 0; i < Q; ++i) rn += (double)fn[i] + (SH ? wgt<double>(i) * (double)a.ph.rho0 : 0.0);
                    }
                    const unsigned sb = __ballot_sync(0xffffffffu, stable);
                    double rsum = 0.0;
                    for (int i = 1; i < Q; ++i) {
                        const double t = __shfl_sync(0xffffffffu, rn, i);
                        if ((sb >> i) & 1u) rsum += t;
                    }
                    const int cnt = __popc(sb);
                    const double rho_bar = cnt > 0 ? rsum / (double)cnt : (double)a.ph.rho_ref;
                    double ub[3];
                    const double wxd[3] = {P.w[1] * d[2] - P.w[2] * d[1], P.w[2] * d[0] - P.w[0] * d[2],
                                           P.w[0] * d[1] - P.w[1] * d[0]};
                    for (int c3 = 0; c3 < 3; ++c3) ub[c3] = P.v[c3] + wxd[c3];
                    const double usq = ub[0] * ub[0] + ub[1] * ub[1] + ub[2] * ub[2];
#pragma unroll
                    for (int i = 0; i < Q; ++i)
                        if (lane == i) {
                            const double cu = cx(i) * ub[0] + cy(i) * ub[1] + cz(i) * ub[2];
                            fi = wgt<double>(i) * rho_bar * (1.0 + 3.0 * cu + 4.5 * cu * cu - 1.5 * usq);
                            S *dst = PAR == 0 ? a.f + (long long)i * np + r
                                              : a.f + (long long)copp(i) * np + cl.idx(-cx(i), -cy(i), -cz(i));
                            const double v = SH ? fi - wgt<double>(i) * (double)a.ph.rho0 : fi;
                            Store<S>::st(dst, (R)v, a.ph.scale);
                        }
                }
                double Pm = 0.0;  // lanes 0..2: the momentum's components
                for (int i = 0; i < Q; ++i) {
                    const double t = __shfl_sync(0xffffffffu, fi, i);
                    Pm += t * (double)cdir(i, lane % 3);
                }
                if (lane < 3) s_pm[j][lane] = Pm;
                if (lane == 0)
                    for (int c3 = 0; c3 < 3; ++c3) s_pm[j][3 + c3] = d[c3];
            }
            __syncthreads();
            if (tid == 0) {
                for (int t = 0; t < m; ++t) {
                    const int k = conv[q0 + t];
                    if (kind[k] != want) continue;
                    const double *Pm = s_pm[t], *d = s_pm[t] + 3;
                    if (want == 2) {
                        dP[0] += Pm[0];
                        dP[1] += Pm[1];
                        dP[2] += Pm[2];
                        dL[0] += d[1] * Pm[2] - d[2] * Pm[1];
                        dL[1] += d[2] * Pm[0] - d[0] * Pm[2];
                        dL[2] += d[0] * Pm[1] - d[1] * Pm[0];
                        if (nf_arr[k] == 0) {
                            int x, y, z;
                            box_cell(a.g, w, k, x, y, z);
                            const unsigned r = cell_index(a.g, x, y, z);
                            for (int c = 0; c < 6; ++c) E.diag[c] += (double)tau[c * np + r];
                        }
                        E.diag[6] += 1.0;
                    } else {
                        dP[0] -= Pm[0];
                        dP[1] -= Pm[1];
                        dP[2] -= Pm[2];
                        dL[0] -= d[1] * Pm[2] - d[2] * Pm[1];
                        dL[1] -= d[2] * Pm[0] - d[0] * Pm[2];
                        dL[2] -= d[0] * Pm[1] - d[1] * Pm[0];
                        E.diag[7] += 1.0;
                    }
                }
            }
            __syncthreads();
        }
    }
    // E: apply the stress moves, then the converted cells' stress and flags
    for (int e = tid; e < 6 * nconv; e += PT) {
        int x, y, z, kb[6], kk[6];
        const int ks = owned(e, x, y, z, kb, kk);
        if (ks < 0) continue;
        const unsigned r = cell_index(a.g, x, y, z);
        for (int c = 0; c < 6; ++c) tau[c * np + r] = (R)((double)tau[c * np + r] + delta[(long long)c * nc + ks]);
    }
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
    // masks change; a cell reached twice gets the same value twice)
    for (int e = tid; e < nconv * Q; e += PT) {
        const int q = e / Q, i = e - q * Q;
        int x, y, z;
        box_cell(a.g, w, conv[q], x, y, z);
        if ((!a.g.per[0] && (x + cx(i) < 0 || x + cx(i) >= a.g.nx)) ||
            (!a.g.per[1] && (y + cy(i) < 0 || y + cy(i) >= a.g.ny)) ||
            (!a.g.per[2] && (z + cz(i) < 0 || z + cz(i) >= a.g.nz)))
            continue;
        const Cell cl(a.g, x, y, z);
        const int xq = cl.X(cx(i)), yq = cl.Y(cy(i)), zq = cl.Z(cz(i));
        E.mask[cell_index(a.g, xq, yq, zq)] = cell_mask(a.g, flag, xq, yq, zq);
    }
    if (tid == 0) {
        P.changed = 1;
        for (int c3 = 0; c3 < 3; ++c3) {
            P.dP[c3] = dP[c3];
            P.dL[c3] = dL[c3];
            P.v[c3] += dP[c3] / P.m;
            P.w[c3] += dL[c3] / P.I;
        }
    }
    __syncthreads();
}

// Particle phase of one step for one solve per cluster: sums of the momentum-exchange
// partials (reduced modes), symplectic Euler, fill/drain of the cells the spheres now cover
// or have left (the particles one after another), links of the particles whose cells
// converted, and the boundary velocities of the cells they cover (set_solid_velocity).
// Every cell of a particle's box is classified each step and few convert, so
// the bounds are latency and the FP64 pipe: the cluster spreads the classification and the
// link list over PC x PT threads and as many SMs, FP64 work runs in single threads or in
// lanes side by side, and the conversions work on a list.  Before, three kernels of one
// block each took 40 us per step of an R = 8 sphere without conversions and about 300
// with them.
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
    __shared__ double s_pm[PT][6];  // momentum and lever arm of a chunk of converted cells
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
        if (tid == 0) {
            w = box_walk(a.g, particle_bbox(a.g, P.X, P.R, 3));
            sf = sphere_filter(a.g, P);
            s_mine = 0;
        }
        __syncthreads();
        // A: classify a consecutive range of the box
        const int per = (w.cells + PC - 1) / PC, lo = min(w.cells, per * rank), hi = min(w.cells, lo + per);
        int mine = 0;
#pragma unroll 4
        for (int q = lo + tid; q < hi; q += PT) {
            int x, y, z;
            box_cell(a.g, w, q, x, y, z);
            const int old = E.flag[cell_index(a.g, x, y, z)];
            int kd = 0;
            if (old == FLAG_FLUID || old == FLAG_PART0 + p) {
                const bool inside = inside_sphere(a.g, P, sf, x, y, z);
                kd = old == FLAG_FLUID ? (inside ? 2 : 1) : (inside ? 0 : 3);
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
                fill_drain<S, 0>(E, a, P, p, w, nconv, s_pm);
            else
                fill_drain<S, 1>(E, a, P, p, w, nconv, s_pm);
        }
        cl.sync();
    }
    // the spheres' surface velocities, by the state the next step works with
    for (int p = 0; p < E.nparts; ++p) {
        __syncthreads();
        if (tid == 0) w = box_walk(a.g, particle_bbox(a.g, E.parts[p].X, E.parts[p].R, 3));
        __syncthreads();
        for (int q = rank * PT + tid; q < w.cells; q += PC * PT) {
            int x, y, z;
            box_cell(a.g, w, q, x, y, z);
            const unsigned r = cell_index(a.g, x, y, z);
            if (E.flag[r] == FLAG_PART0 + p) set_solid_velocity<S>(a, x, y, z, r, a.u_out, a.u_out);
        }
    }
    for (int p = 0; p < E.nparts; ++p)
        if ((changed >> p) & 1ull)
            particle_links<S>(cl, a.g, E.parts[p], p, E.flag, E.links, E.seg_begin, E.seg_count, E.first_seg + p,
                              E.capacity[p], counts, buf, wsum);
    cl.sync();  // no block leaves while another may still write to its shared memory
}

} // namespace lbve
