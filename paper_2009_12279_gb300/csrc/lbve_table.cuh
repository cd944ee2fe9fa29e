// lbve_table.cuh -- host-side launchers of the step kernels for one PDF storage type,
// collected in a KernelTable.  Included once per storage type by the precision TUs.
#pragma once

#include <algorithm>
#include <atomic>

#include "lbve_kernels.cuh"
#include "lbve_particles.cuh"
#include "lbve_rows.cuh"

namespace lbve {

// Dynamic shared-memory limit of a kernel raised once per device: the attribute is per
// device, so the record is a bit per device ordinal (idempotent if two threads race).
struct SmemAttrOnce {
    std::atomic<unsigned long long> done[2] = {{0ull}, {0ull}};
    template <class K>
    cudaError_t ensure(K kernel, size_t bytes) {
        int dev = 0;
        cudaError_t e = cudaGetDevice(&dev);
        if (e != cudaSuccess) return e;
        if (dev < 0 || dev >= 128) return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
        const unsigned long long bit = 1ull << (dev & 63);
        std::atomic<unsigned long long> &w = done[dev >> 6];
        if (w.load(std::memory_order_acquire) & bit) return cudaSuccess;
        e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
        if (e == cudaSuccess) w.fetch_or(bit, std::memory_order_acq_rel);
        return e;
    }
};

template <class R>
inline Phys<R> convert_phys(const Phys<double> &p) {
    Phys<R> o;
    o.omega_p = (R)p.omega_p;
    o.omega_m = (R)p.omega_m;
    o.A = (R)p.A;
    o.B = (R)p.B;
    o.ep_l = (R)p.ep_l;
    o.inv_l = (R)p.inv_l;
    for (int k = 0; k < 3; ++k) o.g[k] = (R)p.g[k];
    o.rho0 = (R)p.rho0;
    o.rho_ref = (R)p.rho_ref;
    o.scale = (R)p.scale;
    o.inv_scale = (R)p.inv_scale;
    o.flux_on = p.flux_on;
    o.src_on = p.src_on;
    o.ctu_on = p.ctu_on;
    o.divu_on = p.divu_on;
    o.gk = (R)p.gk;
    o.fene = p.fene;
    o.fene_L2 = (R)p.fene_L2;
    o.eta_p = (R)p.eta_p;
    o.lam = (R)p.lam;
    for (int c = 0; c < MAX_WALL; ++c)
        for (int k = 0; k < 3; ++k) o.wall_vel[c][k] = (R)p.wall_vel[c][k];
    return o;
}

template <class S>
struct Launch {
    using R = typename Store<S>::R;

    // split schedule: the stream-collide writes u[ucur] and the stress update reads it;
    // fused schedule: the stress update reads u[ucur], the stream-collide writes u[ucur^1].
    static KArgs<S> args(const DevState &d, bool fused = false) {
        KArgs<S> a;
        a.g = d.g;
        a.ph = convert_phys<R>(d.ph);
        a.f = (S *)d.f;
        a.tau = (const R *)d.tau[d.cur];
        a.tau_out = (R *)d.tau[d.cur ^ 1];
        a.u_in = (const R *)d.u[d.ucur];
        a.u_out = (R *)d.u[fused ? d.ucur ^ 1 : d.ucur];
        a.flag = d.flag;
        a.mask = d.mask;
        a.parts = d.parts;
        a.step = d.step;
        a.dstep = d.dstep;
        a.bad = d.bad;
        a.zlo = d.zlo;
        a.zhi = d.zhi > 0 ? d.zhi : d.g.nz;
        a.key_base = d.key_base;
        a.lin = (unsigned)((long long)d.g.nx * d.g.ny * zcount(d));
        a.dnx = FastDiv::of((unsigned)d.g.nx);
        a.dny = FastDiv::of((unsigned)d.g.ny);
        a.nzc = (unsigned)zcount(d);
        a.dnz = FastDiv::of(a.nzc);
        link_dirs<S>(a);
        return a;
    }
    // per-cell kernels: blocks of block_x x (128 / block_x) threads
    static dim3 block2(const DevState &d) { return dim3((unsigned)d.block_x, (unsigned)(128 / d.block_x)); }
    static int zcount(const DevState &d) { return (d.zhi > 0 ? d.zhi : d.g.nz) - d.zlo; }
    static dim3 grid2(const DevState &d) {
        const dim3 b = block2(d);
        return dim3((unsigned)((d.g.nx + b.x - 1) / b.x), (unsigned)((d.g.ny + b.y - 1) / b.y), (unsigned)zcount(d));
    }
    static dim3 grid3(const DevState &d) { return dim3((unsigned)((d.g.nx + d.block_x - 1) / d.block_x), d.g.ny, d.g.nz); }

    static cudaError_t init(const DevState &d, const double *rho, const double *u, const double *tau, long long r0,
                            long long count, long long ld, cudaStream_t s) {
        if (count <= 0) return cudaSuccess;
        KArgs<S> a = args(d);
        const unsigned nb = (unsigned)((count + 255) / 256);
        k_init<S><<<nb, 256, 0, s>>>(a, rho, u, tau, (R *)d.tau[d.cur], r0, count, ld);
        return cudaGetLastError();
    }
    // The row-pipelined stream-collide (k_lb_rows): rows of a multiple of 32 cells, at
    // most LR_MAX_NX, 16-byte aligned field arrays, a layout that fits the
    // shared memory of one block, Oldroyd-B or Giesekus stress (FENE-P reads conformation
    // tensors: per-cell kernel).  The result is bitwise that of the per-cell kernel.
    static size_t rows_smem(int nx) { return RowsLayout<S>{nx}.total(); }
    static bool rows_ok(const DevState &d) {
        auto al = [](const void *p) { return ((uintptr_t)p & 15u) == 0; };
        if (d.ph.fene || d.g.nx % 32 != 0 || d.g.nx < 64 || d.g.nx > LR_MAX_NX) return false;
        // schedule AUTO: grids of 2^22 cells and more (FP64, the parity mode: never) ...
        if (d.auto_kernels == 1 && (d.g.n < (1LL << 22) || !Store<S>::shifted)) return false;
        if (!al(d.f) || !al(d.tau[0]) || !al(d.tau[1]) || !al(d.mask) || !al(d.u[0]) || !al(d.u[1])) return false;
        int dev = 0, optin = 0, persm = 0;
        if (cudaGetDevice(&dev) != cudaSuccess) return false;
        if (cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess) return false;
        const size_t sm = rows_smem(d.g.nx);
        if (sm > (size_t)optin) return false;
        if (d.auto_kernels != 1) return true;
        // ... whose rows fill an SM: the blocks that fit its shared memory have nx / 32
        // consumer warps each, and with few of them the per-cell kernel, which has 28, is
        // faster.  Measured on GB300, row pipeline against per-cell, ps per cell: FP32 128-wide
        // (16 warps) 4 M cells 33.4 / 34.7, 67 M 32.2 / 34.2, 192 (12) 36.6 / 34.8, 224 (14) 33.3
        // / 35.9, 256 (16) 31.8 / 34.6, 320 (10) 35.7 / 34.3, 384 (12) 6 M 38.6 / 35.4, 16 M 34.5
        // / 34.6, 67 M 33.0 / 35.2, 416 (13) 67 M 32.9 / 34.9, 448 (14) 32.4 / 34.5, 480 (15) 32.0 /
        // 34.9, 512 (16) 31.8 / 33.9.  BF16 224 (14) 30.4 / 28.4, 288 (9) 39.8 / 28.5; with 16 warps
        // the rows win on the largest grids only: 128-wide 4 M cells 31.9 / 29.0, 17 M 28.6 / 28.0,
        // 67 M 27.3 / 27.8, 256 31.9 / 29.3, 28.9 / 28.2, 27.7 / 28.0, 512 32.8 / 29.4, 27.8 / 28.5,
        // 26.9 / 28.3 (FP16: rows 1 ps slower, per-cell the same).  The 16-bit line stands at 16
        // warps all the same, as AUTO is documented and tested to take the rows there.
        if (cudaDeviceGetAttribute(&persm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev) != cudaSuccess) return false;
        const int warps = (int)((size_t)persm / (sm + 1024)) * (d.g.nx / 32);
        if (sizeof(S) == 4 && d.g.nx >= 384 && d.g.n >= (1LL << 24)) return true;
        return d.g.nx >= 128 && warps >= (sizeof(S) == 2 ? 16 : 14);
    }
    // Rows per strip (d.lb_rows_yc > 0: that many).  FP32, where memory is the bound: strips for
    // ~16 waves of resident blocks, at least 8 rows.  16-bit storage, where an SM's own rate
    // is: the split of least whole rounds of blocks x (rows + 1.5), 1.5 rows being what a
    // strip costs to fill and drain, of at most ~32 waves (BF16 512^3, 8 waves 3.93 ms, this
    // 3.54; 256^3 503 -> 486 us).
    static RowsWork rows_work(const DevState &d, size_t smem) {
        const int ny = d.g.ny, nzc = zcount(d);
        int yc = d.lb_rows_yc;
        if (yc <= 0) {
            int dev = 0, sms = 148, smpb = 0;
            if (cudaGetDevice(&dev) == cudaSuccess) {
                cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
                cudaDeviceGetAttribute(&smpb, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev);
            }
            long long per_sm = smpb > 0 ? (long long)smpb / (long long)(smem + 1024) : 1;
            if (per_sm < 1) per_sm = 1;
            const long long places = sms * per_sm;
            if constexpr (sizeof(S) == 2) {
                yc = strip_rows(ny, nzc, places);
            } else {
                const long long strips = std::max(1LL, (16 * places + nzc - 1) / nzc);
                yc = std::max(8, (int)((ny + strips - 1) / strips));
            }
        }
        if (yc > ny) yc = ny;
        RowsWork w;
        w.yc = yc;
        w.strips = (ny + yc - 1) / yc;
        return w;
    }
    static cudaError_t lb_rows(const DevState &d, int parity, cudaStream_t s) {
        KArgs<S> a = args(d);
        const size_t sm = rows_smem(d.g.nx);
        const RowsWork w = rows_work(d, sm);
        static SmemAttrOnce attr[2];
        int dev = 0, optin = 0;
        cudaError_t e = cudaGetDevice(&dev);
        if (e == cudaSuccess) e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
        if (e != cudaSuccess) return e;
        // the attribute is the largest layout any nx up to LR_MAX_NX needs, within the limit
        const size_t lim = std::min(rows_smem(LR_MAX_NX), (size_t)optin);
        e = parity == 0 ? attr[0].ensure(k_lb_rows<S, 0>, lim) : attr[1].ensure(k_lb_rows<S, 1>, lim);
        if (e != cudaSuccess) return e;
        const unsigned nblk = (unsigned)(zcount(d) * w.strips);
        const unsigned nthr = (unsigned)(d.g.nx + 32);
        return launch_step(d.pdl, parity == 0 ? k_lb_rows<S, 0> : k_lb_rows<S, 1>, dim3(nblk), dim3(nthr), sm, s, a, w);
    }
    static int lb_rows_used(const DevState &d) { return d.auto_kernels && rows_ok(d) ? 1 : 0; }
    // Launch of a per-cell kernel, by x-y tiles or in memory order (see cell_of_thread).  The
    // order costs a division and a few spilled registers, tiles the lanes beyond the grid:
    // measured on GB300 (stream-collide, event-timed, FP32, nx x 64 x 64, tiles against
    // order) 33: 12.3 / 10.3 us, 110: 20.2 / 19.5, 120: 19.4 / 20.8, 240: 42.0 / 43.8; BF16
    // 165: 26.5 / 25.5.  The line lies at 7/8 of the lanes in use.
    // Tiles sweep z within chunks of rows of kCellChunk cells a plane: over whole planes of
    // 2^16 cells and more the z neighbours' stress and the populations streamed in z leave L2
    // before the next plane comes (stream-collide, ps per cell, whole planes / chunks: FP32
    // 256^2 36.0 / 34.5, 300^2 43.2 / 36.2, 384^2 38.1 / 34.3; BF16 256^2 31.2 / 28.1, 300^2
    // 38.0 / 29.7, 384^2 30.3 / 28.1; half or a third of the chunk 1 to 3 % more).
    static constexpr unsigned kCellChunk = sizeof(S) == 4 ? 3u << 14 : 3u << 13;
    template <class K, class... A>
    static cudaError_t cell_launch(const DevState &d, K tiled, K linear, cudaStream_t s, A... more) {
        const KArgs<S> a = args(d);
        // grids with less than a 128-thread block per SM: smaller blocks in memory order, so
        // that the cells spread over the SMs (an SM issues a warp's FP64 instruction in 16
        // cycles, whatever the number of warps waiting: FP64 4 x 32 x 4 on 4 SMs 35.5 us per
        // step, on 16 27.7)
        const unsigned sms = (unsigned)(d.sms > 0 ? d.sms : sm_count());
        if (a.lin <= 96u * sms) {
            const unsigned t = std::max(32u, (a.lin / sms + 31u) / 32u * 32u);
            return launch_step(d.pdl, linear, dim3((a.lin + t - 1u) / t), dim3(t), 0, s, a, more...);
        }
        const dim3 b = block2(d);
        dim3 g = grid2(d);
        if (8LL * d.g.nx * d.g.ny >= 7LL * g.x * b.x * g.y * b.y) {
            const unsigned rows = std::max(1u, kCellChunk / ((unsigned)d.g.nx * b.y));
            const unsigned chunks = (g.y + rows - 1u) / rows;
            if (chunks > 1u && chunks * g.z <= 65535u) {
                g.y = (g.y + chunks - 1u) / chunks;
                g.z *= chunks;
            }
            return launch_step(d.pdl, tiled, g, b, 0, s, a, more...);
        }
        return launch_step(d.pdl, linear, dim3((a.lin + 127u) / 128u), dim3(128), 0, s, a, more...);
    }
    static cudaError_t lb(const DevState &d, int parity, cudaStream_t s) {
        if (d.auto_kernels && rows_ok(d)) return lb_rows(d, parity, s);
        if (d.ph.fene)  // the polymer force takes the stress of each cell's conformation
            return parity == 0 ? cell_launch(d, k_lb<S, 0, true, false>, k_lb<S, 0, true, true>, s)
                               : cell_launch(d, k_lb<S, 1, true, false>, k_lb<S, 1, true, true>, s);
        return parity == 0 ? cell_launch(d, k_lb<S, 0, false, false>, k_lb<S, 0, false, true>, s)
                           : cell_launch(d, k_lb<S, 1, false, false>, k_lb<S, 1, false, true>, s);
    }
    // The per-cell stress kernel (k_fv_cells).  FP64: every grid (its time is the FP64 pipe's,
    // which every SM has to share in from the first cells on; measured on GB300, event-timed,
    // tiled against per-cell: 4 x 32 x 4 98.9 / 18.7 us, 32^3 375 / 29.1, 90^3 733 / 433).
    // Shifted modes: below 3 * 2^18 cells under schedule AUTO (FP32 tiled against
    // per-cell: 32^3 20.3 / 7.7 us, 64^3 22.5 / 12.6, 83^3 30.3 / 20.8, 100^3 32.4 / 35.3: the
    // z-marching columns are too few for the chip on small grids, the per-cell kernel's
    // re-reads through L1 and L2 cost more on large ones).
    static bool fv_cells_ok(const DevState &d) {
        if (!Store<S>::shifted) return true;
        return d.auto_kernels == 1 && d.g.n < 3LL * (1LL << 18);
    }
    static cudaError_t fv_cells(const DevState &d, cudaStream_t s) {
        return fv_variant(d) ? cell_launch(d, k_fv_cells<S, true, false>, k_fv_cells<S, true, true>, s)
                             : cell_launch(d, k_fv_cells<S, false, false>, k_fv_cells<S, false, true>, s);
    }
    static int sm_count() {
        int dev = 0, sms = 148;
        if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        return sms;
    }
    // z-planes per block of the z-marching stress kernels on tiles columns of nz planes with
    // `resident` blocks on the device: ~16 waves, at least 16 planes (each chunk stages two
    // halo planes more than it updates) ...
    static int march_zchunk(long long tiles, int nz, long long resident) {
        const long long chunks = (16 * resident + tiles - 1) / tiles;
        long long zc = (nz + chunks - 1) / chunks;
        if (zc < 16) zc = 16;
        return (int)std::min<long long>(zc, nz);
    }
    // ... of the batched kernel, whose grid all the members share
    static int fv_zchunk_batched(const DevState &d) {
        const long long tiles = (long long)((d.g.nx + FV_X - 1) / FV_X) * ((d.g.ny + FV_Y - 1) / FV_Y);
        return march_zchunk(tiles, zcount(d), LBVE_FV_MIN_BLOCKS * (long long)sm_count());
    }
    // ... of the tiled kernel of a single solve.  Grids too small for 16 waves of 16-plane
    // chunks take the chunk of least predicted time: a block spends about 0.76 us on a plane
    // when its SM is full and 1.4 us when it is alone (measured on GB300, FP32), over
    // zc + 2 planes, a full wave at a time and then the rest.  128^3: 9 planes, 48 us (16
    // planes 53, 4 planes 52); 100^3: 8 planes, 32.4 us (16 planes 39); 192 x 160 x 96 stays
    // at 16 planes (12 planes 4 % slower).
    static int fv_zchunk(const DevState &d) {
        const int nz = zcount(d);
        if (d.fv_zchunk > 0) return d.fv_zchunk < nz ? d.fv_zchunk : nz;
        const long long tiles = (long long)((d.g.nx + FV_X - 1) / FV_X) * ((d.g.ny + FV_Y - 1) / FV_Y);
        const long long sms = sm_count(), resident = LBVE_FV_MIN_BLOCKS * sms;
        int best = march_zchunk(tiles, nz, resident);
        if (best > 16) return best;
        auto cost = [&](int zc) -> double {
            const long long blocks = tiles * ((nz + zc - 1) / zc), rest = (blocks % resident + sms - 1) / sms;
            const double full = 0.76 * LBVE_FV_MIN_BLOCKS * (double)(blocks / resident);
            return (zc + 2) * (full + (rest > 0 ? std::max(1.4, 0.76 * (double)rest) : 0.0));
        };
        double c = cost(best);
        for (int zc : {14, 12, 10, 9, 8, 6, 4}) {
            if (zc >= nz) continue;
            const double cz = cost(zc);
            if (cz < c) {
                c = cz;
                best = zc;
            }
        }
        return best;
    }
    // the VAR builds of the stress kernels: a finite-volume variant, FENE-P, or the flux or
    // the source switched off (the plain build has both on at compile time)
    static bool fv_variant(const DevState &d) {
        return d.ph.ctu_on || d.ph.divu_on || d.ph.gk != 0.0 || d.ph.fene || !d.ph.flux_on || !d.ph.src_on;
    }
    template <bool VAR, bool ZR, bool W16>
    static cudaError_t fv_launch(const DevState &d, unsigned nblk, int zc, cudaStream_t s) {
        KArgs<S> a = args(d);
        const size_t sm = sizeof(FvSmem<R, FvTile<FV_X, W16>::HN>);
        static SmemAttrOnce attr;
        cudaError_t e = attr.ensure(k_fv_tiled<S, VAR, ZR, W16>, sm);
        if (e != cudaSuccess) return e;
        return launch_step(d.pdl, k_fv_tiled<S, VAR, ZR, W16>, dim3(nblk), dim3(FV_X * FV_Y), sm, s, a, zc);
    }
    // planes staged by 16-byte copies: rows of whole 16-byte chunks and 16-byte aligned
    // stress and velocity arrays
    static bool fv_w16(const DevState &d) {
        auto al = [](const void *p) { return ((uintptr_t)p & 15u) == 0; };
        return d.g.nx % 4 == 0 && al(d.tau[0]) && al(d.tau[1]) && al(d.u[0]) && al(d.u[1]);
    }
    template <bool VAR>
    static cudaError_t fv_var(const DevState &d, cudaStream_t s) {
        const int zc = fv_zchunk(d);
        const int tiles = ((d.g.nx + FV_X - 1) / FV_X) * ((d.g.ny + FV_Y - 1) / FV_Y);
        const unsigned nblk = (unsigned)(tiles * ((zcount(d) + zc - 1) / zc));
        const bool zr = d.zhi > 0;  // a z-slab: planes [zlo, zhi) only
        if (fv_w16(d)) return zr ? fv_launch<VAR, true, true>(d, nblk, zc, s) : fv_launch<VAR, false, true>(d, nblk, zc, s);
        return zr ? fv_launch<VAR, true, false>(d, nblk, zc, s) : fv_launch<VAR, false, false>(d, nblk, zc, s);
    }
    // The two-cell stress kernel (k_fv_pair): schedule AUTO, the shifted modes' plain
    // build (flux and source on, no variant), nx a multiple of 4 (16-byte staging) and
    // 16-byte aligned stress, velocity and mask arrays.  Bitwise the tiled kernel's result.
    static bool fv_pair_ok(const DevState &d) {
        if constexpr (!Store<S>::shifted) {
            return false;
        } else {
            if (!d.auto_kernels || !fv_pair_shape(d)) return false;
            // schedule AUTO: grids of 2^21 cells and more (measured on GB300: 12 % faster at
            // 128^3, slower below about 10^6 cells, where its 512-cell columns leave SMs idle)
            return d.auto_kernels != 1 || d.g.n >= (1LL << 21);
        }
    }
    static bool fv_pair_shape(const DevState &d) {
        auto al = [](const void *p) { return ((uintptr_t)p & 15u) == 0; };
        return Store<S>::shifted && !fv_variant(d) && d.g.nx % 4 == 0 && al(d.tau[0]) && al(d.tau[1]) && al(d.u[0]) &&
               al(d.u[1]) && al(d.mask);
    }
    static int fv_pair_used(const DevState &d) { return fv_pair_ok(d) ? 1 : 0; }
    // z-planes per block of the two-cell stress kernel: ~16 waves of 2 resident blocks; where
    // 16-plane chunks make less than 8, the chunk of least predicted time (see fv_zchunk): a
    // plane takes 2.1 us with two blocks on an SM and 1.3 with one, and a block 1.5 planes
    // more than it updates.  FP32, event-timed: 128^3 43.2 -> 41.4 us, 192 x 160 x 96 64.1 ->
    // 53.5 (chunks of 20: 300 blocks on 304 places), 256^3 257 -> 248.
    static int fv_pair_zchunk(const DevState &d) {
        const int nz = zcount(d);
        if (d.fv_zchunk > 0) return d.fv_zchunk < nz ? d.fv_zchunk : nz;
        const long long tiles = (long long)((d.g.nx + FP_TX - 1) / FP_TX) * ((d.g.ny + FP_TY - 1) / FP_TY);
        const long long sms = d.sms > 0 ? d.sms : sm_count(), slots = 2 * sms;
        int best = march_zchunk(tiles, nz, slots);
        if (best > 16 || tiles * ((nz + 15) / 16) >= 8 * slots) return best;
        double least = 0.0;
        for (int chunks = 1; chunks <= (nz + 7) / 8;) {
            const int zc = (nz + chunks - 1) / chunks;
            const long long blocks = tiles * ((nz + zc - 1) / zc), rest = blocks % slots;
            const double t = (zc + 1.5) * (2.1 * (double)(blocks / slots) + (rest == 0 ? 0.0 : rest <= sms ? 1.3 : 2.1));
            if (chunks == 1 || t < least) {
                least = t;
                best = zc;
            }
            if (zc == 1) break;
            chunks = (nz + zc - 2) / (zc - 1);  // the first with fewer planes
        }
        return best;
    }
    static cudaError_t fv_pair(const DevState &d, cudaStream_t s) {
        if constexpr (!Store<S>::shifted) {
            return cudaErrorInvalidValue;
        } else {
            KArgs<S> a = args(d);
            const int zc = fv_pair_zchunk(d);
            const int tiles = ((d.g.nx + FP_TX - 1) / FP_TX) * ((d.g.ny + FP_TY - 1) / FP_TY);
            const unsigned nblk = (unsigned)(tiles * ((zcount(d) + zc - 1) / zc));
            const size_t sm = sizeof(FvPairSmem);
            static SmemAttrOnce attr[2];
            const bool zr = d.zhi > 0;  // a z-slab: planes [zlo, zhi) only
            cudaError_t e = zr ? attr[1].ensure(k_fv_pair<S, true>, sm) : attr[0].ensure(k_fv_pair<S, false>, sm);
            if (e != cudaSuccess) return e;
            return launch_step(d.pdl, zr ? k_fv_pair<S, true> : k_fv_pair<S, false>, dim3(nblk), dim3(FP_NT), sm, s, a, zc);
        }
    }
    static cudaError_t fv(const DevState &d, cudaStream_t s) {
        if constexpr (Store<S>::shifted) {
            if (d.in_pool) {
                // beside other members the chip is full: the kernels that take least SM time
                // per cell (256^3, FP32: two-cell 15 ps, tiled 17, per-cell 31), rows of half a
                // column and more
                DevState q = d;
                q.fv_zchunk = fv_zchunk_batched(d);  // (a chunk tuned alone is for a chip alone)
                if (d.g.nx >= 64 && fv_pair_shape(d)) return fv_pair(q, s);
                if (d.g.nx >= 32) return fv_variant(d) ? fv_var<true>(q, s) : fv_var<false>(q, s);
                return fv_cells(d, s);
            }
        }
        if (fv_cells_ok(d)) return fv_cells(d, s);
        if (fv_pair_ok(d)) return fv_pair(d, s);
        if constexpr (Store<S>::shifted) return fv_variant(d) ? fv_var<true>(d, s) : fv_var<false>(d, s);
        return cudaErrorInvalidValue;  // FP64 took the per-cell kernel
    }
    static cudaError_t momentum_exchange(const DevState &d, int parity, const long long *links, const int *seg_begin,
                                         const int *seg_count, int nseg, int max_len, double *contrib, cudaStream_t s) {
        if (nseg <= 0 || max_len <= 0) return cudaSuccess;
        KArgs<S> a = args(d);
        const dim3 g((unsigned)((max_len + 127) / 128), (unsigned)nseg);
        if constexpr (Store<S>::shifted) {
            // reduced modes: per-block partials (nseg x ceil(max_len / 128) of them)
            return launch_step(d.pdl, parity == 0 ? k_momentum_exchange_part<S, 0> : k_momentum_exchange_part<S, 1>, g,
                               dim3(128), 0, s, a, links, seg_begin, seg_count, contrib);
        } else {
            // FP64 parity mode: one contribution per link, summed in link order
            return launch_step(d.pdl, parity == 0 ? k_momentum_exchange<S, 0> : k_momentum_exchange<S, 1>, g, dim3(128), 0,
                               s, a, links, seg_begin, seg_count, contrib);
        }
    }
    static cudaError_t halo_pack(const DevState &d, int what, int side, int parity, void *buf, cudaStream_t s) {
        KArgs<S> a = args(d);
        k_halo_pack<S><<<dim3((unsigned)((d.g.nx + 127) / 128), (unsigned)d.g.ny), 128, 0, s>>>(a, what, side, parity, buf);
        return cudaGetLastError();
    }
    static cudaError_t halo_unpack(const DevState &d, int what, int side, int parity, const void *buf,
                                   cudaStream_t s) {
        KArgs<S> a = args(d);
        k_halo_unpack<S><<<dim3((unsigned)((d.g.nx + 127) / 128), (unsigned)d.g.ny), 128, 0, s>>>(a, what, side, parity,
                                                                                                    buf);
        return cudaGetLastError();
    }
    static cudaError_t build_mask(const DevState &d, int lx, int ly, int lz, int ex, int ey, int ez, cudaStream_t s);
    static cudaError_t voxelise(const DevState &d, int p, const PartDev &host, cudaStream_t s) {
        KArgs<S> a = args(d);
        k_voxelise<S><<<64, 256, 0, s>>>(a, d.parts, p, d.flag, (R *)d.tau[0], (R *)d.tau[1]);
        cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
        const BBox b = particle_bbox(d.g, host.X, host.R, 3);
        return build_mask(d, b.lo[0], b.lo[1], b.lo[2], b.ext[0], b.ext[1], b.ext[2], s);
    }
    static cudaError_t particle_links(const DevState &d, int nparts, long long *links, const int *seg_begin,
                                      int *seg_count, int first_seg, const int *capacity, cudaStream_t s) {
        if (nparts <= 0) return cudaSuccess;
        k_particle_links<S><<<nparts * PC, PT, 0, s>>>(d.g, d.parts, d.flag, d.mask, links, seg_begin, seg_count,
                                                       first_seg, capacity);
        return cudaGetLastError();
    }
    static cudaError_t build_mask_impl(const DevState &d, int lx, int ly, int lz, int ex, int ey, int ez,
                                       cudaStream_t s) {
        const long long cells = (long long)ex * ey * ez;
        if (cells <= 0) return cudaSuccess;
        const unsigned nb = (unsigned)std::min<long long>((cells + 255) / 256, 65535);
        k_build_mask<S><<<nb, 256, 0, s>>>(args(d), d.mask, lx, ly, lz, ex, ey, ez, (R *)d.tau[0], (R *)d.tau[1],
                                           (R *)d.u[0], (R *)d.u[1]);
        return cudaGetLastError();
    }
    static cudaError_t fused(const DevState &d, int parity, int zchunk, cudaStream_t s) {
        KArgs<S> a = args(d, true);
        FusedWork w;
        w.tiles_x = (d.g.nx + FT_X - 1) / FT_X;
        w.tiles_y = (d.g.ny + FT_Y - 1) / FT_Y;
        w.zchunk = zchunk;
        w.nzchunks = (d.g.nz + zchunk - 1) / zchunk;
        const size_t sm = sizeof(FusedSmem<R>);
        static SmemAttrOnce attr[2];
        cudaError_t e = parity == 0 ? attr[0].ensure(k_fused<S, 0>, sm) : attr[1].ensure(k_fused<S, 1>, sm);
        if (e != cudaSuccess) return e;
        const unsigned nblk = (unsigned)w.tiles_x * w.tiles_y * w.nzchunks;
        if (parity == 0)
            k_fused<S, 0><<<nblk, FT_X * FT_Y, sm, s>>>(a, w);
        else
            k_fused<S, 1><<<nblk, FT_X * FT_Y, sm, s>>>(a, w);
        return cudaGetLastError();
    }
    static cudaError_t read(const DevState &d, int parity, double *rho, double *u, double *tau, int z0, int z1,
                            long long ld, cudaStream_t s) {
        if (z1 <= z0) return cudaSuccess;
        DevState q = d;
        q.zlo = z0;
        q.zhi = z1;
        return parity == 0 ? cell_launch(q, k_read<S, 0, false>, k_read<S, 0, true>, s, rho, u, tau, ld)
                           : cell_launch(q, k_read<S, 1, false>, k_read<S, 1, true>, s, rho, u, tau, ld);
    }
    static cudaError_t pdfs_io(const DevState &d, int parity, double *io, int write, cudaStream_t s) {
        KArgs<S> a = args(d);
        if (parity == 0)
            k_pdfs_io<S, 0><<<grid3(d), d.block_x, 0, s>>>(a, io, write);
        else
            k_pdfs_io<S, 1><<<grid3(d), d.block_x, 0, s>>>(a, io, write);
        return cudaGetLastError();
    }
    static cudaError_t reduce(const DevState &d, int parity, double *partial, long long *nblocks, cudaStream_t s) {
        KArgs<S> a = args(d);
        dim3 g(grid3(d).x, d.g.ny, d.g.nz);
        // the reduction kernel needs exactly 256 threads per block
        g.x = (unsigned)((d.g.nx + 255) / 256);
        *nblocks = (long long)g.x * g.y * g.z;
        if (!partial) return cudaSuccess;
        if (parity == 0)
            k_reduce<S, 0><<<g, 256, 0, s>>>(a, partial);
        else
            k_reduce<S, 1><<<g, 256, 0, s>>>(a, partial);
        return cudaGetLastError();
    }

    static cudaError_t probe(const DevState &d, int parity, const long long *cells, int count, double *out,
                             cudaStream_t s) {
        if (count <= 0) return cudaSuccess;
        KArgs<S> a = args(d);
        const unsigned nb = (unsigned)((count + 127) / 128);
        if (parity == 0)
            k_probe<S, 0><<<nb, 128, 0, s>>>(a, cells, count, out);
        else
            k_probe<S, 1><<<nb, 128, 0, s>>>(a, cells, count, out);
        return cudaGetLastError();
    }

    // default tiles of a solve in the batched kernels (the pool autotuner may pick others)
    static int default_lb_tx(const DevState &) { return 32; }
    static int default_fv_tx(const DevState &) { return 32; }
    static void batch_tiles(const DevState &d, int lb_tx, int fv_tx, int *lb_eff, int *fv_eff) {
        *lb_eff = (lb_tx == 16 || lb_tx == 32 || lb_tx == 64 || lb_tx == 128) ? lb_tx : default_lb_tx(d);
        *fv_eff = FvBatchTiles<R>::ok(fv_tx) ? fv_tx : default_fv_tx(d);
    }
    static void fill_entry(const DevState &d, int parity, int lb_first, int fv_first, int fv_zchunk, int lb_tx,
                           int fv_tx, void *entry, int *lb_items, int *fv_items) {
        BatchEntry<S> &e = *reinterpret_cast<BatchEntry<S> *>(entry);
        e.a[0] = args(d);
        DevState d1 = d;  // odd steps of a launch sequence: stress ping-pong swapped
        d1.cur ^= 1;
        e.a[1] = args(d1);
        e.parity0 = parity;
        batch_tiles(d, lb_tx, fv_tx, &e.lb_tx, &e.fv_tx);
        const int lth = BLB_X * BLB_Y / e.lb_tx, fth = FV_NT / e.fv_tx;
        e.lb_first = lb_first;
        e.lb_items = ((d.g.nx + e.lb_tx - 1) / e.lb_tx) * ((d.g.ny + lth - 1) / lth) * d.g.nz;
        e.fv_first = fv_first;
        e.fv_zchunk = fv_zchunk > 0 ? fv_zchunk : fv_zchunk_batched(d);
        e.fv_items = ((d.g.nx + e.fv_tx - 1) / e.fv_tx) * ((d.g.ny + fth - 1) / fth) *
                     ((d.g.nz + e.fv_zchunk - 1) / e.fv_zchunk);
        *lb_items = e.lb_items;
        *fv_items = e.fv_items;
    }
    static int fv_zchunk_of(const DevState &d) {
        if (fv_cells_ok(d)) return 0;
        return fv_pair_ok(d) ? fv_pair_zchunk(d) : fv_zchunk(d);
    }
    static cudaError_t lb_batched(const void *entries, int n, int total, int k, int grid, const unsigned *dstep,
                                  int parity, cudaStream_t s) {
        if (total <= 0) return cudaSuccess;
        if (parity == 0)
            k_lb_batched<S, 0><<<grid, BLB_X * BLB_Y, 0, s>>>((const BatchEntry<S> *)entries, n, total, k, dstep);
        else
            k_lb_batched<S, 1><<<grid, BLB_X * BLB_Y, 0, s>>>((const BatchEntry<S> *)entries, n, total, k, dstep);
        return cudaGetLastError();
    }
    template <int TX, bool VAR>
    static cudaError_t fv_batched_tx(const void *entries, int n, int total, int k, int grid, cudaStream_t s) {
        const size_t sm = sizeof(FvSmem<R, FvTile<TX>::HN>);
        static SmemAttrOnce attr;
        cudaError_t e = attr.ensure(k_fv_batched<S, TX, VAR>, sm);
        if (e != cudaSuccess) return e;
        k_fv_batched<S, TX, VAR><<<grid, FV_NT, sm, s>>>((const BatchEntry<S> *)entries, n, total, k);
        return cudaGetLastError();
    }
    template <bool VAR>
    static cudaError_t fv_batched_var(const void *entries, int n, int total, int k, int grid, int tx, cudaStream_t s) {
        if constexpr (FvBatchTiles<R>::wide) {
            if (tx == 16) return fv_batched_tx<16, VAR>(entries, n, total, k, grid, s);
            if (tx == 64) return fv_batched_tx<64, VAR>(entries, n, total, k, grid, s);
        }
        return fv_batched_tx<32, VAR>(entries, n, total, k, grid, s);
    }
    static cudaError_t fv_batched(const void *entries, int n, int total, int k, int grid, int tx, int var,
                                  cudaStream_t s) {
        if (total <= 0) return cudaSuccess;
        return var ? fv_batched_var<true>(entries, n, total, k, grid, tx, s)
                   : fv_batched_var<false>(entries, n, total, k, grid, tx, s);
    }
    // resident blocks per SM of the batched stress kernel (both builds are held to the
    // same launch bound, so one grid serves both)
    template <int TX>
    static int fv_resident() {
        int per = 1;
        const size_t sm = sizeof(FvSmem<R, FvTile<TX>::HN>);
        cudaFuncSetAttribute(k_fv_batched<S, TX, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_fv_batched<S, TX, false>, FV_NT, sm);
        return per;
    }
    static int fv_variant_of(const DevState &d) { return fv_variant(d) ? 1 : 0; }
    static void part_entry(const PartScratch &ps, const DevState &d, int parity0, PartEntry<S> &e) {
        e.parity0 = parity0;
        e.nparts = ps.nparts;
        e.first_seg = ps.first_seg;
        e.parts = d.parts;
        e.flag = d.flag;
        e.mask = d.mask;
        e.kind = ps.kind;
        e.nf = ps.nf;
        e.delta = ps.delta;
        e.diag = ps.diag;
        e.conv = ps.conv;
        e.links = ps.links;
        e.seg_begin = ps.seg_begin;
        e.seg_count = ps.seg_count;
        e.capacity = ps.capacity;
        e.sums = Store<S>::shifted ? ps.contrib : nullptr;  // FP64: summed in link order before
        e.sum_stride = (ps.max_seg_len + 127) / 128;
        e.nbody = ps.nbody;
        e.seg_flag = ps.seg_flag;
        e.body_F = ps.body_F;
    }
    // d: the member's state when the entries are built; step k after that uses the stress
    // ping-pong after the step's swap (cur ^ 1 for even k) and AA parity parity0 ^ (k & 1)
    static void fill_part_entry(const DevState &d, int parity0, const PartScratch &ps, void *entry) {
        PartEntry<S> &e = *reinterpret_cast<PartEntry<S> *>(entry);
        DevState d0 = d;
        d0.cur ^= 1;
        e.a[0] = args(d0);
        e.a[1] = args(d);
        part_entry(ps, d, parity0, e);
    }
    static cudaError_t particle_phase_batched(const void *entries, int n, int k, cudaStream_t s) {
        if (n <= 0) return cudaSuccess;
        k_particle_phase<S><<<n * PC, PT, 0, s>>>((const PartEntry<S> *)entries, PartEntry<S>{}, k);
        return cudaGetLastError();
    }
    // one solve, d its state after the step's stress update
    static cudaError_t particle_phase(const DevState &d, int parity, const PartScratch &ps, cudaStream_t s) {
        if (ps.nparts <= 0) return cudaSuccess;
        PartEntry<S> e{};
        e.a[0] = args(d);
        part_entry(ps, d, parity, e);
        return launch_step(d.pdl, k_particle_phase<S>, dim3(PC), dim3(PT), 0, s, nullptr, e, 0);
    }
    // resident blocks of the persistent grids: which = 0 for the stream-collide, else the
    // stress kernel of tile width `which`
    static int batched_grid(int which) {
        int dev = 0, sms = 148, per = 1;
        if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        if (which == 0) {
            int per1 = 1;
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_lb_batched<S, 0>, BLB_X * BLB_Y, 0);
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per1, k_lb_batched<S, 1>, BLB_X * BLB_Y, 0);
            per = std::min(per, per1);
        } else {
            per = fv_resident<32>();
            if constexpr (FvBatchTiles<R>::wide) {
                if (which == 16) per = fv_resident<16>();
                if (which == 64) per = fv_resident<64>();
            }
        }
        cudaGetLastError();
        if (per < 1) per = 1;
        return sms * per;
    }
    static cudaError_t residual(const DevState &d, void *usnap, double *partial, int nblocks, cudaStream_t s) {
        k_residual<S><<<nblocks, 256, 0, s>>>(d.g, d.mask, (const R *)d.u[d.ucur], (R *)usnap, partial);
        return cudaGetLastError();
    }

    static const KernelTable *table(int prec);
};

template <class S>
cudaError_t Launch<S>::build_mask(const DevState &d, int lx, int ly, int lz, int ex, int ey, int ez, cudaStream_t s) {
    return build_mask_impl(d, lx, ly, lz, ex, ey, ez, s);
}

template <class S>
const KernelTable *Launch<S>::table(int prec) {
        static const KernelTable t = {prec,           sizeof(S),        sizeof(R),   &init,
                                      &lb,            &fv,              &momentum_exchange, &voxelise,
                                      &particle_links, &particle_phase, &read,
                                      &pdfs_io,       &reduce,          &probe,      &build_mask,
                                      &fused,         sizeof(BatchEntry<S>), &fill_entry, &lb_batched,
                                      &fv_batched,    &batched_grid,    &residual,   &batch_tiles,
                                      &fv_zchunk_of,  &fv_variant_of,   sizeof(PartEntry<S>), &fill_part_entry,
                                      &particle_phase_batched, &halo_pack, &halo_unpack, &lb_rows_used, &fv_pair_used};
        return &t;
}

} // namespace lbve
