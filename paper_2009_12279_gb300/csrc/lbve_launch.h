// lbve_launch.h -- internal interface between the host library (lbve_api.cu) and the
// per-precision kernel translation units: parameter structs passed by value to the
// kernels and a table of host-side launchers per PDF storage type.
#pragma once

#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

namespace lbve {

constexpr int Q = 19;
constexpr int FLAG_FLUID = 0;
constexpr int FLAG_NOSLIP = 1;
constexpr int FLAG_WALL0 = 2;
constexpr int MAX_WALL = 16;
constexpr int FLAG_PART0 = 64;
constexpr int MAX_PART = 64;

struct Geo {
    int nx, ny, nz;
    int per[3];
    long long n;  // nx*ny*nz
    long long np; // stride between the arrays of one field (n rounded up to 64)
};

template <class R>
struct Phys {
    R omega_p, omega_m;
    R A, B;        // 3 (1 - omega-/2) and 1 - omega+/2 of the forcing term
    R ep_l, inv_l; // eta_p / lambda_p and 1 / lambda_p
    R g[3];
    R rho0;        // shift base of the stored deviations (0 in FP64 mode)
    R rho_ref;     // reference density rho0 of the solve (all modes)
    R scale, inv_scale;
    int flux_on, src_on;
    int ctu_on;   // face fluxes scaled by the transverse overlap of the displaced donor cell
    int divu_on;  // the tau div(u) source term
    R gk;         // alpha / eta_p of the Giesekus source term (0: Oldroyd-B)
    int fene;     // FENE-P: the stress arrays hold the conformation tensor A
    R fene_L2;    // its maximum extensibility L^2
    R eta_p, lam; // polymer viscosity and relaxation time (stress <-> conformation)
    R wall_vel[MAX_WALL][3];
};

// FP64 rigid-sphere state used by the particle kernels.
struct PartDev {
    double X[3], v[3], w[3];
    double R, rho_p, m, I;
    double Fext[3], Text[3];
    double Fme[3], Tme[3];
    double dP[3], dL[3];
    int changed;  // 1 when the last fill/drain converted cells (links must be rebuilt)
};

// A solve's particle scratch and link arrays, as the particle-phase kernels take them.
struct PartScratch {
    int nparts, first_seg;
    uint8_t *kind, *nf;
    double *delta, *diag;
    int *conv;
    long long *links;
    const int *seg_begin;
    int *seg_count;
    const int *capacity;
    // bodies (wall classes and particles) and their momentum-exchange contributions
    int nbody, max_seg_len;
    const int *seg_flag;
    const double *contrib;
    double *body_F;
};

// Device buffers of one solve.
struct DevState {
    Geo g;
    Phys<double> ph;  // converted to the kernel's real type by the launchers
    void *f;          // 19 * np PDF storage elements
    void *tau[2];     // 6 * np reals each (ping-pong)
    void *u[2];       // 3 * np reals each (velocity of the last stream-collide, ping-pong)
    int ucur;         // index of the velocity written by the last stream-collide
    uint32_t *mask;   // np neighbour masks
    uint8_t *flag;    // np bytes
    PartDev *parts;   // MAX_PART entries
    int cur;          // index of tau^t in tau[]
    int block_x;      // threads per block along x
    int fv_zchunk;    // z-planes per block of the stress kernel (0: by the SM count)
    unsigned step;    // index of the step the next stream-collide performs (low 32 bits)
    // instability flag: a word of mapped page-locked host memory (its device address)
    // that the stream-collide sets to 1 when a fluid cell has rho <= 0, |u|^2 >= 1/3
    // (the lattice sound speed squared) or a NaN; nullptr: no check
    unsigned *bad = nullptr;
    // planes [zlo, zhi) that the step kernels compute (zhi 0: all); the planes outside are
    // the ghost planes of a z-slab of a decomposed domain, filled by the halo exchange
    int zlo = 0, zhi = 0;
    // offset of this grid's cell indices in the decomposed domain's (rounding keys of the
    // 16-bit stores use global cells, so a slab rounds as the undecomposed domain does)
    unsigned key_base = 0;
    // the row-pipelined stream-collide (k_lb_rows) and the two-cell stress kernel
    // (k_fv_pair) where the grid allows them: 0 never (schedule SPLIT), 1 on large grids
    // only (AUTO), 2 always (PIPELINED); else the per-cell stream-collide and the tiled
    // stress kernel.  lb_rows_yc: rows per strip of the row pipeline (0: by the SM count)
    int auto_kernels = 0;
    int lb_rows_yc = 0;
    // 1: the step's kernels are launched as programmatic dependents of one another (see
    // launch_step); 0: plain launches (pools, phases, captured streams)
    int pdl = 0;
    int sms = 0;  // SMs of the device (0: asked for when needed)
    // a member of a pool stepped by kernels of its own beside the others': the stress kernel
    // of most cells per SM and time, whatever the grid's size, and rounding keys counted from
    // *dstep on (the launches are replayed from a graph)
    int in_pool = 0;
    const unsigned *dstep = nullptr;
};

#ifdef __CUDACC__
// A step kernel may be launched before its predecessor in the stream has finished: it waits
// here, before it reads or writes anything, until that one is complete and its writes are
// visible.  Every thread of every step kernel passes here first.  What its predecessors write
// changes during its own lifetime, so no step kernel takes an array that a step kernel writes
// as `const ... *__restrict__`: that would promise the compiler that nobody does, and allow it
// a non-coherent load or one above this wait.
__device__ __forceinline__ void step_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
// ... and lets its own successor be launched once all its blocks have come here.  After
// a block's loads, not at its start: blocks that wait from early on take the slots of, and
// were measured to spread unevenly among, those at work (FP64 32^3: 185 us per step instead
// of 65).  FP64 kernels, whose time is arithmetic, leave it to their blocks' ends.
__device__ __forceinline__ void step_next() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
#endif

// Launch of a step kernel.  With pdl its launch latency overlaps the tail of the kernel
// before it: measured on GB300, FP32, per step of two kernels 32^3 8.4 -> 5.4 us, 64^3
// 18.6 -> 14.7.
template <class... P, class... A>
inline cudaError_t launch_step(int pdl, void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t s,
                               A &&...args) {
    cudaLaunchConfig_t c{};
    c.gridDim = grid;
    c.blockDim = block;
    c.dynamicSmemBytes = smem;
    c.stream = s;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    c.attrs = &at;
    c.numAttrs = pdl ? 1 : 0;
    return cudaLaunchKernelEx(&c, kernel, static_cast<P>(args)...);
}

// Steps of a pool's replayed graph, an even number, for steps of `nodes` kernels each: at most
// about GRAPH_NODES kernels to capture, instantiate and keep, however long a call is.  A call
// of more steps than the longest block takes the block of at least half of it that leaves the
// fewest steps to capture (100 steps, at most 30: six blocks of 16 and four steps).  48 members
// of the serving mix, some 130 kernels a step, BF16, ms of the first call after an admission
// and of a replay: 25 steps in one graph 27.0 / 16.9; with blocks of at most 1024, 2048 and 4096
// kernels 20.0 / 17.0, 21.3 / 17.0 and 27.7 / 16.8 (one graph); 100 steps 111 / 68.0; 71.9 / 68.3,
// 73.5 / 67.6, 75.8 / 67.9; 1000 steps 1201 / 686 (402 MB on the device); 692 / 684, 690 / 679,
// 692 / 679 (54 MB).
constexpr long long GRAPH_NODES = 4096;
inline int graph_block_steps(long long nodes, int nsteps) {
    const long long fit = GRAPH_NODES / (nodes > 0 ? nodes : 1);
    const int most = fit < 2 ? 2 : (int)(fit / 2 * 2);
    if (nsteps <= most) return most;
    int best = most, least = most + (nsteps - 1) % most + 1;
    for (int b = most - 2; b >= 2 && 2 * b >= most; b -= 2) {
        const int captured = b + (nsteps - 1) % b + 1;
        if (captured < least) best = b, least = captured;
    }
    return best;
}

// Rows per strip of a split of ny rows on each of nz planes into n equal strips, n nz at most
// 32 places: the split of least whole rounds of `places` blocks x (rows + 1.5).  Every launch
// asks: only the n at which the rows change are looked at, 2 sqrt(ny) of them at most
// (128 x 32768 x 1 cells: every n took 62 us per launch).
inline int strip_rows(int ny, int nz, long long places) {
    int yc = ny;
    long long best = -1;
    for (long long n = 1; n <= ny && (n == 1 || n * nz <= 32 * places);) {
        const long long rows = (ny + n - 1) / n, strips = (ny + rows - 1) / rows;
        const long long cost = (strips * nz + places - 1) / places * (2 * rows + 3);
        if (best < 0 || cost < best) best = cost, yc = (int)rows;
        if (rows == 1) break;
        n = (ny + rows - 2) / (rows - 1);  // the first n with fewer rows
    }
    return yc;
}

struct KernelTable {
    int prec;          // lbve_pdf_prec
    size_t pdf_bytes;  // bytes per stored PDF
    size_t real_bytes; // bytes per stress / velocity value
    cudaError_t (*init)(const DevState &, const double *rho, const double *u, const double *tau, long long r0,
                        long long count, long long ld, cudaStream_t);
    cudaError_t (*lb)(const DevState &, int parity, cudaStream_t);
    cudaError_t (*fv)(const DevState &, cudaStream_t);
    // FP64: 8 doubles per link in contrib; shifted modes: 8 doubles per (segment, block of
    // 128 links), ceil(max_len / 128) blocks per segment
    cudaError_t (*momentum_exchange)(const DevState &, int parity, const long long *links, const int *seg_begin,
                                     const int *seg_count, int nseg, int max_len, double *contrib, cudaStream_t);
    cudaError_t (*voxelise)(const DevState &, int p, const PartDev &host, cudaStream_t);
    cudaError_t (*particle_links)(const DevState &, int nparts, long long *links, const int *seg_begin, int *seg_count,
                                  int first_seg, const int *capacity, cudaStream_t);
    // particle phase of one solve after its stress update: in the reduced modes the body
    // sums of the step's momentum exchange, then the particles' update, fill/drain (on PDFs
    // in AA parity `parity`) and links
    cudaError_t (*particle_phase)(const DevState &, int parity, const PartScratch &, cudaStream_t);
    cudaError_t (*read)(const DevState &, int parity, double *rho, double *u, double *tau, int z0, int z1,
                        long long ld, cudaStream_t);
    cudaError_t (*pdfs_io)(const DevState &, int parity, double *io, int write, cudaStream_t);
    cudaError_t (*reduce)(const DevState &, int parity, double *partial, long long *nblocks, cudaStream_t);
    cudaError_t (*probe)(const DevState &, int parity, const long long *cells, int count, double *out, cudaStream_t);
    cudaError_t (*build_mask)(const DevState &, int lx, int ly, int lz, int ex, int ey, int ez, cudaStream_t);
    cudaError_t (*fused)(const DevState &, int parity, int zchunk, cudaStream_t);
    // batched schedule (pools)
    size_t batch_entry_bytes;
    // lb_tx / fv_tx: the solve's tile widths in the batched kernels (0: default by nx)
    void (*fill_entry)(const DevState &, int parity, int lb_first, int fv_first, int fv_zchunk, int lb_tx, int fv_tx,
                       void *entry, int *lb_items, int *fv_items);
    // dstep: device counter of the steps since the entries were built (their step index base)
    cudaError_t (*lb_batched)(const void *entries, int n, int total, int k, int grid, const unsigned *dstep,
                              int parity, cudaStream_t);  // entries all at AA parity `parity` at step k
    // stress update of the solves with stress tile width tx (entries: that group only);
    // var: some solve of the group uses a finite-volume variant
    cudaError_t (*fv_batched)(const void *entries, int n, int total, int k, int grid, int tx, int var, cudaStream_t);
    int (*batched_grid)(int which);  // resident blocks: 0 stream-collide, else stress tile width
    cudaError_t (*residual)(const DevState &, void *usnap, double *partial, int nblocks, cudaStream_t);
    // the tile widths fill_entry will use for requested widths (0: default by nx)
    void (*batch_tiles)(const DevState &, int lb_tx, int fv_tx, int *lb_eff, int *fv_eff);
    // z-planes per block the stress kernel will use, 0: the per-cell kernel, which has no chunks
    int (*fv_zchunk_of)(const DevState &);
    int (*fv_variant_of)(const DevState &);  // 1 when the solve uses a finite-volume variant
    // pools: the particle phase of every member with particles in one launch; entries
    // built per member like the batch entries
    size_t part_entry_bytes;
    void (*fill_part_entry)(const DevState &, int parity0, const PartScratch &, void *entry);
    cudaError_t (*particle_phase_batched)(const void *entries, int n, int k, cudaStream_t);
    // z-slab halo exchange: what 0 PDFs of the last stream-collide (its AA parity), 1 u,
    // 2 tau; side 0 the low z side, 1 the high one; buf a device buffer of plane-major
    // values (halo_values(what) per cell of an x-y plane, storage type for the PDFs)
    cudaError_t (*halo_pack)(const DevState &, int what, int side, int parity, void *buf, cudaStream_t);
    cudaError_t (*halo_unpack)(const DevState &, int what, int side, int parity, const void *buf, cudaStream_t);
    int (*lb_rows_used)(const DevState &);  // 1 when the stream-collide runs the row pipeline
    int (*fv_pair_used)(const DevState &);  // 1 when the stress update runs two cells per thread
};

// Bounding-box side used to size the per-particle scratch (cells within R + margin).
inline int particle_box_side(double R, int margin) {
    int c = (int)R;
    if ((double)c < R) ++c;
    return 2 * c + 2 * margin + 3;
}

const KernelTable *table_f64();
const KernelTable *table_f32();
const KernelTable *table_f16();
const KernelTable *table_bf16();

} // namespace lbve
