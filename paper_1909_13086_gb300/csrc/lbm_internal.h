// lbm_internal.h -- shared between the host API (lbm_api.cu) and the sweep
// kernels (sweep_*.cu).  Not part of the public C ABI (include/lbm.h).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace btrirt {

enum Problem { kCavity = 0, kStefan = 1 };

// What one launch of the lattice kernel does.
enum Mode {
    kSweep = 0,      // stream + collide, write the next populations
    kSweepDiag = 1,  // same, plus the fused diagnostics reductions
    kFields = 2,     // stream + macroscopic step only: write the fields, no populations
};

// How populations move from one step to the next.  Pull: two buffers, every
// sweep pulls f*_i(x - c_i) from src and writes f*_i(x) into its own slot i of
// dst ("the pull layout": slot i of cell x holds f*_i(x)).  One buffer, two
// alternating sweeps (src == dst; the AA pattern of Bailey et al. 2009):
//   push  -- from the pull layout: pull as above, then put f*_i(x) into slot
//            opp(i) of cell x + c_i, or into the cell's own slot i where
//            x + c_i lies beyond a wall;
//   local -- from the pushed layout: f_i(x) is the cell's own slot opp(i) (a
//            wall's incoming population then takes the wall rule), and f*_i(x)
//            goes to its own slot i: the pull layout again.
// Each cell reads and writes the same 18 locations in either sweep, so no two
// cells touch one location, and the populations are those of the pull sweeps.
// The narrow forms are the same sweeps with one cell per thread and accesses of one value
// each, where the others take two (launch_mode).
enum Streaming { kPull = 0, kAAPush = 1, kAALocal = 2, kPullNarrow = 3, kAAPushNarrow = 4, kAALocalNarrow = 5 };

// Population layout in device memory ("tile-major structure of arrays").
// The lattice is cut into column tiles of kTW cells.  Within a tile, each row
// holds the 18 planes (f_0..f_8, g_0..g_8) one after the other, kTW values
// each, and rows follow one another:
//     index(x, y, p) = ((x / kTW) * ny + y) * 18 * kTW + p * kTW + x % kTW.
// A warp's 18 loads of one cell row are then one base register plus
// compile-time offsets (plane p: p*kTW; row above / below: -/+ 18*kTW).
constexpr int kTW = 128;  // tile width (fastest of 128/256/512 on GB300); a sweep's block has kTW
                          // threads, or kTW / 2 with two cells each
constexpr int kPlanes = 18;
constexpr int kRS = kPlanes * kTW;  // elements per tile row

__host__ __device__ inline long long pop_index(int x, int y, int p, int ny) {
    return ((long long)(x / kTW) * ny + y) * kRS + (long long)p * kTW + (x % kTW);
}

// FP64 diagnostics record living in device memory (one per handle).
struct DevRecord {
    double step;      // step the record belongs to
    double melt_sum;  // sum f_l
    double H_sum;     // sum H
    double Q_last;    // heated-wall inflow of the last step
    double Q_cum;     // running sum of Q_last
    double max_u;     // max |u|
    double nan_flag;  // 1 if a non-finite H or rho was seen
    double valid;     // 1 once the fields of `step` have been reduced
    unsigned long long counter;  // steps taken: advanced by every sweep on the
                                 // device, so that replayed CUDA graphs stamp
                                 // records correctly (an integer: GB300's FP64
                                 // pipe is narrow, and a sweep's warps would
                                 // each issue the predicated FP64 add)
    unsigned long long rng[2];   // stochastic-rounding step seeds, one word per buffer parity
    double timeout;   // 1 once a bounded device wait ran out (staged sweep)
};

// Arguments of every lattice kernel, passed by value.  16-byte aligned, so
// that a batch entry's argument sets start on 16-byte pieces.
template <typename real>
struct alignas(16) SweepArgs {
    // Population buffers, tile-major, of the storage type S the launcher was
    // instantiated with (float, double, __half or __nv_bfloat16).
    const void *src;       // populations of the previous step
    void *dst;             // populations written by this step
    void *aux;             // init only: the other buffer, whose f planes are also
                           // set to w_i (they are never rewritten when flow is off)
    int nx, ny;            // lattice size
    int ntx;               // number of column tiles
    int parity;            // index of the source buffer (selects the rounding seed word
                           // and the direction of the sweep over the row bands)
    int rows;              // rows per block (each thread walks them)
    int prefetch;          // > 0: each block asks L2 for the tile rows `prefetch`
                           // rows ahead of its own in the sweep's direction
                           // (one bulk prefetch per row)
    real k0, k1, k2;       // g rates (Eq. 2)
    real k0f, k1f, k2f;    // f rates
    real Lh, gbeta;        // latent heat, g*beta
    real inv_Lh;           // 1 / Lh
    // combinations of the rates in the working precision, for the collisions:
    // k1 - k0, k2 - k0, k1f - k0f, k2f - k0f, 1 - k0, 1 - k0f, 1 - k1f/2, 1 - k2f/2
    real d1, d2, e1, e2, a0, a0f, s1, s2;
    int unit;              // k0 = 1, and k0f = 1 with flow: a0 = a0f = 0
    int strip_on;          // cavity: 1 if the heated segment is non-empty
    int lo2, hi2;          // cavity: crossing heated iff lo2 <= 2x + 1 - c_ix <= hi2
    // heated-wall inflow reduction (every sweep)
    double *qpart;         // one partial per wall-adjacent block
    unsigned *qcount;      // ticket counter, reset to 0 by the last block
    int nq;                // number of wall-adjacent blocks
    // diagnostics (kSweepDiag, init): 4 partials per block, folded into the
    // record by a fold kernel launched right after on the same stream
    double *dpart;
    double *dpart2;        // fold kernel: 4 partials per fold block
    unsigned *dticket;     // fold kernel: ticket counter, reset by its last block
    DevRecord *rec;
    // optional history ring (lbm_set_history): entry k = 4 doubles {step, Q,
    // melt fraction, unused} for step k mod hist_cap; NULL = off
    double *hist;
    long long hist_cap;
    long long step;        // step index the launch produces (host bookkeeping only;
                           // the record takes its step from rec->counter)
    // staged sweep (16-bit storage): 1 = launch staged_kernel over the band
    // grid; its mbarrier waits give up after wait_limit + 1 tries, and
    // force_timeout = 1 makes each block first wait on a barrier that nothing
    // completes (tests of the timeout path)
    int staged;
    int force_timeout;
    long long wait_limit;
    // field outputs (kFields), nx*ny doubles each, row-major; NULL = skip
    double *oH, *oT, *oFL, *oUX, *oUY, *oRHO;
    int sms;  // SMs of the device (share_smem; the host's)
};

// Several steps of a small lattice in one launch (tile.cuh): T steps by blocks
// that own cores of W x H cells each.
constexpr int kTileThreads = 768;     // block size limit, FP32 arithmetic (80 registers)
constexpr int kTileThreads64 = 256;   // FP64 (its pipe is busy with four warps; no spills)
constexpr int kTileMaxSteps = 16;
constexpr int kTileMaxNx = 4096;      // the inflow's fold: 32 lanes x 128 columns
constexpr size_t kTileSmemMax = 230400;
// Dynamic shared memory with which an SM holds its even share of a launch's blocks and
// no more; 0 where that is more than `most` (7 at most).  For FP64: two blocks on one SM
// take twice as long, and with programmatic launches a launch's blocks find the previous
// ones still resident and gather on what is free.
inline unsigned share_smem(long long blocks, int sms, int most) {
    const long long share = (blocks + sms - 1) / sms;
    return share <= most ? (unsigned)(kTileSmemMax / (share + 1) + 1024) / 16 * 16 : 0u;
}
struct TileArgs {
    int T;                 // steps of this launch, 1 .. kTileMaxSteps
    int W, H;              // core of a block; W a multiple of 32 in the cavity
    int tiles_x, tiles_y;  // cores in the lattice (Stefan: tiles_y = 1, H = ny <= 32)
    int pitch;             // shared-memory cells per row: W + 2 T
    int threads;           // block size
    unsigned smem;         // dynamic shared memory: the slots, then at q_offset T x 3 x (W, or
    unsigned q_offset;     // H in the Stefan problem) inflow terms in the working precision
    double *qgroup;        // device scratch: T x (heated groups of 32 wall cells)
};

// Two steps of a large cavity per pass over memory (band.cuh): one block per
// strip of columns and band of rows.
constexpr int kBandThreads = 128;  // block size limit; two columns a thread
constexpr int kBandWarps = 12;     // per SM: up to 168 registers a thread, no spills
constexpr int kBandMaxStrips = 2048;
constexpr size_t kBandSmemMax = 4 * 6 * 2 * kBandThreads * 2 * sizeof(float);  // band_args
struct BandArgs {
    int strips, bands;
    int threads;     // one per two columns of the widest strip and its halo pairs
    unsigned smem;
    double *qgroup;  // device scratch: 2 x strips
};

// Launchers, instantiated in sweep_fp32.cu / sweep_fp64.cu / sweep_f16.cu /
// sweep_bf16.cu for (compute real, storage codec S) = (float, float),
// (double, double), (float, F16<SR>), (float, BF16<SR>), SR = round to
// nearest (false) or stochastically (true).
template <bool SR>
struct F16;
template <bool SR>
struct BF16;
// pdl: launch the sweep with programmatic stream serialization, so that it
// is scheduled while the previous kernel of the stream drains (the kernel
// waits for that kernel's completion before it touches memory).
template <typename real, typename S>
cudaError_t launch_lattice(const SweepArgs<real> &a, int problem, bool flow, int mode,
                           dim3 grid, dim3 block, cudaStream_t s, bool pdl, int streaming = kPull);
template <typename S>
cudaError_t launch_band(const SweepArgs<float> &a, const BandArgs &b, cudaStream_t s);
// The same for every lattice of a batch (cavities with flow): tl / b hold what the
// lattices share, the entries their tiles, or strips and bands; mstarts[r] is entry
// r's first block of nblocks; j: the launch's number in its call, which selects the
// buffers (parity[r] ^ (j & 1)) as for a batch's sweeps.
template <typename S>
cudaError_t launch_batch_tile(const void *entries, const int *mstarts, const int *parity, int n, int nblocks, int j,
                              const TileArgs &tl, cudaStream_t s);
template <typename S>
cudaError_t launch_batch_band(const void *entries, const int *mstarts, const int *parity, int n, int nblocks, int j,
                              const BandArgs &b, cudaStream_t s);
template <typename real, typename S>
cudaError_t launch_tile(const SweepArgs<real> &a, const TileArgs &tl, int problem, bool flow, cudaStream_t s);
template <typename real, typename S>
cudaError_t launch_init(const SweepArgs<real> &a, double amp, uint64_t seed, dim3 grid,
                        dim3 block, cudaStream_t s);
template <typename real, typename S>
cudaError_t launch_fields0(const SweepArgs<real> &a, bool flow, dim3 grid, dim3 block,
                           cudaStream_t s);
// One lattice of a batch launch: its arguments for both buffer parities and
// its place in the launch's block numbering.
template <typename real>
struct BatchEntry {
    SweepArgs<real> a[2];  // [p]: source buffer p, destination buffer 1 - p
    int start;             // first block of this lattice in the launch
    int gx, gy;            // tile columns and row bands
    int mx, my;            // several steps per launch: tiles, or strips and bands,
    int mstart;            // their first block,
    double *qgroup;        // and the inflow's scratch
};

// One step of a batch: `entries` points at n device BatchEntry<real> records
// whose blocks, nblocks in all, run in one launch; starts[r] is entry r's first
// block (the entries' start fields, as a compact array for the block search);
// parity[r] is entry r's source buffer at step j = 0; uniform > 0 when every
// entry has that many blocks (0 otherwise); interleave (uniform batches only):
// block b belongs to entry b mod n instead of b / uniform.  diag: diagnostic
// sweep plus the per-entry fold.  streaming: kPull (buffer parity[r] ^ (j & 1)
// into the other), or the push (even j) / local (odd j) sweep of one-buffer
// streaming in buffer parity[r].
template <typename real, typename S>
cudaError_t launch_batch(const void *entries, const int *starts, const int *parity, int n,
                         int uniform, int interleave, int nblocks, int problem, bool flow, bool diag,
                         int j, cudaStream_t s, bool pdl, int streaming = kPull);
// Tile-major buffer <-> plane-major FP64 staging (18 planes of nx*ny, f then g).
// to_staging = true packs buf into stage; false unpacks stage into buf (and,
// if buf2 is non-NULL, the f planes into buf2 as well).  Values in the staging
// are the populations themselves, whatever the storage encoding.
template <typename S>
cudaError_t launch_repack(void *buf, void *buf2, double *stage, int nx, int ny, bool to_staging,
                          cudaStream_t s);

}  // namespace btrirt
