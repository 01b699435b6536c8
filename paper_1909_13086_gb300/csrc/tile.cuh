// tile.cuh -- several time steps of a small lattice per launch (device code).
//
// A step of a small lattice costs far less than a launch: on GB300 the sweep of
// a 256 x 128 cavity takes 5.5 us however little it computes (launch, two trips
// to L2, drain).  Here a block owns a core of W x H cells and advances it T steps
// in one launch: it pulls the first step from the source buffer on the core plus
// a halo of T - 1 cells, keeps the populations in shared memory, and after step
// t computes only what the remaining steps still need (halo T - t), so the last
// step is the core alone, which goes to the destination buffer.  No block waits
// for another one.  Halo cells are computed by every block that needs them, from
// the same values in the same order, so every block gets the same bits, and they
// are those of T sweeps.
//
// In shared memory the steps run in place by the AA pattern (lbm_internal.h):
// odd steps pull and push, even steps take and leave a cell's own slots; each
// cell reads and writes the same nine slots, so one barrier per step suffices.
// A cell's nine slots lie next to each other (f_i and g_i together in one): the
// strides of 9 x 4, 8 or 16 bytes from lane to lane meet no bank twice, and all
// nine are one base plus immediate offsets.
//
// On GB300, us per step, sweeps and tiles: 64 x 32 FP32 4.9 and 1.4, 256 x 128 FP32 5.4
// and 1.6, BF16-SR 7.8 and 1.8, 512 x 512 FP32 7.1 and 4.6, 1024 x 4 Stefan FP64 8.6 and
// 2.9.  Bound by latency: 4.2 us a launch, then per step one cell's chain and the
// barrier (256 x 128: 43 % issue active).  Two cells per thread, as in the sweeps, has
// half the warps and is slower (512 x 512 5.4).  FP64 is bound by its pipe: an SM holds
// its share of the tiles and no more (tile_args).
#pragma once

#include "sweep.cuh"

namespace btrirt {

__device__ __forceinline__ float stored_value(float v) { return v; }
__device__ __forceinline__ double stored_value(double v) { return v; }
__device__ __forceinline__ float stored_value(__half v) { return __half2float(v); }
__device__ __forceinline__ float stored_value(__nv_bfloat16 v) { return __bfloat162float(v); }

// What a shared-memory slot holds: f_i and g_i as stored (16-bit: their word),
// or g_i alone without flow.
template <typename S, bool FLOW>
struct Slot;
template <>
struct Slot<float, true> {
    using T = float2;
    __device__ static void get(T v, float &f, float &g) { f = v.x, g = v.y; }
    __device__ static T make(float f, float g) { return make_float2(f, g); }
};
template <>
struct Slot<double, true> {
    using T = double2;
    __device__ static void get(T v, double &f, double &g) { f = v.x, g = v.y; }
    __device__ static T make(double f, double g) { return make_double2(f, g); }
};
template <typename S>
struct Slot<S, true> {
    using T = uint32_t;
    __device__ static void get(T v, float &f, float &g) { f = Store<S>::lo(v), g = Store<S>::hi(v); }
};
template <typename S>
struct Slot<S, false> {
    using T = typename Store<S>::elem;
    template <typename real>
    __device__ static void get(T v, real &, real &g) { g = stored_value(v); }
};

// The walls a cell touches.
struct Walls {
    bool left = false, right = false, bottom = false, top = false;
    // the neighbour against c_i lies beyond a wall
    __device__ __forceinline__ bool from_wall(int i) const {
        const int cx = cx_of(i), cy = cy_of(i);
        return (cx > 0 && left) || (cx < 0 && right) || (cy > 0 && bottom) || (cy < 0 && top);
    }
};
// A cell's slots in shared memory, and those of the rows below and above.
template <typename T>
struct TileCell : Walls {
    T *s, *sm, *sp;
    __device__ __forceinline__ T *at(int dx, int dy) const { return (dy < 0 ? sm : (dy > 0 ? sp : s)) + 9 * dx; }
};

// The first step's pull from the source buffer, b at the cell's element of plane
// 0, bL / bR as in pull_fast, below / above: elements to the rows y - 1 / y + 1.
// Directions from beyond a wall take the cell's own opposite population.
template <typename real, typename S, bool FLOW>
__device__ __forceinline__ void pull_first(const typename Store<S>::elem *b, const typename Store<S>::elem *bL,
                                           const typename Store<S>::elem *bR, const Walls &n,
                                           long long below, long long above, real f[9], real g[9]) {
#pragma unroll
    for (int i = 0; i < 9; ++i) {
        const int cx = cx_of(i), cy = cy_of(i);
        const typename Store<S>::elem *from = (cx > 0 ? bL : (cx < 0 ? bR : b)) - cx * col_step<S>() +
                                              (cy > 0 ? below : (cy < 0 ? above : 0));
        const bool wall = n.from_wall(i);
        real fv = real(0), gv;
        load_own<real, S, FLOW>(wall ? b : from, wall ? opp_of(i) : i, fv, gv);
        if (FLOW) f[i] = fv;
        g[i] = gv;
    }
}

// Rounds and packs the nine (f_i, g_i) of a cell to what is stored, in the order
// of finish_cell (the rounding stream of the cell and step), and hands each to
// put(i, value).
template <typename real, typename S, bool FLOW, typename Put>
__device__ __forceinline__ void emit_slots(const SweepArgs<real> &a, int x, int y, const Macro<real> &m,
                                           const real f[9], const real g[9], uint32_t step_seed, Put &&put) {
    if constexpr (!Store<S>::kDev) {
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            if constexpr (FLOW) put(i, Slot<S, FLOW>::make(f[i], g[i]));
            else put(i, g[i]);
        }
    } else if (!Store<S>::kSR || (!FLOW && !isfinite(m.H))) {
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            if constexpr (FLOW) {
                put(i, Store<S>::pack_rn(g[i], f[i]));
            } else {
                typename Store<S>::elem v;
                Store<S>::str_rn(&v, g[i]);
                put(i, v);
            }
        }
    } else {
        uint32_t rs = hash32(step_seed ^ (uint32_t)((long long)y * a.nx + x));
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            if constexpr (FLOW) {
                put(i, Store<S>::pack_sr(g[i], f[i], lcg_next32(rs)));
            } else {
                typename Store<S>::elem v;
                Store<S>::strs(&v, g[i], lcg_next(rs));
                put(i, v);
            }
        }
    }
}

// A value as the slots hold it into the tile-major buffer (d: the cell's element
// of plane 0).
template <typename S, bool FLOW, typename T>
__device__ __forceinline__ void put_global(typename Store<S>::elem *d, int i, T v) {
    if constexpr (Store<S>::kDev) {
        if constexpr (FLOW) reinterpret_cast<uint32_t *>(d)[i * kTW] = v;
        else d[2 * i * kTW + 1] = v;
    } else if constexpr (FLOW) {
        d[i * kTW] = v.x;
        d[(9 + i) * kTW] = v.y;
    } else {
        d[(9 + i) * kTW] = v;
    }
}

// One thread, the last of a launch that took `steps` steps: their inflows into
// the record and the history, as a sweep's last heated block does.
template <typename real>
__device__ __forceinline__ void put_inflow(const SweepArgs<real> &a, const double *inflow, int steps) {
    double cum = a.rec->Q_cum;
    for (int t = 0; t < steps; ++t) cum += inflow[t];
    a.rec->Q_cum = cum;
    a.rec->Q_last = inflow[steps - 1];
    *a.qcount = 0u;
    if (!a.hist) return;
    const long long done = (long long)__ldcg(&a.rec->counter);
    for (int t = 0; t < steps; ++t) {
        const long long st = done - steps + 1 + t;
        double *e = a.hist + 4 * (st % a.hist_cap);
        e[0] = (double)st;
        e[1] = inflow[t];
        e[2] = __longlong_as_double(0x7ff8000000000000ll);
    }
}

// The block's work: tile (tx, ty) of the lattice described by a, advanced tl.T
// steps.  sm: shared memory of tile_smem_bytes.
//   The heated-wall inflow of each step: core cells on the heated wall leave
// their directions' terms in shared memory; after the last step each warp sums one step's 32
// columns at a time (the groups a sweep's warps sum, in the same order), and
// the last heated block folds the groups of all steps as the sweep's blocks and
// its fold do, so that the flux is bitwise the sweep's in FP64 as well.
template <typename real, typename S, int PROB, bool FLOW>
__device__ __forceinline__ void tile_block(const SweepArgs<real> &a, const TileArgs &tl, const int tx,
                                           const int ty, unsigned char *sm) {
    using SL = Slot<S, FLOW>;
    using T = typename SL::T;
    using E = typename Store<S>::elem;
    const E *const src = static_cast<const E *>(a.src);
    E *const dst = static_cast<E *>(a.dst);
    const int nthr = blockDim.x, steps = tl.T;
    const int x0 = tx * tl.W, x1 = min(x0 + tl.W, a.nx);
    const int y0 = ty * tl.H, y1 = min(y0 + tl.H, a.ny);
    // shared-memory origin: the first step's region and the ring its pushes reach
    const int gx = x0 - steps, gy = PROB == kStefan ? 0 : y0 - steps;
    T *const slots = reinterpret_cast<T *>(sm);
    real *const qs = reinterpret_cast<real *>(sm + tl.q_offset);  // [step][direction][wall cell]
    const bool heated = PROB == kCavity ? (a.strip_on && ty == 0) : tx == 0;
    const int qw = PROB == kCavity ? tl.W : tl.H;  // wall cells of a core

    if (tx == 0 && ty == 0 && threadIdx.x == 0) a.rec->counter += (unsigned long long)steps;
    unsigned long long seed = 0;
    if (Store<S>::kSR) {
        seed = a.rec->rng[a.parity];
        if (tx == 0 && ty == 0 && threadIdx.x == 0) a.rec->rng[a.parity ^ 1] = seed + (unsigned long long)steps;
    }
    for (int t = 1; t <= steps; ++t) {
        const int h = steps - t;
        const int xa = max(0, x0 - h), wr = min(a.nx, x1 + h) - xa;
        const int ya = PROB == kStefan ? 0 : max(0, y0 - h);
        const int hr = PROB == kStefan ? a.ny : min(a.ny, y1 + h) - ya;
        const unsigned inv = ((1u << 20) + wr - 1) / (unsigned)wr;  // c / wr = c inv >> 20 (c wr < 2^20)
        const uint32_t step_seed = Store<S>::kSR ? hash32((uint32_t)(seed + (t - 1)) ^ 0x5bd1e995u) : 0u;
        const bool push = t & 1;
        for (int c = threadIdx.x; c < wr * hr; c += nthr) {
            const int ry = (int)(((unsigned)c * inv) >> 20), rx = c - ry * wr;
            const int x = xa + rx, y = ya + ry;
            TileCell<T> n;
            n.s = slots + 9 * ((y - gy) * tl.pitch + (x - gx));
            n.sm = n.s - 9 * tl.pitch;
            n.sp = n.s + 9 * tl.pitch;
            n.left = x == 0;
            n.right = x == a.nx - 1;
            n.bottom = PROB == kCavity && y == 0;
            n.top = PROB == kCavity && y == a.ny - 1;
            if (PROB == kStefan) {  // periodic: the first and last rows are neighbours
                if (y == 0) n.sm = n.s + 9 * (a.ny - 1) * tl.pitch;
                if (y == a.ny - 1) n.sp = n.s - 9 * (a.ny - 1) * tl.pitch;
            }
            // warps with an edge cell select per direction; the others take fixed offsets
            const bool edge = __any_sync(__activemask(), n.left || n.right || n.bottom || n.top);
            real f[9], g[9];
            if (t == 1) {
                constexpr int cs = col_step<S>();
                const int lx = x % kTW;
                const long long i0 = cell_index<S>(x, y, 0, a.ny);
                const long long iL = lx == 0 && x > 0 ? cell_index<S>(x - 1, y, 0, a.ny) + cs : i0;
                const long long iR = lx == kTW - 1 && !n.right ? cell_index<S>(x + 1, y, 0, a.ny) - cs : i0;
                if (!edge && PROB == kCavity) {
                    pull_fast<real, S, FLOW>(src + i0, src + iL, src + iR, f, g);
                } else {
                    const long long below = PROB == kStefan && y == 0 ? (long long)(a.ny - 1) * kRS : -kRS;
                    const long long above = PROB == kStefan && y == a.ny - 1 ? -(long long)(a.ny - 1) * kRS : kRS;
                    pull_first<real, S, FLOW>(src + i0, src + iL, src + iR, n, below, above, f, g);
                }
            } else if (!push) {
#pragma unroll
                for (int i = 0; i < 9; ++i) SL::get(n.s[opp_of(i)], f[i], g[i]);
            } else if (!edge) {
#pragma unroll
                for (int i = 0; i < 9; ++i) SL::get(n.at(-cx_of(i), -cy_of(i))[i], f[i], g[i]);
            } else {
#pragma unroll
                for (int i = 0; i < 9; ++i) {
                    const T *p = n.at(-cx_of(i), -cy_of(i)) + i;
                    if (n.from_wall(i)) p = n.s + opp_of(i);
                    SL::get(*p, f[i], g[i]);
                }
            }
            if (PROB == kCavity ? n.bottom : n.left) {
                real q[3];
                hot_wall<real, S, PROB>(a, x, g, q);
                if (heated && (PROB == kStefan || (x >= x0 && x < x1))) {
#pragma unroll
                    for (int k = 0; k < 3; ++k) qs[((t - 1) * 3 + k) * qw + (PROB == kCavity ? x - x0 : y)] = q[k];
                }
            }
            const Macro<real> m = cell_update<real, S, FLOW, true>(a, f, g);
            if (t == steps) {
                E *const d = dst + cell_index<S>(x, y, 0, a.ny);
                emit_slots<real, S, FLOW>(a, x, y, m, f, g, step_seed,
                                          [&](int i, T v) { put_global<S, FLOW>(d, i, v); });
            } else if (!push) {
                emit_slots<real, S, FLOW>(a, x, y, m, f, g, step_seed, [&](int i, T v) { n.s[i] = v; });
            } else if (!edge) {
                emit_slots<real, S, FLOW>(a, x, y, m, f, g, step_seed,
                                          [&](int i, T v) { n.at(cx_of(i), cy_of(i))[opp_of(i)] = v; });
            } else {
                emit_slots<real, S, FLOW>(a, x, y, m, f, g, step_seed, [&](int i, T v) {
                    T *p = n.at(cx_of(i), cy_of(i)) + opp_of(i);
                    if (n.from_wall(opp_of(i))) p = n.s + i;
                    *p = v;
                });
            }
        }
        __syncthreads();
    }
    if (!heated) return;

    // ---- heated-wall inflow of the steps
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = nthr >> 5;
    const int groups = PROB == kCavity ? tl.W / 32 : 1;        // groups of 32 wall cells in this core
    const int all = PROB == kCavity ? tl.tiles_x * groups : 1;  // in the lattice
    const int mine = PROB == kCavity ? x1 - x0 : a.ny;
    for (int k = warp; k < steps * groups; k += nwarps) {
        const int t = k / groups, gr = k - t * groups, w = 32 * gr + lane;
        double v = 0.0;
        if (w < mine) {
#pragma unroll
            for (int j = 0; j < 3; ++j) v += (double)qs[(t * 3 + j) * qw + w];
        }
        v = warp_sum(v);
        if (lane == 0) __stcg(tl.qgroup + t * all + tx * groups + gr, v);
    }
    __shared__ bool last;
    __shared__ double inflow[kTileMaxSteps];
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        const unsigned blocks = PROB == kCavity ? tl.tiles_x : 1;
        last = atomicAdd(a.qcount, 1u) == blocks - 1u;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    for (int t = warp; t < steps; t += nwarps) {
        double v = 0.0;  // lane: the four groups of one of a sweep's blocks (128 columns)
        if (PROB == kCavity) {
            double u[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const int gr = 4 * lane + k;
                u[k] = gr < all ? __ldcg(tl.qgroup + t * all + gr) : 0.0;
            }
            v = (u[0] + u[2]) + (u[1] + u[3]);
        } else if (lane == 0) {
            v = __ldcg(tl.qgroup + t);
        }
        v = warp_sum(v);
        if (lane == 0) inflow[t] = v;
    }
    __syncthreads();
    if (threadIdx.x == 0) put_inflow(a, inflow, steps);
}

template <typename real, typename S, int PROB, bool FLOW>
__global__ void __launch_bounds__(sizeof(real) == 8 ? kTileThreads64 : kTileThreads)
    tile_kernel(const SweepArgs<real> a, const TileArgs tl) {
    extern __shared__ __align__(16) unsigned char tile_sm[];
    pdl_launch_dependents();
    pdl_wait();  // the previous launch's populations, tickets and record
    tile_block<real, S, PROB, FLOW>(a, tl, blockIdx.x, blockIdx.y, tile_sm);
}

// A launch with dynamic shared memory and programmatic serialization.
template <typename... KArgs, typename... Args>
static cudaError_t launch_shared(void (*kernel)(KArgs...), dim3 grid, dim3 block, unsigned smem, cudaStream_t s,
                                 Args &&...args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, std::forward<Args>(args)...);
}

// The entry of a batch that this block belongs to (number r), copied into shared
// memory (sh, of sizeof(BatchEntry<float>)); the table is written only by copies the host
// orders before the batch's launches, so this may precede pdl_wait.
__device__ __forceinline__ const BatchEntry<float> &batch_entry(const BatchEntry<float> *entries, const int *mstarts,
                                                                int n, unsigned char *sh, int &r) {
    __shared__ int found;
    if (threadIdx.x == 0) found = batch_find(mstarts, n, blockIdx.x);
    __syncthreads();
    r = found;
    const int4 *s4 = reinterpret_cast<const int4 *>(entries + r);
    for (unsigned k = threadIdx.x; k < sizeof(BatchEntry<float>) / 16; k += blockDim.x)
        reinterpret_cast<int4 *>(sh)[k] = __ldg(s4 + k);
    __syncthreads();
    return *reinterpret_cast<const BatchEntry<float> *>(sh);
}

template <typename S>
__global__ void __launch_bounds__(kTileThreads)
    batch_tile_kernel(const BatchEntry<float> *entries, const int *mstarts, const int *parity, int n, int j,
                      const TileArgs common) {
    extern __shared__ __align__(16) unsigned char tile_sm[];
    __shared__ __align__(16) unsigned char entry_sh[sizeof(BatchEntry<float>)];
    pdl_launch_dependents();
    int r;
    const BatchEntry<float> &e = batch_entry(entries, mstarts, n, entry_sh, r);
    const int l = (int)blockIdx.x - e.mstart;
    TileArgs tl = common;
    tl.tiles_x = e.mx;
    tl.tiles_y = e.my;
    tl.qgroup = e.qgroup;
    const int p = __ldg(parity + r) ^ (j & 1);
    pdl_wait();
    tile_block<float, S, kCavity, true>(e.a[p], tl, l % tl.tiles_x, l / tl.tiles_x, tile_sm);
}

template <typename S>
cudaError_t launch_batch_tile(const void *entries, const int *mstarts, const int *parity, int n, int nblocks, int j,
                              const TileArgs &tl, cudaStream_t s) {
    cudaError_t e = cudaFuncSetAttribute(batch_tile_kernel<S>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)kTileSmemMax);
    if (e != cudaSuccess) return e;
    return launch_shared(batch_tile_kernel<S>, dim3(nblocks), dim3(tl.threads), tl.smem, s,
                         static_cast<const BatchEntry<float> *>(entries), mstarts, parity, n, j, tl);
}

template <typename real, typename S, int PROB, bool FLOW>
static cudaError_t launch_tile_k(const SweepArgs<real> &a, const TileArgs &tl, cudaStream_t s) {
    auto *kernel = tile_kernel<real, S, PROB, FLOW>;
    // per device and idempotent; no state is kept here
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kTileSmemMax);
    if (e != cudaSuccess) return e;
    return launch_shared(kernel, dim3(tl.tiles_x, tl.tiles_y), dim3(tl.threads), tl.smem, s, a, tl);
}

template <typename real, typename S>
cudaError_t launch_tile(const SweepArgs<real> &a, const TileArgs &tl, int problem, bool flow, cudaStream_t s) {
    if (problem == kCavity)
        return flow ? launch_tile_k<real, S, kCavity, true>(a, tl, s) : launch_tile_k<real, S, kCavity, false>(a, tl, s);
    return flow ? launch_tile_k<real, S, kStefan, true>(a, tl, s) : launch_tile_k<real, S, kStefan, false>(a, tl, s);
}

#define BTRIRT_INSTANTIATE_BATCH_TILE(S)                                                                         \
    template cudaError_t launch_batch_tile<S>(const void *, const int *, const int *, int, int, int,           \
                                              const TileArgs &, cudaStream_t);
#define BTRIRT_INSTANTIATE_TILE(REAL, S) \
    template cudaError_t launch_tile<REAL, S>(const SweepArgs<REAL> &, const TileArgs &, int, bool, cudaStream_t);

}  // namespace btrirt
