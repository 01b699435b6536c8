// band.cuh -- two time steps of a large cavity per pass over memory (device
// code; FP32 arithmetic, with flow).
//
// A sweep reads and writes every population once per step: 144 bytes a cell in
// FP32, and a lattice beyond L2 waits for them.  Here a block marches over a band
// of rows of a strip of columns and takes two steps on the way: at each row it
// pulls, collides and keeps step 1 of that row, then does step 2 of the row
// before, whose three rows of step 1 are now complete, and only that goes to
// memory.  Populations are read and written once per two steps, and half as many
// launches remain.
//
// A thread has two neighbouring columns: all of the collision runs packed (one
// issue slot for both cells), and addresses, uniform terms and loop overhead are
// paid once for two.  Step 1 of a row goes to the other columns through a ring of
// four rows in shared memory (the six directions with c_x != 0; a row is written
// while the three before it may still be read, so one barrier a row suffices); a
// thread keeps its columns' directions 0, 2 and 4 in registers.  Step 1 is
// computed on a pair of columns and a row more than the core on every side that is
// not a wall, by the same operations as in the neighbouring block, so the bits are
// those of two sweeps.  The bands of one lattice run at the same time, one wave of
// blocks (of a large batch in several); successive launches march them in opposite directions, so that each
// starts on the rows the previous one wrote last.
//
// 2048 x 1024 FP32 on GB300: 36.7 us per step with one-buffer sweeps, 26.3 here: 137
// MB of DRAM traffic per step (161 before) at 5.2 TB/s, 0.77 of the copy bandwidth.
// What is left is latency: the loads of the next row wait in registers through step 2
// of the row before, which leaves 12 warps per SM.  Without them 16 warps fit, and it
// takes 36.6 us: the larger rings leave too little L1 for the lines that a pair's two
// halves share.
#pragma once

#include "tile.cuh"

namespace btrirt {

__host__ __device__ constexpr int ring_dir(int i) { return i == 1 ? 0 : (i == 3 ? 1 : i - 3); }

template <typename S>
__device__ __forceinline__ void band_block(const SweepArgs<float> &a, const BandArgs &b, const int strip,
                                           const int band, unsigned char *sm) {
    using P = Two<S>;
    using T = typename P::T;
    using E = typename Store<S>::elem;
    const E *const src = static_cast<const E *>(a.src);
    E *const dst = static_cast<E *>(a.dst);
    // cores start on even columns, so that a pair never spans two tiles
    const int pairs = (a.nx + 1) / 2;
    const int xs = 2 * (int)((long long)strip * pairs / b.strips);
    const int xe = min(a.nx, 2 * (int)((long long)(strip + 1) * pairs / b.strips));
    const int ya = (int)((long long)band * a.ny / b.bands), yb = (int)((long long)(band + 1) * a.ny / b.bands);
    const int r0 = max(0, ya - 1), r1 = min(a.ny, yb + 1), rows = r1 - r0;
    const bool up = a.parity == 0;
    const int c = 2 * (int)threadIdx.x, x = max(0, xs - 2) + c;
    const bool active = x < min(a.nx, xe + 2), core = x >= xs && x < xe;
    const bool heated = a.strip_on && ya == 0;

    if (strip == 0 && band == 0 && threadIdx.x == 0) a.rec->counter += 2ull;
    uint32_t seed1 = 0, seed2 = 0;
    if (Store<S>::kSR) {
        const unsigned long long sd = a.rec->rng[a.parity];
        if (strip == 0 && band == 0 && threadIdx.x == 0) a.rec->rng[a.parity ^ 1] = sd + 2ull;
        seed1 = hash32((uint32_t)sd ^ 0x5bd1e995u);
        seed2 = hash32((uint32_t)(sd + 1ull) ^ 0x5bd1e995u);
    }
    const int step = up ? kRS : -kRS, yfirst = up ? r0 : r1 - 1;
    const PairPlace<S> at(x, a.nx, a.ny);
    long long i0 = cell_index<S>(min(x, a.nx - 1), yfirst, 0, a.ny);  // the pair's element of the row in hand

    const int plane = 2 * (int)blockDim.x, ring_row = 6 * P::kPlanes * plane;  // words
    uint32_t *const ring = reinterpret_cast<uint32_t *>(sm);
    T c0{}, c2{}, c4{}, old{};  // step 1 of the row before: directions 0, 2, 4; of the one before that: 2 (up) or 4
    double q1 = 0.0, q2 = 0.0;
    T raw[9];
    auto load = [&](int y) {
        if (active) at.pull(src + i0, y == 0, y == a.ny - 1, raw);
    };
    load(yfirst);
    const int last = (up ? yb == a.ny : ya == 0) ? rows : rows - 1;  // at a wall its row has no row after it
    for (int k = 0; k <= last; ++k) {
        const int y = up ? r0 + k : r1 - 1 - k;
        uint32_t *const rn = ring + (k & 3) * ring_row;
        T v0{}, v2{}, v4{};
        if (k < rows) {
            if (active) {
                float2 f[9], g[9];
#pragma unroll
                for (int i = 0; i < 9; ++i) P::get(raw[i], f[i], g[i]);
                if (y == 0) q1 += hot_wall_two<S>(a, x, xs, xe, g);
                cell_update_two<S>(a, f, g);
                emit_two<S>(a, x, y, f, g, seed1, [&](int i, const T &v) {
                    if (i == 0) v0 = v;
                    else if (i == 2) v2 = v;
                    else if (i == 4) v4 = v;
                    else P::put(rn + ring_dir(i) * P::kPlanes * plane, c, plane, v);
                });
            }
        }
        const long long irow = i0 - step;  // the row before
        i0 += step;
        if (k + 1 < rows) load(up ? y + 1 : y - 1);  // in flight during step 2 of the row before
        __syncthreads();
        const int r = up ? y - 1 : y + 1;
        if (core && r >= ya && r < yb) {
            const bool bottom = r == 0, top = r == a.ny - 1;
            const uint32_t *const rc = ring + ((k - 1) & 3) * ring_row, *const ro = ring + ((k - 2) & 3) * ring_row;
            const uint32_t *const lo = up ? ro : rn, *const hi = up ? rn : ro;
            float2 f[9], g[9];
            P::get(c0, f[0], g[0]);
            P::get(bottom ? c4 : (up ? old : v2), f[2], g[2]);
            P::get(top ? c2 : (up ? v4 : old), f[4], g[4]);
            const bool edge = at.side || bottom || top;
#pragma unroll
            for (int i = 1; i < 9; ++i) {
                if (i == 2 || i == 4) continue;
                const int cx = cx_of(i), cy = cy_of(i), d = ring_dir(i) * P::kPlanes * plane;
                const int o = ring_dir(opp_of(i)) * P::kPlanes * plane;
                const uint32_t *const p = (cy > 0 ? lo : (cy < 0 ? hi : rc)) + d;
                T v;
                if (edge) {
                    const bool w0 = at.wall0(i, bottom, top), w1 = at.wall1(i, bottom, top);
                    v = P::take(w0 ? rc + o : p, w0 ? c : c - cx, w1 ? rc + o : p, w1 ? c + 1 : c + 1 - cx, plane);
                } else {
                    v = P::take(p, c - cx, p, c + 1 - cx, plane);
                }
                P::get(v, f[i], g[i]);
            }
            if (bottom) q2 += hot_wall_two<S>(a, x, xs, xe, g);
            cell_update_two<S>(a, f, g);
            E *const d = dst + irow;
            emit_two<S>(a, x, r, f, g, seed2, [&](int i, const T &v) { at.put_own(d, i, v); });
        }
        old = up ? c2 : c4;
        c0 = v0;
        c2 = v2;
        c4 = v4;
    }
    if (!heated) return;

    // ---- heated-wall inflow of both steps (FP64 sums of FP32 terms)
    __shared__ double part[2][kBandThreads / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    q1 = warp_sum(q1);
    q2 = warp_sum(q2);
    if (lane == 0) {
        part[0][warp] = q1;
        part[1][warp] = q2;
    }
    __syncthreads();
    if (threadIdx.x < 2) {
        double s = 0.0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) s += part[threadIdx.x][w];
        __stcg(b.qgroup + threadIdx.x * b.strips + strip, s);
    }
    __shared__ bool fold;
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        fold = atomicAdd(a.qcount, 1u) == (unsigned)b.strips - 1u;
    }
    __syncthreads();
    if (!fold) return;
    __threadfence();
    if (threadIdx.x < 32) {
        double s[2] = {0.0, 0.0};
        for (int w = lane; w < b.strips; w += 32) {
            s[0] += __ldcg(b.qgroup + w);
            s[1] += __ldcg(b.qgroup + b.strips + w);
        }
        s[0] = warp_sum(s[0]);
        s[1] = warp_sum(s[1]);
        if (lane == 0) put_inflow(a, s, 2);
    }
}

template <typename S>
__global__ void __launch_bounds__(kBandThreads, kBandWarps / (kBandThreads / 32))
    band_kernel(const SweepArgs<float> a, const BandArgs b) {
    extern __shared__ __align__(16) unsigned char band_sm[];
    pdl_launch_dependents();
    pdl_wait();  // the previous launch's populations, tickets and record
    band_block<S>(a, b, blockIdx.x, blockIdx.y, band_sm);
}

template <typename S>
cudaError_t launch_band(const SweepArgs<float> &a, const BandArgs &b, cudaStream_t s) {
    cudaError_t e = cudaFuncSetAttribute(band_kernel<S>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)kBandSmemMax);
    if (e != cudaSuccess) return e;
    return launch_shared(band_kernel<S>, dim3(b.strips, b.bands), dim3(b.threads), b.smem, s, a, b);
}

template <typename S>
__global__ void __launch_bounds__(kBandThreads, kBandWarps / (kBandThreads / 32))
    batch_band_kernel(const BatchEntry<float> *entries, const int *mstarts, const int *parity, int n, int j,
                      const BandArgs common) {
    extern __shared__ __align__(16) unsigned char band_sm[];
    __shared__ __align__(16) unsigned char entry_sh[sizeof(BatchEntry<float>)];
    pdl_launch_dependents();
    int r;
    const BatchEntry<float> &e = batch_entry(entries, mstarts, n, entry_sh, r);
    const int l = (int)blockIdx.x - e.mstart;
    BandArgs b = common;
    b.strips = e.mx;
    b.bands = e.my;
    b.qgroup = e.qgroup;
    const int p = __ldg(parity + r) ^ (j & 1);
    pdl_wait();
    band_block<S>(e.a[p], b, l % b.strips, l / b.strips, band_sm);
}

template <typename S>
cudaError_t launch_batch_band(const void *entries, const int *mstarts, const int *parity, int n, int nblocks, int j,
                              const BandArgs &b, cudaStream_t s) {
    cudaError_t e = cudaFuncSetAttribute(batch_band_kernel<S>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)kBandSmemMax);
    if (e != cudaSuccess) return e;
    return launch_shared(batch_band_kernel<S>, dim3(nblocks), dim3(b.threads), b.smem, s,
                         static_cast<const BatchEntry<float> *>(entries), mstarts, parity, n, j, b);
}

#define BTRIRT_INSTANTIATE_BATCH_BAND(S)                                                                         \
    template cudaError_t launch_batch_band<S>(const void *, const int *, const int *, int, int, int,           \
                                              const BandArgs &, cudaStream_t);
#define BTRIRT_INSTANTIATE_BAND(S) \
    template cudaError_t launch_band<S>(const SweepArgs<float> &, const BandArgs &, cudaStream_t);

}  // namespace btrirt
