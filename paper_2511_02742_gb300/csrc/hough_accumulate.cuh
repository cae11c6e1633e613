// Steps A-B alone with every window's accumulator written out: the (theta,
// rho) histogram of Eq. (1) binned as in Section 5, one per time window
// (Section 6), without peaks or association.  Included by hough_api.cu after
// hough_kernels.cuh; shares its hit staging, votes and export with the find
// kernel, so the histograms equal the ones the find writes in export mode.
#pragma once

namespace hk {

constexpr int kAccStage = 1024;   // hits accumulate_kernel holds in shared memory

// Rows [part * 128 * k, ...) of one window, k tiles of 128 rows a part: the
// unit of work of accumulate_kernel.
struct AccParams {
    KParams k;
    int part_tiles;        // tiles of 128 rows per part
    int parts;             // parts of a window
};

// Theta rows [t0, t0 + R) of a window in counters of P per word.  SUM (P = 4
// with more hits than a byte counts): the bytes are summed as they are
// exported, and false returned when a counter overflowed.
template <class S, int P, bool SUM>
__device__ __forceinline__ bool acc_tile(const KParams &p, long long w, long long beg, int H, int nv,
                                         int t0, uint32_t *tile, int2 *stage, int *wtot,
                                         unsigned *total, WinScalars &ws)
{
    constexpr int R = 32 * P;
    constexpr int lgP = P == 4 ? 2 : (P == 2 ? 1 : 0);
    const int lo = p.lo_tab ? __ldg(p.lo_tab + lgP * p.lo_stride + t0 / R) : 0;
    const unsigned acc0 = (unsigned)__cvta_generic_to_shared(tile) + kGuard * 128u;
    const bool fast = p.in_range && t0 + R <= p.n_theta;
    unsigned votes = (unsigned)nv;
    if (nv >= 0) {
        if (fast)
            vote_tile<S, P, true>(p, acc0, 0u, stage, nv, t0, lo, ws);
        else
            vote_tile<S, P, false>(p, acc0, 0u, stage, nv, t0, lo, ws);
    } else {
        votes = 0u;
        for (long long s0 = 0; s0 < H; s0 += p.hit_stage) {
            const int n = (int)min((long long)p.hit_stage, (long long)H - s0);
            const int ns = stage_hits<S>(p, beg + s0, n, stage, wtot, ws);
            votes += (unsigned)ns;
            if (fast)
                vote_tile<S, P, true>(p, acc0, 0u, stage, ns, t0, lo, ws);
            else
                vote_tile<S, P, false>(p, acc0, 0u, stage, ns, t0, lo, ws);
            __syncthreads();
        }
    }
    if (SUM && threadIdx.x == 0)
        *total = 0u;
    __syncthreads();
    unsigned sum = export_tile_end<S, P, SUM>(p, tile + kGuard * 32, t0, R, lo, w);
    if (SUM) {
        sum = __reduce_add_sync(0xffffffffu, sum);
        if ((threadIdx.x & 31) == 0)
            atomicAdd(total, sum);
    }
    __syncthreads();
    const bool ok = !SUM || *total == votes * (unsigned)min(R, p.n_theta - t0);
    zero_tile<S>(p, tile);
    __syncthreads();
    return ok;
}

// Persistent CTAs stride over (window, part): several per SM, so that one
// CTA's stores run beside another's votes, and parts small enough that the
// last ones end together.  Shared memory: the tile (32 word rows, the bins its
// rows can reach, aligned to 128-byte lines of the output where n_rho allows)
// then the stage of hit_stage (phi, z) pairs.
//
// Bound: HBM writes, 4 n_theta n_rho bytes per window.  500 windows of 960
// hits at 1024 x 1024 (2.1 GB): one full-width tile and one CTA per SM, a
// window each, 587 us; this, 375 us (5.6 TB/s; 5000 windows 6.3 TB/s).
template <class S>
__device__ __forceinline__ void accumulate_body(const AccParams &q)
{
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ WinScalars ws;
    __shared__ int wtot[64];
    __shared__ unsigned total;
    const KParams &p = q.k;
    uint32_t *tile = reinterpret_cast<uint32_t *>(smem);
    int2 *stage = reinterpret_cast<int2 *>(smem + tile_words(32, p.n_b) * 4);
    zero_tile<S>(p, tile);
    const long long n_items = p.n_windows * q.parts;
    for (long long x = blockIdx.x; x < n_items; x += gridDim.x) {
        const long long w = x / q.parts;
        const int part = (int)(x - w * q.parts);
        const long long beg = p.offsets[w], end = p.offsets[w + 1];
        if (!(beg >= 0 && beg <= end && end <= p.n_hits && end - beg < (1ll << 30))) {
            if (part == 0 && threadIdx.x == 0)
                p.status[w] = HOUGH_WIN_BAD_OFFSETS;
            continue;                                  // uniform
        }
        const int H = (int)(end - beg);
        __syncthreads();                               // ws and the stage are reused
        if (threadIdx.x == 0)
            ws.flags = 0u;
        __syncthreads();
        const int nv = H <= p.hit_stage ? stage_hits<S>(p, beg, H, stage, wtot, ws) : -1;
        const int end_t = min(p.n_theta, (part + 1) * q.part_tiles * 128);
        for (int t0 = part * q.part_tiles * 128; t0 < end_t; t0 += 128) {
            bool ok = false;
            if (H <= 255)
                ok = acc_tile<S, 4, false>(p, w, beg, H, nv, t0, tile, stage, wtot, &total, ws);
            else if (p.in_range && H <= 8 * p.n_b)     // as the find: bytes while few hits per bin
                ok = acc_tile<S, 4, true>(p, w, beg, H, nv, t0, tile, stage, wtot, &total, ws);
            if (ok)
                continue;
            const int t1 = min(t0 + 128, end_t);
            if (H <= 65534)
                for (int t = t0; t < t1; t += 64)
                    acc_tile<S, 2, false>(p, w, beg, H, nv, t, tile, stage, wtot, &total, ws);
            else
                for (int t = t0; t < t1; t += 32)
                    acc_tile<S, 1, false>(p, w, beg, H, nv, t, tile, stage, wtot, &total, ws);
        }
        if (part == 0 && threadIdx.x == 0)             // one part where votes may miss the range
            p.status[w] = ws.flags;
    }
}

__global__ void __launch_bounds__(256, 4) accumulate_kernel_256(const __grid_constant__ AccParams q)
{
    accumulate_body<Shape<256, 32>>(q);
}
__global__ void __launch_bounds__(512, 2) accumulate_kernel_512(const __grid_constant__ AccParams q)
{
    accumulate_body<Shape<512, 32>>(q);
}
__global__ void __launch_bounds__(1024, 1) accumulate_kernel_1024(const __grid_constant__ AccParams q)
{
    accumulate_body<Shape<1024, 32>>(q);
}

}  // namespace hk
