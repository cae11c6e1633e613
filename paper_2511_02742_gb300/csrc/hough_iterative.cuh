// hough_iterative.cuh -- device code of the iterative highest-bin search (the
// literal reading of the paper's peak step, repeated): vote the hits not yet
// assigned, take the accumulator's highest bin (ties: first in row-major
// order), stop below T, else give track k every remaining hit within tol
// bins of it in its row, remove them and vote again.
//
// Two kernels.  iterative_kernel takes the windows it has room for: it votes
// the window's hits once, tile by tile as the find does, and lists every bin
// with at least T votes.  Counts only fall as tracks leave, so the highest bin
// of every iteration is a listed one, and taking a track's hits back is a few
// comparisons per listed bin: an iteration is two passes over short lists and
// two barriers, and no accumulator is kept.  iterative_tiles_kernel takes the
// rest: every iteration re-votes the find kernel's theta tiles (32 word rows,
// stored without guard columns), leaving out those that cannot hold the
// highest bin.
#pragma once

#include "hough_kernels.cuh"

namespace hk {

struct IterParams {
    KParams k;                  // hits, tables, shape, thresholds, launch shape
    int max_tracks;
    int4 *tracks;               // [n_windows * max_tracks]: theta, rho, votes, n_hits
    int32_t *n_tracks;          // [n_windows]
    int cap_hits, cap_list;     // iterative_kernel: staged hits and listed bins
};

constexpr int kIterLeft = -1;   // n_tracks of a window left to iterative_tiles_kernel

__host__ __device__ inline size_t iter_smem_bytes(int n_b, int cap_hits, int cap_list)
{
    return tile_words(32, n_b) * 4 + (size_t)cap_hits * 18 + (size_t)cap_list * 4;
}

// Stage the window's valid hits (in order) with their window-local indices;
// invalid hits get hit_track = -2, valid ones -1.  Returns the staged count
// (uniform), or -1 when they do not fit in the stage.
__device__ int iter_stage(const KParams &p, long long beg, int H, int2 *stage, int *sidx,
                          int *wtot)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    int total = 0;
    for (int c0 = 0; c0 < H; c0 += blockDim.x) {
        const int i = c0 + threadIdx.x;
        int phi = 0, z = 0;
        bool ok = false;
        if (i < H) {
            ok = load_hit(p, beg + i, phi, z);
            p.hit_track[beg + i] = ok ? -1 : -2;
        }
        const unsigned m = __ballot_sync(0xffffffffu, ok);
        if (lane == 0)
            wtot[warp] = __popc(m);
        __syncthreads();
        int pre = 0, tot = 0;
        for (int k = 0; k < nw; ++k) {
            const int v = wtot[k];
            pre += k < warp ? v : 0;
            tot += v;
        }
        const int pos = total + pre + __popc(m & lanemask_lt());
        if (ok && pos < p.hit_stage) {
            stage[pos] = make_int2(phi, z);
            sidx[pos] = i;
        }
        total += tot;
        __syncthreads();
    }
    return total <= p.hit_stage ? total : -1;
}

// Highest counter of the voted tile as a key (count << 32 | ~(t << 16 | b)):
// the block maximum is the highest count, first in row-major order.
__device__ __forceinline__ unsigned long long block_max_u64(unsigned long long k,
                                                            unsigned long long *red)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) {
        const unsigned long long o = __shfl_xor_sync(0xffffffffu, k, d);
        k = o > k ? o : k;
    }
    __syncthreads();
    if (lane == 0)
        red[warp] = k;
    __syncthreads();
    unsigned long long m = 0ull;
    for (int i = 0; i < nw; ++i)
        m = red[i] > m ? red[i] : m;
    return m;
}

// The tile's highest bin as the key (count << 32) | (2^32 - 1 - (t << 16 | b)):
// the highest count, then the first bin in row-major order.  Two passes over
// the counters: the highest count (fields only: rows past n_theta never get a
// vote, so every non-zero field is a bin of the accumulator), then the words
// holding that count.  Every thread gets the result.
template <int P>
__device__ unsigned long long tile_best(const KParams &p, const uint32_t *acc, int t0, int lo,
                                        unsigned long long *red)
{
    constexpr int CW = 32 / P;
    constexpr unsigned MASK = P == 1 ? 0xffffffffu : ((1u << CW) - 1u);
    const int words = p.word_rows * p.n_b;
    unsigned m = 0u;
    for (int f = threadIdx.x; f < words; f += blockDim.x) {
        const uint32_t wv = acc[f];
#pragma unroll
        for (int s = 0; s < P; ++s)
            m = max(m, (wv >> (s * CW)) & MASK);
    }
    const unsigned top = (unsigned)(block_max_u64(m, red) & 0xffffffffu);
    if (top == 0u)
        return 0ull;
    unsigned long long best = 0ull;
    for (int f = threadIdx.x; f < words; f += blockDim.x) {
        const uint32_t wv = acc[f];
        if (!has_field<P>(wv, top))
            continue;
        const int b = (f >> 5) + lo;                        // the tile stores bins lo ..
        const int wr = f & 31;
#pragma unroll
        for (int s = 0; s < P; ++s) {
            if (((wv >> (s * CW)) & MASK) != top)
                continue;
            const int t = t0 + wr * P + s;
            const unsigned long long key = ((unsigned long long)top << 32) |
                                           (unsigned long long)(0xffffffffu -
                                                                (((unsigned)t << 16) | (unsigned)b));
            best = key > best ? key : best;
        }
    }
    return block_max_u64(best, red);
}

// One pass over every tile: the highest bin of the remaining hits' votes.
// ub[tile]: an upper bound of the tile's highest count (its highest count
// when it was last voted: removing hits only lowers counts), valid while the
// counter width P, and so the tiling, stays the same.  The tiles are taken in
// decreasing order of their bound (ties: the earlier tile first), so that the
// best count is found early; a tile is voted only if it could still hold the
// highest bin: a bound of at least T and above the best count so far, or
// equal to it in a tile before the best bin's (the first bin in row-major
// order wins a tie).  done: one bit per tile, this call's visits.
template <int P>
__device__ unsigned long long iter_best(const KParams &p, uint32_t *acc, const int2 *stage, int nv,
                                        unsigned long long *red, WinScalars &ws, int *ub,
                                        unsigned *done, int T)
{
    const int R = p.word_rows * P;
    const int n_tiles = (p.n_theta + R - 1) / R;
    const int lane = threadIdx.x & 31;
    constexpr int lgP = P == 4 ? 2 : (P == 2 ? 1 : 0);
    const int32_t *lo_row = p.lo_tab ? p.lo_tab + lgP * p.lo_stride : nullptr;
    unsigned long long best = 0ull;
    int best_tile = n_tiles;
    const unsigned acc0 = (unsigned)__cvta_generic_to_shared(acc);
    for (int i = threadIdx.x; i < (n_tiles + 31) / 32; i += blockDim.x)
        done[i] = 0u;
    __syncthreads();
    for (;;) {
        // every warp picks the same tile: the largest (bound, -index) not yet visited
        unsigned long long pick = 0ull;
        for (int x = lane; x < n_tiles; x += 32) {
            if ((done[x >> 5] >> (x & 31)) & 1u)
                continue;
            const unsigned long long k = ((unsigned long long)(unsigned)ub[x] << 32) |
                                         (unsigned long long)(0xffffffffu - (unsigned)x);
            pick = k > pick ? k : pick;
        }
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) {
            const unsigned long long o = __shfl_xor_sync(0xffffffffu, pick, d);
            pick = o > pick ? o : pick;
        }
        if (pick == 0ull)
            break;                                   // every tile visited
        const int tile = (int)(0xffffffffu - (unsigned)(pick & 0xffffffffu));
        const unsigned bound = (unsigned)(pick >> 32);
        const unsigned top = (unsigned)(best >> 32);
        if ((int)bound < T || bound < top || (bound == top && tile > best_tile))
            break;                                   // no unvisited tile can hold the highest bin
        const int t0 = tile * R;
        const int lo = lo_row ? __ldg(lo_row + tile) : 0;
        uint4 *acc4 = reinterpret_cast<uint4 *>(acc);
        for (int i = threadIdx.x; i < (p.word_rows * p.n_b) >> 2; i += blockDim.x)
            acc4[i] = make_uint4(0u, 0u, 0u, 0u);
        __syncthreads();
        if (p.in_range && t0 + R <= p.n_theta)
            vote_tile<Shape<512, 32>, P, true>(p, acc0, 0u, stage, nv, t0, lo, ws);
        else
            vote_tile<Shape<512, 32>, P, false>(p, acc0, 0u, stage, nv, t0, lo, ws);
        __syncthreads();
        const unsigned long long k = tile_best<P>(p, acc, t0, lo, red);
        if (threadIdx.x == 0) {
            ub[tile] = (int)(k >> 32);
            done[tile >> 5] |= 1u << (tile & 31);
        }
        if (k > best) {
            best = k;
            best_tile = tile;
        }
        __syncthreads();
    }
    return best;
}

__global__ void __launch_bounds__(512, 1) iterative_tiles_kernel(IterParams q)
{
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ WinScalars ws;
    __shared__ unsigned long long red[16];
    __shared__ int wtot[32];
    __shared__ int taken;
    __shared__ unsigned todo[16];
    __shared__ int ub[HOUGH_MAX_THETA / 32];      // per-tile bounds (at most n_theta / 32 tiles)
    __shared__ unsigned done[HOUGH_MAX_THETA / 32 / 32];
    const KParams &p = q.k;
    const int T = p.T;
    uint32_t *acc = reinterpret_cast<uint32_t *>(smem);
    int2 *stage = reinterpret_cast<int2 *>(smem + (size_t)p.word_rows * p.n_b * 4);
    int *sidx = reinterpret_cast<int *>(stage + p.hit_stage);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    // this CTA's windows, 512 looked at together: most are done already
    for (long long k0 = 0; k0 * gridDim.x < p.n_windows; k0 += 512) {
        const long long mine = (k0 + threadIdx.x) * gridDim.x + blockIdx.x;
        const unsigned left = __ballot_sync(0xffffffffu, mine < p.n_windows && q.n_tracks[mine] == kIterLeft);
        __syncthreads();
        if (lane == 0)
            todo[warp] = left;
        __syncthreads();
        for (int x = 0; x < 512; ++x) {
            if (!(todo[x >> 5] >> (x & 31) & 1u)) {
                x |= todo[x >> 5] ? 0 : 31;
                continue;
            }
            const long long w = (k0 + x) * gridDim.x + blockIdx.x;
            const long long beg = p.offsets[w], end = p.offsets[w + 1];
            const int H = (int)(end - beg);
            if (threadIdx.x == 0)
                ws.flags = 0u;
            __syncthreads();
            int nv = iter_stage(p, beg, H, stage, sidx, wtot);
            int found = 0;
            unsigned flags = 0u;
            if (nv < 0) {
                flags |= HOUGH_WIN_TOO_LARGE;
                nv = 0;
            }
            int width = 0;                               // counter fields per word of the bounds
            while (found < q.max_tracks && nv > 0) {
                const int P = nv <= 255 ? 4 : (nv <= 65535 ? 2 : 1);
                if (P != width) {                        // new tiling: no bound known yet
                    for (int i = threadIdx.x; i < HOUGH_MAX_THETA / 32; i += blockDim.x)
                        ub[i] = 0x7fffffff;
                    __syncthreads();
                    width = P;
                }
                unsigned long long best;
                if (P == 4)
                    best = iter_best<4>(p, acc, stage, nv, red, ws, ub, done, T);
                else if (P == 2)
                    best = iter_best<2>(p, acc, stage, nv, red, ws, ub, done, T);
                else
                    best = iter_best<1>(p, acc, stage, nv, red, ws, ub, done, T);
                const int votes = (int)(best >> 32);
                if (votes < T)
                    break;
                const unsigned tb = 0xffffffffu - (unsigned)(best & 0xffffffffu);
                const int bt = (int)(tb >> 16), bb = (int)(tb & 0xffffu);
                const int c = __ldg(p.C + bt), s = __ldg(p.S + bt);
                if (threadIdx.x == 0)
                    taken = 0;
                __syncthreads();
                // mark the line's hits and compact the rest, in order, in place
                int kept = 0, mine = 0;
                for (int c0 = 0; c0 < nv; c0 += blockDim.x) {
                    const int i = c0 + threadIdx.x;
                    int2 h = make_int2(0, 0);
                    int idx = 0;
                    bool keep = false;
                    if (i < nv) {
                        h = stage[i];
                        idx = sidx[i];
                        const int d = rho_bin(h.x, h.y, c, s, p.D, p.K) - bb;
                        if (d <= p.tol && d >= -p.tol) {
                            p.hit_track[beg + idx] = found;
                            ++mine;
                        } else {
                            keep = true;
                        }
                    }
                    const unsigned m = __ballot_sync(0xffffffffu, keep);
                    if (lane == 0)
                        wtot[warp] = __popc(m);
                    __syncthreads();
                    int pre = 0, tot = 0;
                    for (int k = 0; k < nw; ++k) {
                        const int v = wtot[k];
                        pre += k < warp ? v : 0;
                        tot += v;
                    }
                    if (keep) {
                        const int pos = kept + pre + __popc(m & lanemask_lt());
                        stage[pos] = h;
                        sidx[pos] = idx;
                    }
                    kept += tot;
                    __syncthreads();
                }
#pragma unroll
                for (int d = 16; d > 0; d >>= 1)
                    mine += __shfl_xor_sync(0xffffffffu, mine, d);
                if (lane == 0 && mine)
                    atomicAdd(&taken, mine);
                __syncthreads();
                if (threadIdx.x == 0)
                    q.tracks[(size_t)w * q.max_tracks + found] = make_int4(bt, bb, votes, taken);
                nv = kept;
                ++found;
                __syncthreads();
            }
            if (threadIdx.x == 0) {
                q.n_tracks[w] = found;
                p.status[w] = flags | ws.flags;
            }
            __syncthreads();
        }
    }
}

// iterative_kernel's scalars.
struct IterScalars {
    int n_list;          // bins listed (and refused places past the end)
    int taken[2];        // hits of the last track, in turn
    unsigned sum;        // votes in the counters of the tiles so far
    unsigned int flags;
};

// Bins of a voted tile with at least `floor` votes, as keys: votes, then the
// first bin in row-major order, larger is better.
template <class S>
__device__ __forceinline__ void iter_list(const KParams &p, unsigned acc0, int t0, int lo, int floor,
                                          bool count, uint32_t *list, int cap, IterScalars &is)
{
    const int lane = threadIdx.x & 31;
    const int n4 = p.n_b * 8;
    const unsigned low = (1u << (p.tb + p.bb)) - 1u;
    unsigned sum = 0u;
    for (int x = threadIdx.x; x < n4; x += S::threads()) {
        const uint4 v = lds128(acc0 + (unsigned)x * 16u);
        if (count) {
            sum = __dp4a(v.x, 0x01010101u, sum);
            sum = __dp4a(v.y, 0x01010101u, sum);
            sum = __dp4a(v.z, 0x01010101u, sum);
            sum = __dp4a(v.w, 0x01010101u, sum);
        }
        if (!quad_has<4>(v, floor))
            continue;
        const uint32_t y[4] = {v.x, v.y, v.z, v.w};
        const int b = (x >> 3) + lo, t = t0 + (x & 7) * 16;
#pragma unroll
        for (int e = 0; e < 4; ++e)
#pragma unroll
            for (int s = 0; s < 4; ++s) {
                const int n = field<4>(y[e], s);
                if (n >= floor) {
                    const int at = atomicAdd(&is.n_list, 1);
                    if (at < cap)
                        list[at] = (unsigned)n << (p.tb + p.bb) | (low - ((unsigned)(t + e * 4 + s) << p.bb | (unsigned)b));
                }
            }
    }
    if (count) {
        sum = __reduce_add_sync(0xffffffffu, sum);
        if (lane == 0)
            atomicAdd(&is.sum, sum);
    }
}

// One window per CTA, in a grid of all windows: CTAs start as others end, which
// evens windows of different sizes out with no counter in memory that another
// call, or a replayed capture, could be using (5000 windows of 142 hits, and of 1
// to 40 tracks: 0.515 and 3.48 ms with persistent CTAs and a counter, 0.513 and
// 3.48 so; 1e5 windows of 4 hits 0.384 and 0.368).  The staged valid hits, one 8-bit
// tile of 128 rows, and the list of the bins with at least `floor` votes (T, or more
// while the list cannot hold every bin >= T: its tracks are taken first, and
// the hits left are voted again).  Left to iterative_tiles_kernel: windows of
// more hits than are staged or than a key counts, of more than 255 hits where
// the votes cannot be counted back from the bytes (or one overflowed), and
// windows with more equal bins than the list holds.
//
// Bound: instructions -- the vote and scan of the find (once), then per track
// about 5 per listed bin and hit of the track.  5000 windows, 512 x 512, by
// re-voted tiles and by lists: 142 hits 4.53 -> 0.51 ms, 285 hits 9.3 -> 1.7 ms,
// 570 hits 16.3 -> 3.0 ms.  (All rows' 8-bit counters kept in shared memory, the
// votes taken back and the whole accumulator scanned per track: 2.0 ms at 142
// hits, one CTA per SM and four barriers a track.)
template <int NT>
__device__ __forceinline__ void iter_body(const IterParams &q)
{
    using S = Shape<NT, 32>;
    constexpr int nw = NT / 32;
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ WinScalars ws;
    __shared__ IterScalars is;
    __shared__ int wtot[32];
    __shared__ int hist[64];
    const KParams &p = q.k;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const unsigned lt = lanemask_lt();
    const int NB = p.n_b, shift = p.tb + p.bb;
    uint32_t *tile = reinterpret_cast<uint32_t *>(smem);
    int2 *stage = reinterpret_cast<int2 *>(smem + tile_words(32, NB) * 4);
    int2 *tk = stage + q.cap_hits;                       // hits of the last track
    uint32_t *list = reinterpret_cast<uint32_t *>(tk + q.cap_hits);
    uint16_t *sidx = reinterpret_cast<uint16_t *>(list + q.cap_list);
    const unsigned acc0 = (unsigned)__cvta_generic_to_shared(tile) + kGuard * 128u;
    const int n_tiles = (p.n_theta + 127) / 128;
    const int32_t *lo_row = p.lo_tab ? p.lo_tab + 2 * p.lo_stride : nullptr;
    const long long w = blockIdx.x;
    const long long beg = p.offsets[w], end = p.offsets[w + 1];
    if (!(beg >= 0 && beg <= end && end <= p.n_hits && end - beg < (1ll << 30))) {
        if (threadIdx.x == 0) {
            p.status[w] = HOUGH_WIN_BAD_OFFSETS;
            q.n_tracks[w] = 0;
        }
        return;
    }
    const int H = (int)(end - beg);
    if (H > q.cap_hits || H >= 1 << (32 - shift) || (H > 255 && !(p.in_range && H <= 8 * NB))) {
        if (threadIdx.x == 0)
            q.n_tracks[w] = kIterLeft;
        return;
    }
    if (threadIdx.x == 0)
        ws.flags = 0u;
    // stage the valid hits with their window-local indices
    int nv = 0;
    for (int c0 = 0; c0 < H; c0 += NT) {
        const int i = c0 + threadIdx.x;
        int phi = 0, z = 0;
        bool ok = false;
        if (i < H) {
            ok = load_hit(p, beg + i, phi, z);
            p.hit_track[beg + i] = ok ? -1 : -2;
        }
        const unsigned m = __ballot_sync(0xffffffffu, ok);
        if (lane == 0)
            wtot[warp] = __popc(m);
        __syncthreads();
        const int c = lane < nw ? wtot[lane] : 0;
        const int pos = nv + (int)__reduce_add_sync(0xffffffffu, (unsigned)(lane < warp ? c : 0)) + __popc(m & lt);
        if (ok) {
            stage[pos] = make_int2(phi, z);
            sidx[pos] = (uint16_t)i;
        }
        nv += (int)__reduce_add_sync(0xffffffffu, (unsigned)c);
        __syncthreads();
    }
    int found = 0;
    bool left = false;
    while (nv > 0 && found < q.max_tracks) {
        // vote every tile and list its bins >= floor
        int floor = p.T;
        if (threadIdx.x == 0) {
            is.n_list = 0;
            is.sum = 0u;
            is.taken[0] = is.taken[1] = 0;
        }
        __syncthreads();
        for (int k = 0; k < n_tiles && !left; ++k) {
            const int t0 = k * 128;
            const int lo = lo_row ? __ldg(lo_row + k) : 0;
            zero_tile<S>(p, tile);
            __syncthreads();
            if (p.in_range && t0 + 128 <= p.n_theta)
                vote_tile<S, 4, true>(p, acc0, 0u, stage, nv, t0, lo, ws);
            else
                vote_tile<S, 4, false>(p, acc0, 0u, stage, nv, t0, lo, ws);
            int before = is.n_list;                  // of the tiles before (no one adds to it now)
            __syncthreads();
            iter_list<S>(p, acc0, t0, lo, floor, nv > 255, list, q.cap_list, is);
            __syncthreads();
            while (is.n_list > q.cap_list) {
                // raise the floor until half the list is free, drop what
                // falls below it, and list the tile again
                for (int i = threadIdx.x; i < 64; i += NT)
                    hist[i] = 0;
                __syncthreads();
                for (int i = threadIdx.x; i < q.cap_list; i += NT)
                    atomicAdd(&hist[min((int)(list[i] >> shift), 63)], 1);
                __syncthreads();
                int n = 0, v = 64;
                while (v > 0 && n + hist[v - 1] <= q.cap_list / 2)
                    n += hist[--v];
                floor = max(floor + 1, v);
                left = left || v > 63;               // too many to tell apart
                __syncthreads();
                if (warp == 0) {
                    int m = 0;
                    for (int i0 = 0; i0 < before; i0 += 32) {
                        const uint32_t key = i0 + lane < before ? list[i0 + lane] : 0u;
                        const unsigned mk = __ballot_sync(0xffffffffu, (int)(key >> shift) >= floor);
                        if (mk >> lane & 1u)
                            list[m + __popc(mk & lt)] = key;
                        m += __popc(mk);
                        __syncwarp();
                    }
                    if (lane == 0)
                        is.n_list = m;
                }
                __syncthreads();
                before = is.n_list;
                __syncthreads();
                iter_list<S>(p, acc0, t0, lo, floor, false, list, q.cap_list, is);
                __syncthreads();
                if (left)
                    break;
            }
        }
        if (nv > 255 && is.sum != (unsigned)nv * (unsigned)p.n_theta)
            left = true;                             // a byte overflowed
        if (left)
            break;
        // this thread's hits still unassigned: bit k for hit k NT + threadIdx.x
        unsigned alive = 0u;
        for (int k = 0; k * NT + (int)threadIdx.x < nv; ++k)
            alive |= 1u << k;
        // each warp keeps its share of the list, in place, and drops the
        // bins that fall below the floor
        const int first = found, share = (is.n_list + nw - 1) / nw;
        uint32_t *mine = list + warp * share;
        int n = max(min(share, is.n_list - warp * share), 0);
        int n_tk = 0;
        for (;;) {
            // take the last track's votes from the listed bins; the best left
            uint32_t best = 0u;
            int kept = 0;
            for (int i0 = 0; i0 < n; i0 += 32) {
                uint32_t key = i0 + lane < n ? mine[i0 + lane] : 0u;
                if (n_tk > 0) {
                    // a hit is in the bin when its sum is within 2^K of the bin's
                    // first.  Exact mod 2^32 for any geometry: sums are int32, and a
                    // listed bin holds some, so it is [m 2^K, (m + 1) 2^K) inside
                    // int32's range (2^K divides 2^31), which no other sum meets
                    const unsigned at = ((1u << shift) - 1u) - (key & ((1u << shift) - 1u));
                    const int t = min((int)(at >> p.bb), p.n_theta - 1);
                    const unsigned c = (unsigned)__ldg(p.C + t), s = (unsigned)__ldg(p.S + t);
                    const unsigned d = (unsigned)p.D - ((at & ((1u << p.bb) - 1u)) << p.K);
                    const unsigned one = 1u << p.K;
                    const int4 *pair = reinterpret_cast<const int4 *>(tk);
                    unsigned off = 0u;
#pragma unroll 4
                    for (int x = 0; x < n_tk >> 1; ++x) {
                        const int4 h = pair[x];
                        off += (unsigned)h.x * c + (unsigned)h.y * s + d < one ? 1u : 0u;
                        off += (unsigned)h.z * c + (unsigned)h.w * s + d < one ? 1u : 0u;
                    }
                    if (n_tk & 1) {
                        const int2 h = tk[n_tk - 1];
                        off += (unsigned)h.x * c + (unsigned)h.y * s + d < one ? 1u : 0u;
                    }
                    key -= off << shift;
                }
                const bool ok = i0 + lane < n && (int)(key >> shift) >= floor;
                const unsigned mk = __ballot_sync(0xffffffffu, ok);
                if (ok)
                    mine[kept + __popc(mk & lt)] = key;
                kept += __popc(mk);
                best = max(best, ok ? key : 0u);
                __syncwarp();
            }
            n = kept;
            best = __reduce_max_sync(0xffffffffu, best);
            if (lane == 0)
                wtot[warp] = (int)best;
            __syncthreads();
            best = __reduce_max_sync(0xffffffffu, lane < nw ? (unsigned)wtot[lane] : 0u);
            const int votes = (int)(best >> shift);
            if (best == 0u || votes < floor || found == q.max_tracks)
                break;
            const unsigned at = ((1u << shift) - 1u) - (best & ((1u << shift) - 1u));
            const int bt = (int)(at >> p.bb), bb = (int)(at & ((1u << p.bb) - 1u));
            const int c = __ldg(p.C + bt), s = __ldg(p.S + bt);
            int &taken = is.taken[found & 1];
            for (int k = 0; k * NT < nv; ++k) {
                const int i = k * NT + (int)threadIdx.x;
                bool take = false;
                int2 h = make_int2(0, 0);
                if (alive >> k & 1u) {
                    h = stage[i];
                    const int d = rho_bin(h.x, h.y, c, s, p.D, p.K) - bb;
                    take = d <= p.tol && d >= -p.tol;
                }
                const unsigned m = __ballot_sync(0xffffffffu, take);
                if (m != 0u) {
                    int base = 0;
                    if (lane == 0)
                        base = atomicAdd(&taken, __popc(m));
                    base = __shfl_sync(0xffffffffu, base, 0);
                    if (take) {
                        alive &= ~(1u << k);
                        tk[base + __popc(m & lt)] = h;
                        p.hit_track[beg + sidx[i]] = found;
                    }
                }
            }
            __syncthreads();
            n_tk = taken;
            if (threadIdx.x == 0) {
                q.tracks[(size_t)w * q.max_tracks + found] = make_int4(bt, bb, votes, n_tk);
                is.taken[(found + 1) & 1] = 0;
            }
            ++found;
        }
        if (floor == p.T || found == q.max_tracks)
            break;
        if (found == first) {
            left = true;                             // more equal bins than the list holds
            break;
        }
        // the hits left, in order, for the next list
        int kept = 0;
        __syncthreads();
        for (int k = 0; k * NT < nv; ++k) {
            const int i = k * NT + (int)threadIdx.x;
            const bool keep = alive >> k & 1u;
            const int2 h = keep ? stage[i] : make_int2(0, 0);
            const uint16_t ix = keep ? sidx[i] : (uint16_t)0;
            const unsigned m = __ballot_sync(0xffffffffu, keep);
            if (lane == 0)
                wtot[warp] = __popc(m);
            __syncthreads();
            const int c = lane < nw ? wtot[lane] : 0;
            const int pos = kept + (int)__reduce_add_sync(0xffffffffu, (unsigned)(lane < warp ? c : 0)) + __popc(m & lt);
            if (keep) {
                stage[pos] = h;
                sidx[pos] = ix;
            }
            kept += (int)__reduce_add_sync(0xffffffffu, (unsigned)c);
            __syncthreads();
        }
        nv = kept;
    }
    if (threadIdx.x == 0) {
        q.n_tracks[w] = left ? kIterLeft : found;
        p.status[w] = ws.flags;
    }
}

__global__ void __launch_bounds__(128, 4) iterative_kernel_128(IterParams q) { iter_body<128>(q); }
__global__ void __launch_bounds__(256, 2) iterative_kernel_256(IterParams q) { iter_body<256>(q); }
__global__ void __launch_bounds__(512, 1) iterative_kernel_512(IterParams q) { iter_body<512>(q); }

}  // namespace hk
