// hough_coarse_fine.cuh -- device code of the paper's two-stage search
// (coarse 18 x 100 histogram, then a 10 x 10 fine block of the 180 x 1000
// grid; one line per window).  Uses the fixed-point bin of hough_kernels.cuh.
#pragma once

#include <climits>

#include "hough_kernels.cuh"

namespace hk {

// Coarse: every (hit, row) pair of the 18 coarse rows votes into an 18 x 100
// shared histogram; the maximum of (count, -index) gives the coarse bin
// (ties row-major).
// Fine: the (hit, row) pairs of the 10 fine rows inside it vote into a 10 x
// 10 histogram, keeping only the bins of the 10 fine columns; its maximum is
// the line.
constexpr int kCfCoarseT = 18, kCfCoarseR = 100, kCfFineT = 180, kCfFineR = 1000, kCfBlock = 10;

struct CfParams {
    const int32_t *a, *b;          // as KParams
    long long n_hits;
    HitBox box;
    const long long *offsets;
    long long n_windows;
    int32_t Cc[kCfCoarseT], Sc[kCfCoarseT];      // in the kernel's constant bank
    const int32_t *Cf, *Sf;
    int Dc, Kc, Df, Kf;
    int in_range;                  // every valid hit's coarse votes are in range
    int T, tol;
    hough_line *lines;
    int32_t *hit_track;
};

// Windows per CTA (one warp each).
constexpr int kCfWarps = 4;
// Words of a warp's coarse histogram: 9 x 100, two rows to a word; the 8-bit
// form, four rows to a word, needs 5 x 100, and the window's hits (up to 255)
// are kept behind it.
constexpr int kCfWords = 9 * kCfCoarseR, kCfWords8 = 5 * kCfCoarseR;
constexpr int kCfArea = kCfWords8 + 2 * 256;

// The votes of one hit in coarse rows [r0, r0 + n) of the histogram: row
// r0 + r in field r % P of word group r / P.  ALL: every valid hit votes in
// range in every coarse row (the host checked the detector box).
template <int P, bool ALL, int N>
__device__ __forceinline__ void cf_vote(const CfParams &p, unsigned hist, int r0, int phi, int z)
{
    constexpr int CW = 32 / P;
#pragma unroll
    for (int r = 0; r < N; ++r) {
        const int b = rho_bin(phi, z, p.Cc[r0 + r], p.Sc[r0 + r], p.Dc, p.Kc);
        if (ALL || (unsigned)b < (unsigned)kCfCoarseR)
            red_add_shared(hist + (unsigned)((r / P) * kCfCoarseR + b) * 4u, 1u << ((r % P) * CW));
    }
}

// The highest count of a histogram of n_words words (rows r0 ..), and the
// first bin in row-major order that holds it (index row * 100 + bin).
template <int P>
__device__ __forceinline__ void cf_best(const uint32_t *hist, int n_words, int r0, unsigned &top,
                                        unsigned &at)
{
    const int lane = threadIdx.x & 31;
    const uint4 *quad = reinterpret_cast<const uint4 *>(hist);
    unsigned mine;
    if constexpr (P == 4) {
        // odd bytes by their high byte as they are, even bytes shifted up
        uint32_t mo = 0u, me = 0u;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int x = i * 32 + lane;
            if (x < n_words / 4) {
                const uint4 v = quad[x];
                mo = __vimax3_u16x2(__vimax3_u16x2(mo, v.x, v.y), v.z, v.w);
                me = __vimax3_u16x2(__vimax3_u16x2(me, v.x << 8, v.y << 8), v.z << 8, v.w << 8);
            }
        }
        mo = __vmaxu2(mo, me);
        mine = max(mo >> 24, (mo >> 8) & 0xffu);
    } else if constexpr (P == 2) {
        uint32_t m = 0u;
        for (int x = lane; x < n_words / 4; x += 32) {
            const uint4 v = quad[x];
            m = __vimax3_u16x2(__vimax3_u16x2(m, v.x, v.y), v.z, v.w);
        }
        mine = max(m >> 16, m & 0xffffu);
    } else {
        mine = 0u;
        for (int x = lane; x < n_words / 4; x += 32) {
            const uint4 v = quad[x];
            mine = max(max(max(mine, v.x), max(v.y, v.z)), v.w);
        }
    }
    top = __reduce_max_sync(0xffffffffu, mine);
    at = 0xffffffffu;
    if (mine == top) {
        for (int x = lane; x < n_words / 4; x += 32) {
            const uint4 v = quad[x];
            const uint32_t y[4] = {v.x, v.y, v.z, v.w};
            const int g = x / (kCfCoarseR / 4), b = (x - g * (kCfCoarseR / 4)) * 4;
#pragma unroll
            for (int e = 0; e < 4; ++e)
                if (has_field<P>(y[e], top))
#pragma unroll
                    for (int s = 0; s < P; ++s)
                        if ((unsigned)field<P>(y[e], s) == top)
                            at = min(at, (unsigned)((r0 + g * P + s) * kCfCoarseR + b + e));
        }
    }
    at = __reduce_min_sync(0xffffffffu, at);
}

// One window with its hits given by each(f): f(index, valid, phi, z) for the
// lane's hits, in any number of passes.  P: coarse rows per histogram word.
template <int P, class Each>
__device__ __forceinline__ void cf_window(const CfParams &p, long long w, long long beg, bool ok_off,
                                          uint32_t *coarse, uint32_t *fine, Each each)
{
    const int lane = threadIdx.x & 31;
    const unsigned hist = (unsigned)__cvta_generic_to_shared(coarse);
    unsigned top = 0u, at = 0u;
    for (int r0 = 0; r0 < kCfCoarseT; r0 += P == 1 ? 9 : kCfCoarseT) {
        const int n_words = P == 4 ? kCfWords8 : kCfWords;
#pragma unroll 4
        for (int x = lane; x < n_words / 4; x += 32)
            reinterpret_cast<uint4 *>(coarse)[x] = make_uint4(0u, 0u, 0u, 0u);
        __syncwarp();
        each([&](int, bool ok, int phi, int z) {
            if (ok) {
                if constexpr (P == 1)
                    cf_vote<P, false, 9>(p, hist, r0, phi, z);
                else if (p.in_range)
                    cf_vote<P, true, kCfCoarseT>(p, hist, r0, phi, z);
                else
                    cf_vote<P, false, kCfCoarseT>(p, hist, r0, phi, z);
            }
        });
        __syncwarp();
        unsigned t, a;
        cf_best<P>(coarse, n_words, r0, t, a);
        if (r0 == 0 || t > top) {
            top = t;
            at = a;
        }
        __syncwarp();
    }
    // (an empty histogram's first bin is row 0, bin 0)
    const int tc = (int)at / kCfCoarseR, bc = (int)at - tc * kCfCoarseR;
    bool found = (int)top >= p.T;
    int tf = 0, bf = 0, fvotes = 0;
    if (found) {
#pragma unroll
        for (int i = 0; i < 4; ++i)
            fine[i * 32 + lane] = 0u;
        int cf[kCfBlock], sf[kCfBlock];
#pragma unroll
        for (int i = 0; i < kCfBlock; ++i) {
            cf[i] = __ldg(p.Cf + tc * kCfBlock + i);
            sf[i] = __ldg(p.Sf + tc * kCfBlock + i);
        }
        __syncwarp();
        const unsigned fb = (unsigned)__cvta_generic_to_shared(fine);
        each([&](int, bool ok, int phi, int z) {
            if (ok) {
#pragma unroll
                for (int i = 0; i < kCfBlock; ++i) {
                    const int j = rho_bin(phi, z, cf[i], sf[i], p.Df, p.Kf) - bc * kCfBlock;
                    if ((unsigned)j < (unsigned)kCfBlock)
                        red_add_shared(fb + (unsigned)(i * kCfBlock + j) * 4u, 1u);
                }
            }
        });
        __syncwarp();
        unsigned long long fk = 0ull;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int x = i * 32 + lane;
            const unsigned long long k = x < kCfBlock * kCfBlock
                                             ? ((unsigned long long)fine[x] << 32) | (unsigned)(~x)
                                             : 0ull;
            fk = k > fk ? k : fk;
        }
        const unsigned fm = __reduce_max_sync(0xffffffffu, (unsigned)(fk >> 32));
        const unsigned fx = __reduce_max_sync(0xffffffffu, (unsigned)(fk >> 32) == fm ? (unsigned)fk : 0u);
        const int fidx = (int)~fx;
        fvotes = (int)fm;
        tf = tc * kCfBlock + fidx / kCfBlock;
        bf = bc * kCfBlock + fidx % kCfBlock;
        found = fvotes >= p.T;
    }
    // seeds
    int mine = 0;
    const int cft = __ldg(p.Cf + tf), sft = __ldg(p.Sf + tf);
    each([&](int i, bool ok, int phi, int z) {
        int v = -2;
        if (ok) {
            v = -1;
            if (found) {
                const int d = rho_bin(phi, z, cft, sft, p.Df, p.Kf) - bf;
                if (d <= p.tol && d >= -p.tol) {
                    v = 0;
                    ++mine;
                }
            }
        }
        p.hit_track[beg + i] = v;
    });
    mine = (int)__reduce_add_sync(0xffffffffu, (unsigned)mine);
    if (lane == 0) {
        hough_line r;
        r.coarse_theta = ok_off ? tc : 0;
        r.coarse_rho = ok_off ? bc : 0;
        r.coarse_votes = ok_off ? (int)top : 0;
        r.fine_theta = tf;
        r.fine_rho = bf;
        r.fine_votes = fvotes;
        r.n_seeds = mine;
        r.found = found ? 1 : 0;
        p.lines[w] = r;
    }
    __syncwarp();                            // the histograms are cleared next
}

// One warp per window (grid-stride over windows), with its own coarse and
// fine histograms in shared memory, so that no phase waits for a block
// barrier.  A window of up to 255 hits keeps them in shared memory through
// the three passes (coarse, fine, seeds) and counts four coarse rows to a
// word, so that the maximum is four 16-byte loads a lane.  Larger windows read their hits again in each pass, and count in 16
// bits, from 65536 hits in 32 (nine rows at a time).  (Hits in registers with
// the passes unrolled over them overflowed the instruction cache: 0.61 ms.)
//
// Bound: instruction issue (2.0 k warp instructions per window, 76% of issue
// slots).  1e5 windows of 142 hits: 0.44 ms (32-bit counters, hits read and
// encoded three times, 64-bit maxima over 1800 counters) -> 0.24 ms.
__global__ void __launch_bounds__(32 * kCfWarps, 8) coarse_fine_kernel(const __grid_constant__ CfParams p)
{
    __shared__ __align__(16) uint32_t coarse_s[kCfWarps][kCfArea];
    __shared__ __align__(16) uint32_t fine_s[kCfWarps][128];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t *coarse = coarse_s[warp], *fine = fine_s[warp];
    const long long n_warps = (long long)gridDim.x * kCfWarps;
    long long w = (long long)blockIdx.x * kCfWarps + warp;
    long long beg = 0, end = 0;
    if (w < p.n_windows) {
        beg = __ldg(p.offsets + w);
        end = __ldg(p.offsets + w + 1);
    }
    while (w < p.n_windows) {
        const bool ok_off = beg >= 0 && beg <= end && end <= p.n_hits;
        const int H = ok_off ? (int)min(end - beg, (long long)INT_MAX / kCfCoarseT) : 0;
        const long long cur = beg, cw = w;
        w += n_warps;
        if (w < p.n_windows) {               // the next window's, while this one runs
            beg = __ldg(p.offsets + w);
            end = __ldg(p.offsets + w + 1);
        }
        if (H <= 255) {
            int2 *hits = reinterpret_cast<int2 *>(coarse + kCfWords8);
#pragma unroll 4
            for (int h = lane; h < H; h += 32) {
                int phi, z;
                const bool v = encode_hit(p.box, __ldg(p.a + cur + h), __ldg(p.b + cur + h), phi, z);
                hits[h] = make_int2(v ? phi : -1, z);    // valid phi are >= 0
            }
            cf_window<4>(p, cw, cur, ok_off, coarse, fine, [&](auto f) {
#pragma unroll 1
                for (int h = lane; h < H; h += 32) {     // each lane its own
                    const int2 v = hits[h];
                    f(h, v.x >= 0, v.x, v.y);
                }
            });
        } else {
            auto each = [&](auto f) {
#pragma unroll 1
                for (int h = lane; h < H; h += 32) {
                    int phi, z;
                    const bool v = encode_hit(p.box, __ldg(p.a + cur + h), __ldg(p.b + cur + h), phi, z);
                    f(h, v, phi, z);
                }
            };
            if (H <= 65535)
                cf_window<2>(p, cw, cur, ok_off, coarse, fine, each);
            else
                cf_window<1>(p, cw, cur, ok_off, coarse, fine, each);
        }
    }
}

}  // namespace hk
