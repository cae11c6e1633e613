// hough_kernels.cuh -- device code of the track-finding path (sm_103a).
//
// One persistent kernel processes whole time windows (Section 6: one window
// per unit of work).  Per window, in one CTA:
//   1. stage: the window's hits are loaded (encoded on the fly from strip
//      addresses if asked), checked against the detector box and compacted
//      into shared memory;
//   2. for each theta tile: vote (Eq. (1)) into the zeroed shared accumulator
//      tile, scan it for words holding a bin >= T, test those words' bins for
//      3x3 local maxima, feed the peaks to an exact online top-k (Section 4 /
//      Section 5 peak finding), optionally export the tile, and zero it;
//   3. associate every hit with the first peak whose line it lies on and
//      compact the hits per peak (Section 5 seed finding).
//
// Accumulator tile layout.  The tile covers R = WR * P consecutive theta
// rows.  Its WR "word rows" hold P packed counters per 32-bit word: counter s
// of word (wr, j) is the count of bin lo + j in tile row wr*P + s, so the
// rows of a word are neighbours and a whole word's rows above and below come
// from one funnel shift with the word row above or below.  P = 4
// (8-bit) when the window has <= 255 hits, P = 2 (16-bit) when <= 65534, else
// P = 1: a count never exceeds the number of hits, so the packed counters are
// exact.  (Larger windows with few hits for their bins are tried with P = 4
// first and redone if a byte overflowed.)  A tile stores only NB bins [lo, lo + NB) of each row: the bin is
// monotone in phi and in z, so the corners of the detector box bound the bins
// that any hit can reach in a row, and the host gives every tile the first
// bin lo of a window of NB bins that holds every reachable bin inside
// [0, n_rho) of its rows (NB about 0.6 n_rho for 128-row tiles over half a
// turn; NB = n_rho, lo = 0 when no table is given).  Bins outside the window
// are zero in that tile.  Words are stored bank-private: word (wr, j) lives at
//     (kGuard + (wr / 32) * (NB + kGuard) + j) * 32 + wr % 32,
// so every word of word row wr sits in shared-memory bank wr % 32.  kGuard
// columns that no vote reaches stand before, between and after the groups of
// 32 word rows: the 3x3 test reads them as the zeros outside the stored bins.
//
// Voting assigns lane l of a warp to word row 32*g + l and loops the warp over
// hits; each lane adds one vote per packed row.  Lane l only ever touches bank
// l, so a warp's vote is always a single conflict-free wavefront, whatever
// bins the lanes hit (and no two lanes share a word, so no warp aggregation
// is needed).  The votes are reductions without a returned count: about 6
// warp instructions a vote.  (A first version read the returned count and
// listed each bin as it reached T: 13.6 instructions a vote on the batched
// pileup windows and 20 at high pileup, where nearly every vote of a warp
// lists something.)  Finding the bins >= T afterwards is one 16-byte load and
// a few tests per 128 words, once per tile.
#pragma once

#include <cuda_runtime.h>
#include <limits.h>
#include <stddef.h>
#include <stdint.h>

#include "hough.h"

namespace hk {

constexpr int kGuard = 3;       // zero columns around the stored bins of a row group
constexpr int kHistBins = 64;   // peak-vote histogram; last bin = ">= 63"
constexpr int kListCap = 160;   // flagged quads a warp holds: four steps' 128 and 31 left over

// The detector box, and the units of strip addresses.
struct HitBox {
    int raw;                // strip addresses (vane, strip), else encoded (phi, z)
    int vane_step;          // phi units per vane
    int z_min, z_pitch, z_half;
    int z_end;              // z_min + n_z_strips * pitch (at most INT_MAX)
    unsigned phi_end;       // 360 deg in phi units (at most 2^31)
};

struct KParams {
    // hits
    const int32_t *a;   // phi_q, or vane when raw
    const int32_t *b;   // z_q, or strip when raw
    long long n_hits;
    HitBox box;
    // windows
    const long long *offsets;
    long long n_windows;
    // tables
    const int32_t *C;
    const int32_t *S;
    int D;              // tables at scale 2^K: every box hit's sum fits in int32
    int K;
    // the FP64 variant (HOUGH_FLAG_FP64): cos/sin of the row centres and the
    // units, for b = floor((phi/u_phi cos + z/u_z sin - rho_min) / drho)
    const double *Cd;
    const double *Sd;
    double u_phi, u_z, rho_min, drho;
    int fp64;
    int in_range;       // every valid hit votes inside [0, n_rho) in every row
    int n_theta, n_rho;
    // narrowed tiles: NB bins stored per row; the first bin of tile k of
    // counter width P at lo_tab[log2(P) * lo_stride + k] (null: lo = 0)
    int n_b;
    const int32_t *lo_tab;
    int lo_stride;
    int T, tol, max_peaks;
    int export_acc;
    // outputs
    hough_peak *peaks;
    int32_t *n_peaks;
    int32_t *n_found;
    int32_t *hit_track;
    int32_t *track_hits;
    uint32_t *status;
    int32_t *acc;
    // scheduling: [0] next-window counter, [1] finished-CTA counter
    unsigned int *work;
    // launch shape
    int word_rows;      // WR, 32, 64 or 128
    int lw;             // log2(WR)
    int hit_stage;      // HS
    int kp;             // top-k region (power of two >= max(32, max_peaks))
    int pmax;           // counters per word of the find's small windows: 4, or 2 where
                        // 64-row tiles fit n_theta better
    int split;          // CTAs per window (find_split_kernel)
    int tb, bb;         // bits of a theta row and of a rho bin in a 32-bit peak key
    unsigned acc_bytes; // shared memory of the tile (also the association's scratch)
};

// What a kernel instance knows at compile time of its launch shape: threads
// per CTA and word rows of the tile (0: from the launch).  With both known
// the strides of the scan, the votes and the tables are immediate offsets.
template <int NT, int WR>
struct Shape {
    static constexpr int kThreads = NT;
    static __device__ __forceinline__ int threads() { return NT ? NT : (int)blockDim.x; }
    static __device__ __forceinline__ int warps() { return threads() >> 5; }
    static __device__ __forceinline__ int word_rows(const KParams &p) { return WR ? WR : p.word_rows; }
};
using AnyShape = Shape<0, 0>;

// Shared-memory carve-up shared by host (size) and device (pointers).
struct SmemLayout {
    size_t acc, stage, carry, buf, sel, pk, hist, wtot, list, total;
};

__host__ __device__ inline size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

// Words of a tile with its guard columns (n_b: the bins it stores per row).
__host__ __device__ inline size_t tile_words(int word_rows, int n_b)
{
    return ((size_t)(word_rows >> 5) * (n_b + kGuard) + kGuard) * 32;
}

// acc_bytes: the tile, or the association's per-warp counts if they need more.
// kp: the kept peaks, rounded up.
__host__ __device__ inline SmemLayout smem_layout(size_t acc_bytes, int hit_stage, int n_b, int kp,
                                                   int n_warps)
{
    SmemLayout L;
    size_t off = 0;
    L.acc = off;
    off = align_up(off + acc_bytes, 16);
    L.stage = off;
    off = align_up(off + (size_t)hit_stage * 8, 16);
    L.carry = off;                                  // the previous tile's last word rows
    off = align_up(off + (size_t)2 * (n_b + 2 * kGuard) * 4, 16);
    L.buf = off;                                    // kept list, then peaks since the last merge
    off = align_up(off + (size_t)(kp + 256) * 8, 16);
    L.sel = off;                                    // peaks gathered to be ranked
    off = align_up(off + 2048, 16);
    L.hist = off;                                   // peak-vote histogram
    off = align_up(off + kHistBins * 4, 16);
    L.wtot = off;                                   // per-warp counts, two sets
    off = align_up(off + 64 * 4, 16);
    L.list = off;                                   // flagged quads, one list per warp; after
    L.pk = off;                                     // the tiles the kept peaks' lines
    const size_t list = (size_t)n_warps * kListCap * 2, pk = (size_t)kp * 16;
    off = align_up(off + (list > pk ? list : pk), 16);
    L.total = off;
    return L;
}

struct WinScalars {
    unsigned long long kth;   // a peak is kept only if its key < kth
    int n_top;                // kept peaks, sorted, in buf[0 .. n_top)
    int n_buf;                // entries of buf (and refused reservations past the end)
    int fail;                 // first refused reservation (INT_MAX: none)
    int n_sel;                // entries gathered for a merge
    int vk;                   // lower bound of the k-th best vote count
    int n_found;              // local maxima >= T in this window
    unsigned int sum;         // votes in the counters of the tiles so far (SUM)
    unsigned int flags;       // HOUGH_WIN_* for this window
    int next_w;               // next window for this CTA
};

__device__ __forceinline__ unsigned lanemask_lt()
{
    unsigned m;
    asm volatile("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
    return m;
}

// Encoded (phi, z) of a hit, and whether it lies inside the detector box: all
// in 32 bits (a strip address whose phi or z does not fit wraps, as the
// encoded arrays of hough_encode do).
__device__ __forceinline__ bool encode_hit(const HitBox &box, int a, int b, int &phi, int &z)
{
    phi = a;
    z = b;
    if (box.raw) {
        phi = (int)((unsigned)box.vane_step * (unsigned)a);
        z = (int)((unsigned)box.z_min + (unsigned)box.z_pitch * (unsigned)b + (unsigned)box.z_half);
    }
    return (unsigned)phi < box.phi_end && z >= box.z_min && z <= box.z_end;
}

__device__ __forceinline__ bool load_hit(const KParams &p, long long i, int &phi, int &z)
{
    return encode_hit(p.box, __ldg(p.a + i), __ldg(p.b + i), phi, z);
}

// floor((phi*c + z*s + D) / 2^K): the tables' scale keeps the exact sum of
// any hit of the detector box inside int32, so 32-bit wrap-around arithmetic
// gives it exactly; the arithmetic shift is the floor division.
__device__ __forceinline__ int rho_bin(int phi, int z, int c, int s, int D, int K);

// The FP64 variant of the bin: Eq. (1) in double precision with the
// Section 5 binning, each operation rounded to nearest in this order (no
// fused multiply-add), so that it is reproducible: phi_deg = phi / u_phi and
// z_mm = z / u_z once per hit, then per row
// floor(((phi_deg cos + z_mm sin) - rho_min) / drho).
__device__ __forceinline__ int rho_bin64(double phi_deg, double z_mm, double c, double s,
                                         const KParams &p)
{
    const double rho = __dadd_rn(__dmul_rn(phi_deg, c), __dmul_rn(z_mm, s));
    return __double2int_rd(__ddiv_rn(__dsub_rn(rho, p.rho_min), p.drho));
}

__device__ __forceinline__ int rho_bin(int phi, int z, int c, int s, int D, int K)
{
    const unsigned v = (unsigned)phi * (unsigned)c + (unsigned)z * (unsigned)s + (unsigned)D;
    return (int)v >> K;
}

// Stage hits [base, base + n) of the global arrays into `stage`, keeping only
// valid hits, in their original order.  Returns the number staged (uniform).
// wtot: two sets of one count per warp, taken in turn, so that a round of
// blockDim hits passes one block barrier; a last one publishes the stage.
template <class S>
__device__ __forceinline__ int stage_hits(const KParams &p, long long base, int n, int2 *stage, int *wtot,
                                 WinScalars &ws)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = S::warps();
    int total = 0;
    bool bad = false;
    for (int c0 = 0; c0 < n; c0 += S::threads()) {
        int i = c0 + threadIdx.x;
        int phi = 0, z = 0;
        bool ok = false;
        if (i < n) {
            ok = load_hit(p, base + i, phi, z);
            bad |= !ok;
        }
        unsigned m = __ballot_sync(0xffffffffu, ok);
        if (lane == 0)
            wtot[warp] = __popc(m);
        __syncthreads();
        // the counts before this warp's and in all, a warp per lane
        const int c = lane < nw ? wtot[lane] : 0;
        const int pre = (int)__reduce_add_sync(0xffffffffu, (unsigned)(lane < warp ? c : 0));
        if (ok)
            stage[total + pre + __popc(m & lanemask_lt())] = make_int2(phi, z);
        total += (int)__reduce_add_sync(0xffffffffu, (unsigned)c);
        wtot = wtot + ((c0 / S::threads()) & 1 ? -32 : 32);
    }
    if (__syncthreads_or(bad) && threadIdx.x == 0)
        atomicOr(&ws.flags, HOUGH_WIN_HIT_OUT_OF_RANGE);
    return total;
}

__device__ __forceinline__ void red_add_shared(unsigned addr, unsigned v)
{
    asm volatile("red.shared.add.u32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}

__device__ __forceinline__ uint32_t lds32(unsigned addr)
{
    uint32_t v;
    asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(addr) : "memory");
    return v;
}

__device__ __forceinline__ void sts32(unsigned addr, uint32_t v)
{
    asm volatile("st.shared.u32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}

__device__ __forceinline__ uint4 lds128(unsigned addr)
{
    uint4 v;
    asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr) : "memory");
    return v;
}

// Step B on one tile: every staged hit votes once in each of the tile's rows.
// acc0: the shared address of word (0, 0); gstride: bytes from one group of 32
// word rows to the next.  Hits are taken two at a time (one 16-byte broadcast
// load).  FAST: the host proved that every valid hit votes in range, and the
// tile has no row past n_theta, so the per-vote checks are left out.
template <class S, int P, bool FAST, bool F64 = false>
__device__ __forceinline__ void vote_tile(const KParams &p, unsigned acc0, unsigned gstride,
                                          const int2 *stage, int nh, int t0, int lo,
                                          WinScalars &ws)
{
    constexpr int CW = 32 / P;
    const int G = S::word_rows(p) >> 5;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = S::warps();
    const int g = warp % G;
    const int wr = g * 32 + lane;
    const int hstep = nw / G, h0 = warp / G;
    int c[P], s[P];
    double cd[P], sd[P];
    bool act[P];
#pragma unroll
    for (int k = 0; k < P; ++k) {
        const int t = t0 + wr * P + k;
        act[k] = FAST || t < p.n_theta;
        if constexpr (F64) {
            cd[k] = act[k] ? __ldg(p.Cd + t) : 0.0;
            sd[k] = act[k] ? __ldg(p.Sd + t) : 0.0;
            c[k] = s[k] = 0;
        } else {
            if (!FAST) {
                c[k] = act[k] ? __ldg(p.C + t) : 0;
                s[k] = act[k] ? __ldg(p.S + t) : 0;
            }
            cd[k] = sd[k] = 0.0;
        }
    }
    if constexpr (FAST) {                       // P rows at once (t0 is a multiple of 32 P)
        const int t = t0 + wr * P;
        if constexpr (P == 4) {
            const int4 cv = __ldg(reinterpret_cast<const int4 *>(p.C + t));
            const int4 sv = __ldg(reinterpret_cast<const int4 *>(p.S + t));
            c[0] = cv.x, c[1] = cv.y, c[2] = cv.z, c[3] = cv.w;
            s[0] = sv.x, s[1] = sv.y, s[2] = sv.z, s[3] = sv.w;
        } else {
#pragma unroll
            for (int k = 0; k < P; ++k) {
                c[k] = __ldg(p.C + t + k);
                s[k] = __ldg(p.S + t + k);
            }
        }
    }
    // bank-private column of this lane: word (wr, j) at col + 128 j.
    // j = b - lo comes straight from the sum with D - lo 2^K: its exact value
    // lies between 0 and the sum with D for every hit whose bin is >= lo
    // (and lo = 0 when a bin below 0 is reachable), so it fits in int32 too.
    const unsigned col = acc0 + (unsigned)g * gstride + 4u * (unsigned)lane;
    const int K = p.K;
    const int D = (int)((unsigned)p.D - ((unsigned)lo << K));
    // a valid hit's vote is inside [0, n_rho) exactly when j is inside [0, NB)
    const unsigned nr = (unsigned)p.n_b;
    bool oor = false;
    auto vote = [&](int phi, int z) {
        double phd = 0.0, zmm = 0.0;
        if constexpr (F64) {
            phd = __ddiv_rn((double)phi, p.u_phi);
            zmm = __ddiv_rn((double)z, p.u_z);
        }
#pragma unroll
        for (int k = 0; k < P; ++k) {
            int j;
            if constexpr (F64)
                j = rho_bin64(phd, zmm, cd[k], sd[k], p) - lo;
            else
                j = rho_bin(phi, z, c[k], s[k], D, K);
            bool in = true;
            if (!FAST) {
                in = act[k] && (unsigned)j < nr;
                oor |= act[k] && !in;
            }
            if (in)
                red_add_shared(col + (unsigned)j * 128u, 1u << (k * CW));
        }
    };
    const int np = nh >> 1;
    auto each = [&](auto cast) {
        const int4 *stage2 = reinterpret_cast<const int4 *>(stage);
#pragma unroll 2
        for (int h = h0; h < np; h += hstep) {
            const int4 hv = stage2[h];
            cast(hv.x, hv.y);
            cast(hv.z, hv.w);
        }
        if ((nh & 1) && h0 == np % hstep) {     // the odd hit: to the warps that are a pair short
            const int2 hv = stage[nh - 1];
            cast(hv.x, hv.y);
        }
    };
    if constexpr (FAST && P == 4 && S::kThreads >= 512) {
        // The column's place folded into the sum: with its address over 128
        // added to the bin, the sum shifted to K - 7 has the word's address in
        // its upper bits (mod 2^32: they hold addresses below 2^(39 - K)) and
        // the lane's place takes the lower seven -- a shift and one logic
        // operation beside the two multiply-adds, none of them in their pipe,
        // which bounds the votes where an SM has warps enough (high pileup in two
        // CTAs of 512: 0.50 -> 0.48 us per window; four CTAs of 128 threads lost
        // 4%, so they keep the plain form).
        const unsigned base = col - 4u * (unsigned)lane;
        if ((base & 127u) == 0u && base + nr * 128u <= 1u << (39 - K)) {
            const unsigned Df = (unsigned)D + ((base >> 7) << K);
            const int sh = K - 7;
            each([&](int phi, int z) {
#pragma unroll
                for (int k = 0; k < P; ++k) {
                    const unsigned v = (unsigned)phi * (unsigned)c[k] + (unsigned)z * (unsigned)s[k] + Df;
                    red_add_shared(((v >> sh) & ~127u) | (4u * (unsigned)lane), 1u << (k * CW));
                }
            });
            return;
        }
    }
    each(vote);
    if (oor)
        atomicOr(&ws.flags, HOUGH_WIN_VOTE_OUT_OF_RANGE);
}

template <int P>
__device__ __forceinline__ int field(uint32_t w, int s)
{
    constexpr int CW = 32 / P;
    return P == 1 ? (int)w : (int)((w >> (s * CW)) & ((1u << CW) - 1u));
}

// Whether a quad of packed words may hold a counter >= T (never false when it
// does): with the top bit of a field free, adding 2^(cw-1) - T sets it exactly
// when the field is >= T; a word with a top bit set passes as it is.
template <int P>
__device__ __forceinline__ bool quad_has(const uint4 &q, int T)
{
    if constexpr (P == 1) {
        return max(max(q.x, q.y), max(q.z, q.w)) >= (uint32_t)T;
    } else {
        constexpr uint32_t one = P == 4 ? 0x01010101u : 0x00010001u;
        constexpr uint32_t hi = P == 4 ? 0x80808080u : 0x80008000u;
        const uint32_t add = (uint32_t)max((P == 4 ? 128 : 32768) - T, 0) * one;
        return (((q.x + add) | q.x | (q.y + add) | q.y | (q.z + add) | q.z | (q.w + add) | q.w) & hi) != 0u;
    }
}

// Whether some field of w equals v (v < 2^(32/P)): the fields of
// y = w ^ (v in every field) that are zero, by the exact zero-field test
// (y - 0x..01..01) & ~y & 0x..80..80 (non-zero iff some field of y is zero).
template <int P>
__device__ __forceinline__ bool has_field(uint32_t w, unsigned v)
{
    if constexpr (P == 1) {
        return w == v;
    } else if constexpr (P == 2) {
        const uint32_t y = w ^ (v * 0x00010001u);
        return ((y - 0x00010001u) & ~y & 0x80008000u) != 0u;
    } else {
        const uint32_t y = w ^ (v * 0x01010101u);
        return ((y - 0x01010101u) & ~y & 0x80808080u) != 0u;
    }
}

// Peak keys: votes descending, then theta, then rho ascending, as one
// unsigned number (smaller is better; keys are distinct).  32 bits hold it
// while the window's hits (the most votes a bin can have) are below
// 2^(32 - tb - bb): at least 1023 hits in the largest accumulator, always for
// 8-bit counters; larger windows use 64 bits.  Half the shared memory and a
// third of the ranking instructions of 64-bit keys.
template <class Key>
__device__ __forceinline__ Key make_key(const KParams &p, int v, int t, int b)
{
    if constexpr (sizeof(Key) == 4)
        return ((Key)((1u << (32 - p.tb - p.bb)) - 1u - (unsigned)v) << (p.tb + p.bb)) |
               ((Key)t << p.bb) | (Key)b;
    else
        return ((Key)(0xffffffffu - (unsigned)v) << 32) | ((Key)t << 16) | (Key)b;
}

template <class Key>
__device__ __forceinline__ int key_votes(const KParams &p, Key k)
{
    if constexpr (sizeof(Key) == 4)
        return (int)((1u << (32 - p.tb - p.bb)) - 1u - (k >> (p.tb + p.bb)));
    else
        return (int)(0xffffffffu - (unsigned)(k >> 32));
}

template <class Key>
__device__ __forceinline__ int key_theta(const KParams &p, Key k)
{
    if constexpr (sizeof(Key) == 4)
        return (int)((k >> p.bb) & ((1u << p.tb) - 1u));
    else
        return (int)((k >> 16) & 0xffffu);
}

template <class Key>
__device__ __forceinline__ int key_rho(const KParams &p, Key k)
{
    if constexpr (sizeof(Key) == 4)
        return (int)(k & ((1u << p.bb) - 1u));
    else
        return (int)(k & 0xffffu);
}

// The peaks of a window while its tiles are processed: buf holds the kept
// list (sorted, after a merge) and every peak appended since.
template <class Key>
struct PeakStore {
    Key *buf;
    int cap;       // entries buf holds
    Key *sel;
    int sel_cap;   // entries sel holds, at least HOUGH_MAX_PEAKS
    int *hist;     // votes of the appended peaks
};

// A lower bound of the k-th best vote count, from the histogram of the votes
// of every peak appended in the window: the largest v with at least max_peaks
// peaks of >= v votes.  No peak with fewer can be among the best max_peaks.
// Every warp works it out itself.
template <class Key>
__device__ __forceinline__ int vote_bound(const KParams &p, const PeakStore<Key> &st,
                                          const WinScalars &ws)
{
    const int lane = threadIdx.x & 31;
    const int h0 = st.hist[2 * lane], h1 = st.hist[2 * lane + 1];
    const int mine = h0 + h1;
    int suf = mine;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const int y = __shfl_down_sync(0xffffffffu, suf, d);
        if (lane + d < 32)
            suf += y;
    }
    const int above = suf - mine;
    int best = 0;
    if (above + h1 >= p.max_peaks)
        best = 2 * lane + 1;
    else if (suf >= p.max_peaks)
        best = 2 * lane;
    return max((int)__reduce_max_sync(0xffffffffu, (unsigned)best), ws.vk);
}

// Gather the first n entries of buf with >= vk votes into sel, in any order
// (entries past sel's end are counted only).
template <class S, class Key>
__device__ __forceinline__ void gather_peaks(const KParams &p, const PeakStore<Key> &st, int n,
                                             int vk, WinScalars &ws)
{
    const int lane = threadIdx.x & 31;
    for (int i0 = threadIdx.x & ~31; i0 < n; i0 += S::threads()) {
        const int i = i0 + lane;
        const Key key = i < n ? st.buf[i] : (Key)0;
        const bool ok = i < n && key_votes(p, key) >= vk;
        const unsigned m = __ballot_sync(0xffffffffu, ok);
        if (m == 0u)
            continue;
        int base = 0;
        if (lane == 0)
            base = atomicAdd(&ws.n_sel, __popc(m));
        base = __shfl_sync(0xffffffffu, base, 0) + __popc(m & lanemask_lt());
        if (ok && base < st.sel_cap)
            st.sel[base] = key;
    }
}

// place(r, key) for every one of m distinct keys whose rank r (the number of
// smaller keys) is below keep: four lanes a key.
template <class S, class Key, class Place>
__device__ __forceinline__ void rank_peaks(const Key *src, int m, int keep, Place place)
{
    const int sub = threadIdx.x & 3;
    for (int i0 = (int)threadIdx.x >> 2; i0 < ((m + 7) & ~7); i0 += S::threads() >> 2) {
        const Key x = src[min(i0, m - 1)];
        int r = 0;
#pragma unroll 4
        for (int y = sub; y < m; y += 4)
            r += src[y] < x ? 1 : 0;
        r += __shfl_xor_sync(0xffffffffu, r, 1);
        r += __shfl_xor_sync(0xffffffffu, r, 2);
        if (sub == 0 && i0 < m && r < keep)
            place(r, x);
    }
}

// Merge the peaks appended since the last merge into the kept list, while the
// window's tiles go on (all threads call, after a barrier): the entries with
// enough votes are gathered and the best max_peaks written back in order.
template <class S, class Key>
__device__ __forceinline__ void merge_peaks(const KParams &p, const PeakStore<Key> &st, WinScalars &ws)
{
    const int n = min(ws.n_buf, ws.fail);
    const int vk = vote_bound(p, st, ws);
    gather_peaks<S>(p, st, n, vk, ws);
    __syncthreads();
    const int m = ws.n_sel;
    const int keep = min(p.max_peaks, m);
    if (m <= st.sel_cap) {
        rank_peaks<S>(st.sel, m, keep, [&](int r, Key x) { st.buf[r] = x; });
    } else {
        // more ties at vk than sel holds: rank all of buf (entries below vk
        // have larger keys than any other)
        rank_peaks<S>(st.buf, n, keep, [&](int r, Key x) { st.sel[r] = x; });
        __syncthreads();
        for (int i = threadIdx.x; i < keep; i += S::threads())
            st.buf[i] = st.sel[i];
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        ws.n_buf = keep;
        ws.fail = INT_MAX;
        ws.n_sel = 0;
        ws.vk = vk;
        if (keep == p.max_peaks)
            ws.kth = (unsigned long long)st.buf[keep - 1];
    }
    __syncthreads();
}

// The window's kept peaks in order (all threads call, after a barrier), and
// their lines for the association: pk[r] = C, S and the offset D - first bin
// of the r-th peak's line, and its row and bin.  Few entries are ranked as
// they are; more are gathered by votes first.  The caller's next barrier
// publishes both.  Returns the sorted keys and their number.
template <class S, class Key>
__device__ __forceinline__ const Key *finish_peaks(const KParams &p, const PeakStore<Key> &st,
                                                   int4 *pk, int &n_top, WinScalars &ws)
{
    int m = ws.n_buf;
    const Key *src = st.buf;
    Key *dst = st.sel;
    if (m > 96) {
        gather_peaks<S>(p, st, m, vote_bound(p, st, ws), ws);
        __syncthreads();
        if (ws.n_sel <= st.sel_cap) {
            m = ws.n_sel;
            src = st.sel;
            dst = st.buf;
        }
    }
    n_top = min(p.max_peaks, m);
    rank_peaks<S>(src, m, n_top, [&](int r, Key x) {
        const int t = key_theta(p, x), b = key_rho(p, x);
        dst[r] = x;
        pk[r] = make_int4(__ldg(p.C + t), __ldg(p.S + t),
                          (int)((unsigned)p.D - ((unsigned)(b - p.tol) << p.K)), t | b << 16);
    });
    if (threadIdx.x == 0)
        ws.n_top = n_top;
    return dst;
}

// What the 3x3 test of a tile needs: the tile, and the previous tile's last
// word row (carry), whose last row could not be tested without this tile.
struct TileView {
    unsigned acc0;      // shared address of word (0, 0)
    unsigned gstride;   // bytes between groups of 32 word rows
    unsigned zero;      // shared address of a word that is always 0
    unsigned carry_a;   // word row WR-2 of the previous tile (P = 1), bin 0
    unsigned carry_b;   // word row WR-1 of the previous tile, bin 0
    int t0, lo, dlo;    // dlo = lo - the previous tile's lo
    bool last;          // the accumulator's last tile
};

// The rows of one quad (word rows 4q .. 4q + 3 of a row group at one bin)
// that are peaks: > the earlier neighbours in row-major order, >= the later
// ones, and >= T (counted in `peaks`) or >= vk (returned as a mask, bit
// quad_bit of each; vk >= T).  c, m, n: the words at the bin, the one before
// and the one after, from the word row above the quad to the one below.
// top: whether the quad's last row counts (its row below is in this tile).
//
// Packed compare: with the fields' top bits free, the top bit of a field of
// (v | top) - x says v >= x, of (v | top) - 1 - x that v > x, and no field
// borrows from the next; the eight compares of a word's P rows are eight
// subtractions and four three-input ands.  quad_peaks_slow takes the quads
// that hold a count with its top bit set.
template <int P>
__device__ __forceinline__ unsigned quad_peaks(const uint32_t *c, const uint32_t *m,
                                               const uint32_t *n, int T, int vk, bool top,
                                               int &peaks)
{
    constexpr int CW = 32 / P;
    constexpr uint32_t one = P == 4 ? 0x01010101u : 0x00010001u, hi = one << (CW - 1);
    constexpr int half = 1 << (CW - 1);
    // half - T and half - vk per field; with T or vk past the fields, 0 - 1
    // votes more than any field holds
    const uint32_t tt = (uint32_t)max(half - T, 0) * one, kk = (uint32_t)max(half - vk, 0) * one;
    const uint32_t cut = top ? hi : hi & (hi >> CW);
    unsigned am = 0u;
    peaks = 0;
#pragma unroll
    for (int i = 1; i <= 4; ++i) {
        const uint32_t v = c[i] | hi, w = v - one;
        const uint32_t e = (w - __funnelshift_l(m[i - 1], m[i], CW)) & (w - __funnelshift_l(c[i - 1], c[i], CW)) &
                           (w - __funnelshift_l(n[i - 1], n[i], CW)) & (w - m[i]);
        const uint32_t l = (v - __funnelshift_r(m[i], m[i + 1], CW)) & (v - __funnelshift_r(c[i], c[i + 1], CW)) &
                           (v - __funnelshift_r(n[i], n[i + 1], CW)) & (v - n[i]);
        const uint32_t pk = e & l & (i == 4 ? cut : hi);
        peaks += __popc(pk & (c[i] + tt));
        am |= (pk & (c[i] + kk)) >> (4 - i);
    }
    return am;
}

// Row (within the quad's 4 P) of a mask bit of quad_peaks: word bit & 3 =
// 3 - (CW - 1 - bit within the field).
template <int P>
__device__ __forceinline__ int quad_row(int bit)
{
    constexpr int CW = 32 / P;
    const int f = bit / CW;
    return (bit - f * CW - (CW - 4)) * P + f;
}

// The count of a quad's row.
template <int P>
__device__ __forceinline__ int quad_count(const uint32_t *c, int row)
{
    const int i = row / P;
    const uint32_t w = i == 0 ? c[1] : (i == 1 ? c[2] : (i == 2 ? c[3] : c[4]));
    return field<P>(w, row % P);
}

// quad_peaks for any counts, row by row (32-bit counters, and the rare quads
// with a count of half a field's range or more).  a: the quad's shared
// address; au, ad: the words above and below it, su, sd: their distances from
// one bin to the next.
template <int P>
__device__ __noinline__ unsigned quad_peaks_slow(unsigned a, unsigned au, unsigned su, unsigned ad,
                                                 unsigned sd, int T, int vk, bool top, int &peaks)
{
    constexpr int CW = 32 / P;
    // the count in row r of the quad, at the bin before (-1), at it, or after
    auto at = [&](int r, int side) {
        const int i = r < 0 ? -1 : r / P;
        const unsigned w = i < 0 ? au + (unsigned)side * su
                                 : (i > 3 ? ad + (unsigned)side * sd : a + (unsigned)(i * 4 + side * 128));
        return field<P>(lds32(w), i < 0 ? P - 1 : r % P);
    };
    unsigned am = 0u;
    peaks = 0;
    for (int r = 0; r < 4 * P - (top ? 0 : 1); ++r) {
        const int v = at(r, 0);
        if (v < T)
            continue;
        const int e = max(max(at(r - 1, -1), at(r - 1, 0)), max(at(r - 1, 1), at(r, -1)));
        const int l = max(max(at(r + 1, -1), at(r + 1, 0)), max(at(r + 1, 1), at(r, 1)));
        if (v <= e || v < l)
            continue;
        ++peaks;
        if (v >= vk)
            am |= 1u << ((r % P) * CW + CW - 4 + r / P);
    }
    return am;
}

// Step C on one voted tile.  The previous tile's last row comes first, a lane
// per bin.  Then each warp scans its share of the tile (16 bytes a lane: a
// quad of four word rows of a bin; four bins a warp step), lists the quads
// that hold a bin >= T, and tests 32 listed quads at a time, one per lane,
// all 4 P rows of a quad at once: the twelve words and six edge words they
// need come from three 16-byte and six 4-byte loads, and the zero columns
// beside the stored bins stand for the bins outside them.  The scan's lanes that hold the last word row save
// it for the next tile (carry_next).  A peak enters the store if it can still
// be among the best; a lane that finds the store full keeps its quad listed,
// and the block merges and the warps go on.  Every warp leaves through the
// same barrier.  Returns this lane's count of peaks.
//
// Bound: the scan is one 16-byte load and about 20 instructions per 128
// words, whatever they hold; the tests grow with the bins >= T (about 200
// instructions for 32 quads).  2e4 windows of 142 hits at 512 x 512 take 0.99
// ms: votes 0.28, scan 0.20, tests 0.24, association 0.14, the rest 0.14.  The
// warps' last lists are tested partly filled: dealing them out 32 to a warp
// halves those tests but needs one more barrier a tile, and took 1.08 ms.
template <class S, int P, class Key, bool SUM>
__device__ __forceinline__ int find_peaks(const KParams &p, const TileView &tv,
                                          unsigned carry_next, uint16_t *list,
                                          const PeakStore<Key> &st, WinScalars &ws)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = S::warps();
    const unsigned lt = lanemask_lt();
    const int WR = S::word_rows(p), G = WR >> 5, NB = p.n_b, NBQ = NB >> 2, T = p.T;
    const int n_carry = tv.t0 > 0 ? NB : 0;
    int y = warp * 32;               // next carried bin
    unsigned todo = ~0u;             // lanes of that chunk still to be taken
    int gl = 0, x = warp;            // row group, and its next scan step
    int n = 0;                       // listed quads (of that row group)
    int found = 0;
    unsigned sum = 0u;               // votes in the fields scanned
    int seen = p.max_peaks;          // peaks stored when vk was last worked out
    Key kth = (Key)ws.kth;
    int vk = ws.vk;
    // reserve room for c peaks: the first place, or -1 when the store is full
    auto reserve = [&](int c) {
        const int base = atomicAdd(&ws.n_buf, c);
        if (base + c <= st.cap)
            return base;
        atomicMin(&ws.fail, base);
        return -1;
    };
    auto store = [&](int at, Key key, int v) {
        st.buf[at] = key;
        atomicAdd(st.hist + min(v, kHistBins - 1), 1);
    };
    for (;;) {
        bool stop = false;
        while (y < n_carry) {
            const int j = y + lane;
            const unsigned a = tv.carry_b + (unsigned)(j * 4);
            bool full = false;
            if (j < NB && (todo >> lane & 1u)) {
                const uint32_t w = lds32(a);
                const int v = field<P>(w, P - 1);
                if (v >= T) {
                    const uint32_t wm = lds32(a - 4u), wn = lds32(a + 4u);
                    int u0, um, un;
                    if constexpr (P == 1) {
                        const unsigned b = tv.carry_a + (unsigned)(j * 4);
                        u0 = (int)lds32(b), um = (int)lds32(b - 4u), un = (int)lds32(b + 4u);
                    } else {
                        u0 = field<P>(w, P - 2), um = field<P>(wm, P - 2), un = field<P>(wn, P - 2);
                    }
                    const unsigned d = tv.acc0 + (unsigned)(min(max(j - tv.dlo, -2), NB + 1) * 128);
                    const int d0 = field<P>(lds32(d), 0), dm = field<P>(lds32(d - 128u), 0),
                              dn = field<P>(lds32(d + 128u), 0);
                    const int e = max(max(um, u0), max(un, field<P>(wm, P - 1)));
                    const int l = max(max(dm, d0), max(dn, field<P>(wn, P - 1)));
                    if (v > e && v >= l) {
                        const Key key = make_key<Key>(p, v, tv.t0 - 1, j + tv.lo - tv.dlo);
                        if (v >= vk && key < kth) {
                            const int at = reserve(1);
                            full = at < 0;
                            if (!full)
                                store(at, key, v);
                        }
                        found += full ? 0 : 1;
                    }
                }
            }
            todo = __ballot_sync(0xffffffffu, full);
            if (todo != 0u) {
                stop = true;
                break;
            }
            todo = ~0u;
            y += nw * 32;
        }
        while (!stop) {
            // scan, four steps at a time, until 32 quads are listed
            const unsigned scan0 = tv.acc0 + (unsigned)gl * tv.gstride + (unsigned)lane * 16u;
            const unsigned save0 = carry_next + (unsigned)(lane >> 3) * 4u;
            const bool save = P > 1 && carry_next && gl == G - 1 && (lane & 7) == 7;
            while (n < 32 && x < NBQ) {
                uint4 q[4];
                bool f[4];
                bool any = false;
#pragma unroll
                for (int k = 0; k < 4; ++k)
                    q[k] = k == 0 || x + k * nw < NBQ ? lds128(scan0 + (unsigned)x * 512u + (unsigned)(k * nw) * 512u)
                                                      : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    if (save && (k == 0 || x + k * nw < NBQ))
                        sts32(save0 + (unsigned)x * 16u + (unsigned)(k * nw) * 16u, q[k].w);
                    if (SUM) {
                        sum = __dp4a(q[k].x, 0x01010101u, sum);
                        sum = __dp4a(q[k].y, 0x01010101u, sum);
                        sum = __dp4a(q[k].z, 0x01010101u, sum);
                        sum = __dp4a(q[k].w, 0x01010101u, sum);
                    }
                    f[k] = quad_has<P>(q[k], T);
                    any |= f[k];
                }
                if (__any_sync(0xffffffffu, any)) {
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        const unsigned mk = __ballot_sync(0xffffffffu, f[k]);
                        if (f[k])
                            list[n + __popc(mk & lt)] = (uint16_t)((x + k * nw) * 32 + lane);
                        n += __popc(mk);
                    }
                }
                x += 4 * nw;
            }
            if (n == 0) {
                if (gl + 1 == G)
                    break;
                ++gl;
                x = warp;
                continue;
            }
            __syncwarp();
            // test up to 32 listed quads
            const int m = min(n, 32);
            const bool in = lane < m;
            const int id = in ? list[n - m + lane] : 0;
            const int jj = id >> 3, wr = gl * 32 + (id & 7) * 4;
            const unsigned a = tv.acc0 + (unsigned)gl * tv.gstride + (unsigned)id * 16u;
            // the word rows above (the carry for the tile's first) and below
            unsigned au = a - 4u, su = 128u, ad = a + 16u, sd = 128u;
            if ((wr & 31) == 0) {
                au = a - tv.gstride + 124u;          // word row 31 of the group before
                if (wr == 0) {
                    au = tv.t0 > 0 ? tv.carry_b + (unsigned)(min(max(jj + tv.dlo, -2), NB + 1) * 4) : tv.zero;
                    su = tv.t0 > 0 ? 4u : 0u;
                }
            }
            if ((wr & 31) == 28) {
                ad = a - 112u + tv.gstride;          // word row 0 of the group after
                if (wr + 4 == WR) {
                    ad = tv.zero;
                    sd = 0u;
                }
            }
            const uint4 qc = lds128(a), qm = lds128(a - 128u), qn = lds128(a + 128u);
            const uint32_t cw[6] = {lds32(au), qc.x, qc.y, qc.z, qc.w, lds32(ad)};
            const uint32_t mw[6] = {lds32(au - su), qm.x, qm.y, qm.z, qm.w, lds32(ad - sd)};
            const uint32_t nx[6] = {lds32(au + su), qn.x, qn.y, qn.z, qn.w, lds32(ad + sd)};
            const bool top = tv.last || wr + 4 < WR;
            int peaks;
            unsigned am;
            uint32_t big = 0u;                       // a top bit set among the fields
#pragma unroll
            for (int i = 0; i < 6; ++i)
                big |= cw[i] | mw[i] | nx[i];
            bool fast = false;
            if constexpr (P > 1) {
                fast = !__any_sync(0xffffffffu, (big & (P == 4 ? 0x80808080u : 0x80008000u)) != 0u);
                if (fast)
                    am = quad_peaks<P>(cw, mw, nx, T, max(vk, T), top, peaks);
            }
            if (!fast)
                am = quad_peaks_slow<P>(a, au, su, ad, sd, T, max(vk, T), top, peaks);
            if (!in) {
                am = 0u;
                peaks = 0;
            }
            bool full = false;
            if (__any_sync(0xffffffffu, am != 0u)) {
                const int t = tv.t0 + wr * P, b = tv.lo + jj;
                auto key_of = [&](unsigned r, int &v) {
                    const int row = quad_row<P>(__ffs(r) - 1);
                    v = quad_count<P>(cw, row);
                    return make_key<Key>(p, v, t + row, b);
                };
                int v;
                // windows of 256 hits and more find hundreds of peaks per tile:
                // as they are stored the bound rises, so take it from the
                // histogram as it stands, not only at a merge (uneven heavy
                // windows 427 -> 406 us; smaller windows lost 1%)
                if constexpr (SUM) {
                    // one lane's look, for all: other warps are adding to it, and
                    // the bound below is worked out by the whole warp
                    int stored = 0;
                    if (lane == 0)
                        stored = *reinterpret_cast<volatile int *>(&ws.n_buf);
                    stored = __shfl_sync(0xffffffffu, stored, 0);
                    if (stored - seen >= p.max_peaks) {
                        seen = stored;
                        vk = vote_bound(p, st, ws);
                        for (unsigned r = am; r != 0u; r &= r - 1u)
                            if (quad_count<P>(cw, quad_row<P>(__ffs(r) - 1)) < vk)
                                am &= ~(r & (0u - r));
                    }
                }
                if (kth != (Key)~(Key)0)             // with vk votes, the k-th best may still be before it
                    for (unsigned r = am; r != 0u; r &= r - 1u)
                        if (key_of(r, v) >= kth)
                            am &= ~(r & (0u - r));
                if (am != 0u) {
                    int at = reserve(__popc(am));
                    full = at < 0;
                    for (unsigned r = full ? 0u : am; r != 0u; r &= r - 1u) {
                        const Key key = key_of(r, v);
                        store(at++, key, v);
                    }
                }
            }
            found += full ? 0 : peaks;
            const unsigned left = __ballot_sync(0xffffffffu, full);
            n -= m;
            if (left != 0u) {
                __syncwarp();
                if (full)
                    list[n + __popc(left & lt)] = (uint16_t)id;
                n += __popc(left);
                stop = true;
            }
            __syncwarp();
        }
        if (SUM && !stop) {
            sum = __reduce_add_sync(0xffffffffu, sum);
            if (lane == 0)
                atomicAdd(&ws.sum, sum);
            sum = 0u;
        }
        if (!__syncthreads_or(stop))
            return found;
        merge_peaks<S>(p, st, ws);
        kth = (Key)ws.kth;
        vk = ws.vk;
        seen = p.max_peaks;
    }
}

// The P counters of four packed words as four int32 (field s of each).
template <int P>
__device__ __forceinline__ int4 fields4(const uint4 &v, int s)
{
    constexpr int CW = 32 / P;
    constexpr unsigned MASK = P == 1 ? 0xffffffffu : ((1u << CW) - 1u);
    return make_int4((int)((v.x >> (s * CW)) & MASK), (int)((v.y >> (s * CW)) & MASK),
                     (int)((v.z >> (s * CW)) & MASK), (int)((v.w >> (s * CW)) & MASK));
}

// Export mode, at the end of a tile (after the check, when the tile is not
// read again): the tile's rows written as int32 to acc[w][t][b].  Each warp
// takes blocks of 32 word rows x 32 stored bins (1024 consecutive words): it
// holds the block in registers, writes it back transposed in place -- word
// row r becomes 32 consecutive words, its 16-byte chunk c stored at chunk
// c ^ (r & 7), so that the 16-byte writes and reads that follow take the
// fewest wavefronts -- then each lane reads four bins of one word row and
// writes each of its P theta rows with one 16-byte store (a warp store covers
// four whole 128-byte lines).  lo is a multiple of 4, so those stores are
// aligned.  Stored bins past the last whole block, tiles with rows past
// n_theta and accumulators that are not 16-byte aligned go out with 4-byte
// stores; the bins the tile does not store are written as zeros.
// SUM: returns this lane's share of the sum of the tile's bytes (P = 4).
template <class S, int P, bool SUM = false>
__device__ __forceinline__ unsigned export_tile_end(const KParams &p, uint32_t *acc, int t0, int R,
                                                    int lo, long long w)
{
    constexpr int CW = 32 / P;
    constexpr unsigned MASK = P == 1 ? 0xffffffffu : ((1u << CW) - 1u);
    const int G = S::word_rows(p) >> 5, NB = p.n_b;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = S::warps();
    const int nblk = NB >> 5;
    int32_t *out = p.acc + (size_t)w * p.n_theta * p.n_rho;
    const bool vec = (reinterpret_cast<uintptr_t>(p.acc) & 15u) == 0u;
    const bool fast = t0 + R <= p.n_theta && vec;
    unsigned sum = 0u;
    for (int item = warp; item < G * nblk; item += nw) {
        const int g = item / nblk, j0 = (item - g * nblk) * 32;
        uint32_t *blk = acc + (size_t)(g * (NB + kGuard) + j0) * 32;
        uint32_t r[32];
#pragma unroll
        for (int j = 0; j < 32; ++j)
            r[j] = blk[j * 32 + lane];                 // word (g*32 + lane, j0 + j)
        if (SUM)
#pragma unroll
            for (int j = 0; j < 32; ++j)
                sum = __dp4a(r[j], 0x01010101u, sum);
        __syncwarp();
#pragma unroll
        for (int c = 0; c < 8; ++c)
            *reinterpret_cast<uint4 *>(blk + lane * 32 + ((c ^ (lane & 7)) << 2)) =
                make_uint4(r[4 * c], r[4 * c + 1], r[4 * c + 2], r[4 * c + 3]);
        __syncwarp();
        if (fast) {
            // lane: word row q + (lane >> 3), bins lo + j0 + 4 (lane & 7) .. + 3
            const int rs = lane >> 3, c = lane & 7;
            int32_t *o = out + (size_t)(t0 + (g * 32 + rs) * P) * p.n_rho + lo + j0 + 4 * c;
#pragma unroll 4
            for (int q = 0; q < 32; q += 4) {
                const int row = q + rs;
                const uint4 v = *reinterpret_cast<const uint4 *>(blk + row * 32 + ((c ^ (row & 7)) << 2));
#pragma unroll
                for (int s = 0; s < P; ++s)
                    __stcs(reinterpret_cast<int4 *>(o + (size_t)(q * P + s) * p.n_rho), fields4<P>(v, s));
            }
        } else {
            for (int q = 0; q < 32; ++q) {
                const uint32_t v = blk[q * 32 + ((((lane >> 2) ^ (q & 7))) << 2) + (lane & 3)];
#pragma unroll
                for (int s = 0; s < P; ++s) {
                    const int t = t0 + (g * 32 + q) * P + s;
                    if (t < p.n_theta)
                        out[(size_t)t * p.n_rho + lo + j0 + lane] = (int)((v >> (s * CW)) & MASK);
                }
            }
        }
    }
    // stored bins past the last whole block: one bin of 32 word rows per warp
    // step, one lane per word row
    const int rb = nblk * 32, nr = NB - rb;
    for (int x = warp; x < G * nr; x += nw) {
        const int g = x / nr, j = rb + (x - g * nr);
        const int wr = g * 32 + lane;
        const uint32_t v = acc[(size_t)(g * (NB + kGuard) + j) * 32 + lane];
        if (SUM)
            sum = __dp4a(v, 0x01010101u, sum);
#pragma unroll
        for (int s = 0; s < P; ++s) {
            const int t = t0 + wr * P + s;
            if (t < p.n_theta)
                out[(size_t)t * p.n_rho + lo + j] = (int)((v >> (s * CW)) & MASK);
        }
    }
    // the bins the tile does not store, [0, lo) and [lo + NB, n_rho) of every
    // row: zeros, four bins per store (lo, NB and n_rho are multiples of 4)
    const int nq = (p.n_rho - NB) >> 2;
    if (nq > 0) {
        const int nrows = min(R, p.n_theta - t0);
        for (int i = warp; i < nrows; i += nw) {         // a row per warp step
            int32_t *row = out + (size_t)(t0 + i) * p.n_rho;
            for (int k = lane; k < nq; k += 32) {
                int32_t *o = row + (4 * k < lo ? 4 * k : 4 * k + NB);
                if (vec) {
                    __stcs(reinterpret_cast<int4 *>(o), make_int4(0, 0, 0, 0));
                } else {
                    o[0] = 0;
                    o[1] = 0;
                    o[2] = 0;
                    o[3] = 0;
                }
            }
        }
    }
    return sum;
}

// Zero the whole tile, guard columns included.
template <class S>
__device__ __forceinline__ void zero_tile(const KParams &p, uint32_t *tile)
{
    uint4 *a = reinterpret_cast<uint4 *>(tile);
    const int n4 = (int)(tile_words(S::word_rows(p), p.n_b) >> 2);
#pragma unroll 4
    for (int i = threadIdx.x; i < n4; i += S::threads())
        a[i] = make_uint4(0u, 0u, 0u, 0u);
}

// Returns the number of valid hits left in `stage` (in their original order),
// or -1 when the window was streamed through the stage in parts.  SUM (P = 4
// with more hits than a field holds): the scan also sums every counter, and
// a sum below the votes cast means that a counter overflowed (each carry out
// of a field takes 255 or more from the sum): the window's result is void and
// -2 returned.  On entry
// the tile is all zero (the kernel zeroes it before its first window, and
// every tile zeroes it again when done); so it is on return.  Per tile the
// CTA passes three block barriers in the common case: after the votes, at
// the end of the peak search, and after the tile is zeroed.  tile: the tile's
// words, guard columns included; carry: two rows of NB + 2 kGuard words.
// [ta, tb): the theta rows of this CTA's tiles (a range that does not start at
// row 0 starts on a tile and needs the window's hits staged at once).
template <class S, int P, class Key, bool F64, bool SUM>
__device__ __forceinline__ int process_tiles(const KParams &p, long long beg, int H, uint32_t *tile, int2 *stage,
                             uint32_t *carry, uint16_t *list, unsigned char *buf,
                             unsigned char *sel, int4 *pk, int *hist, int *wtot, WinScalars &ws,
                             long long w, int ta, int tb, const Key *&keys, int &n_top)
{
    const int WR = S::word_rows(p), R = WR * P, NB = p.n_b;
    const int n_tiles = (p.n_theta + R - 1) / R, k0 = ta / R, k1 = min(n_tiles, (tb + R - 1) / R);
    const bool single = H <= p.hit_stage;
    const int lane = threadIdx.x & 31;
    constexpr int lgP = P == 4 ? 2 : (P == 2 ? 1 : 0);
    const int32_t *lo_row = p.lo_tab ? p.lo_tab + lgP * p.lo_stride : nullptr;
    const unsigned gstride = (unsigned)(NB + kGuard) * 128u;
    const unsigned tile0 = (unsigned)__cvta_generic_to_shared(tile);
    const unsigned acc0 = tile0 + kGuard * 128u;
    const unsigned carry0 = (unsigned)__cvta_generic_to_shared(carry) + kGuard * 4u;
    const unsigned carry_row = (unsigned)(NB + 2 * kGuard) * 4u;
    const PeakStore<Key> st{reinterpret_cast<Key *>(buf), (p.kp + 256) * 8 / (int)sizeof(Key),
                            reinterpret_cast<Key *>(sel), 2048 / (int)sizeof(Key),
                            hist};
    int lo_prev = 0, found = 0;
    int nv = 0;                       // valid hits, of the whole window if single
    unsigned votes = 0u;
    if (single)
        nv = stage_hits<S>(p, beg, H, stage, wtot, ws);

    if (k0 > 0 && k0 < k1) {
        // the last two rows before the range, voted straight into the carry
        const int t0 = k0 * R;
        lo_prev = lo_row ? __ldg(lo_row + k0 - 1) : 0;
        const unsigned cb = carry0 + (P == 1 || (k0 & 1) ? carry_row : 0u);
        for (int j = threadIdx.x; j < NB; j += S::threads()) {
            sts32(cb + (unsigned)j * 4u, 0u);
            if (P == 1)
                sts32(carry0 + (unsigned)j * 4u, 0u);
        }
        __syncthreads();
        for (int i = threadIdx.x; i < 2 * nv; i += S::threads()) {
            const int2 h = stage[i >> 1];
            const int up = i & 1, t = t0 - 1 - up;
            const int j = rho_bin(h.x, h.y, __ldg(p.C + t), __ldg(p.S + t), p.D, p.K) - lo_prev;
            if ((unsigned)j < (unsigned)NB) {
                if constexpr (P == 1)
                    red_add_shared((up ? carry0 : cb) + (unsigned)j * 4u, 1u);
                else
                    red_add_shared(cb + (unsigned)j * 4u, 1u << ((P - 1 - up) * (32 / P)));
            }
        }
    }
    for (int k = k0; k < k1; ++k) {
        const int t0 = k * R;
        const bool last = k == n_tiles - 1;
        const bool fast = !F64 && p.in_range && t0 + R <= p.n_theta;
        const int lo = lo_row ? __ldg(lo_row + k) : 0;
        if (single) {
            if (fast)
                vote_tile<S, P, !F64, F64>(p, acc0, gstride, stage, nv, t0, lo, ws);
            else
                vote_tile<S, P, false, F64>(p, acc0, gstride, stage, nv, t0, lo, ws);
        } else {
            for (long long s0 = 0; s0 < H; s0 += p.hit_stage) {
                const int n = (int)min((long long)p.hit_stage, (long long)H - s0);
                const int ns = stage_hits<S>(p, beg + s0, n, stage, wtot, ws);
                if (SUM)
                    votes += (unsigned)ns * (unsigned)min(R, p.n_theta - t0);
                if (fast)
                    vote_tile<S, P, !F64, F64>(p, acc0, gstride, stage, ns, t0, lo, ws);
                else
                    vote_tile<S, P, false, F64>(p, acc0, gstride, stage, ns, t0, lo, ws);
                __syncthreads();
            }
        }
        __syncthreads();                             // the votes are complete
        // the last word row goes from one carry row to the other with every
        // tile (P = 1 keeps the last two word rows, saved after the search)
        const unsigned cur = carry0 + (P == 1 ? carry_row : (k & 1 ? carry_row : 0u));
        const unsigned next = P == 1 || last ? 0u : carry0 + (k & 1 ? 0u : carry_row);
        const TileView tv{acc0, gstride, tile0, carry0, cur, t0, lo, lo - lo_prev, last};
        found += find_peaks<S, P, Key, SUM>(p, tv, next, list, st, ws);
        if (SUM) {
            if (single)
                votes += (unsigned)nv * (unsigned)min(R, p.n_theta - t0);
            if (ws.sum != votes) {
                zero_tile<S>(p, tile);
                __syncthreads();
                return -2;
            }
        }
        // the search ended in a barrier: the tile and the carry are read no more
        if (P == 1 && !last) {
            const int c = ((WR >> 5) - 1) * (NB + kGuard) + kGuard;
            for (int j = threadIdx.x; j < NB; j += S::threads()) {
                carry[kGuard + j] = tile[(size_t)(c + j) * 32 + 30];
                carry[NB + 3 * kGuard + j] = tile[(size_t)(c + j) * 32 + 31];
            }
            __syncthreads();
        }
        if (p.export_acc) {
            export_tile_end<S, P>(p, tile + kGuard * 32, t0, R, lo, w);
            __syncthreads();
        }
        zero_tile<S>(p, tile);
        lo_prev = lo;
        __syncthreads();
    }
    found = (int)__reduce_add_sync(0xffffffffu, (unsigned)found);
    if (lane == 0 && found)
        atomicAdd(&ws.n_found, found);
    keys = finish_peaks<S>(p, st, pk, n_top, ws);
    return single ? nv : -1;
}

// Step D: first matching peak in order, then the stable per-peak compaction.
// Categories: peak index q < n_top, n_top for a hit on no peak's line,
// n_top + 1 for a hit outside the detector box.  hits_s: the window's hits
// in shared memory when every one of them is valid (else NULL: read from
// global memory); cat_s: room for H categories in shared memory (else NULL:
// re-read from hit_track).  Each warp takes its own contiguous slice of the
// hits, one hit per lane: it finds their categories (the peaks' lines are
// broadcast loads, and |bin - b| <= tol is one unsigned compare of the sum
// against the line's range, five instructions a peak), counts them (wcat, one
// row per warp), and from all warps' counts works out the first slot of each
// of its categories (a prefix over the categories, then over the warps
// before it) into its row of wpos; then it scatters its slice in order.  Two
// block barriers, and no warp waits for a single one of them.  (Four lanes a hit with
// one warp counting and scattering windows of up to 512 hits took 17% of the
// batched pileup windows' time.)  wcat and wpos are all zero on entry and on
// return; the caller's next barrier ends the step.
template <class S, class Key, bool F64>
__device__ __forceinline__ void associate(const KParams &p, long long w, long long beg, int H,
                                          int n_top, const Key *keys, const int4 *pk,
                                          const int2 *hits_s,
                                          int *cat_s, int *wcat, int *wpos)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = S::warps();
    const int D = p.D, K = p.K, tol = p.tol;
    __syncthreads();                         // keys and pk are in place
    const int NC = n_top + 2;
    // Every sum lies in [0, n_rho 2^K) when the box votes in range, so its
    // distance from a line's first bin is below 2^31 + tol 2^K either way and
    // taken mod 2^32 is below (2 tol + 1) 2^K only on the line itself, as long
    // as (3 tol + 1) 2^K is at most 2^31.
    const bool wrap_ok = !F64 && p.in_range && 3ll * tol + 1 <= 1ll << (31 - K);
    const unsigned width = (unsigned)(2 * tol + 1) << K;
    // slices of whole 32-hit blocks
    const int chunk = ((H + nw - 1) / nw + 31) & ~31;
    const int h0 = min(H, warp * chunk), h1 = min(H, h0 + chunk);
    const unsigned lt = lanemask_lt();
    int *mine = wcat + warp * NC, *slot = wpos + warp * NC;
    int cat = -1;
    unsigned m = 0u;
    for (int base = h0; base < h1; base += 32) {
        const int i = base + lane;
        int phi = 0, z = 0;
        bool ok = false;
        if (i < h1) {
            if (hits_s) {
                const int2 h = hits_s[i];
                phi = h.x;
                z = h.y;
                ok = true;
            } else {
                ok = load_hit(p, beg + i, phi, z);
            }
        }
        int first = n_top;
        if (wrap_ok) {
#pragma unroll 4
            for (int q = n_top - 1; q >= 0; --q) {
                const int4 l = pk[q];
                const unsigned v = (unsigned)phi * (unsigned)l.x + (unsigned)z * (unsigned)l.y + (unsigned)l.z;
                first = v < width ? q : first;
            }
        } else {
            double phd = 0.0, zmm = 0.0;
            if constexpr (F64) {
                phd = __ddiv_rn((double)phi, p.u_phi);
                zmm = __ddiv_rn((double)z, p.u_z);
            }
            for (int q = n_top - 1; q >= 0; --q) {
                const int4 l = pk[q];
                const int t = l.w & 0xffff, b = l.w >> 16;
                int d;
                if constexpr (F64)
                    d = rho_bin64(phd, zmm, __ldg(p.Cd + t), __ldg(p.Sd + t), p) - b;
                else
                    d = rho_bin(phi, z, l.x, l.y, D, K) - b;
                first = d <= tol && d >= -tol ? q : first;
            }
        }
        cat = i < h1 ? (ok ? first : n_top + 1) : -1;
        if (i < h1) {
            p.hit_track[beg + i] = cat < n_top ? cat : (cat == n_top ? -1 : -2);
            if (cat_s)
                cat_s[i] = cat;
        }
        m = __match_any_sync(0xffffffffu, cat);
        if (i < h1 && lane == __ffs(m) - 1)
            mine[cat] += __popc(m);          // leaders of distinct categories
        __syncwarp();
    }
    __syncthreads();
    if (h0 < h1 || warp == 0) {
        const int used = chunk > 0 ? min(nw, (H + chunk - 1) / chunk) : 0;   // warps with hits
        int run = 0;
        for (int b0 = 0; b0 < NC; b0 += 32) {
            const int q = b0 + lane;
            int tot = 0, before = 0;
            if (q < NC)
                for (int k = 0; k < used; ++k) {
                    const int c = wcat[k * NC + q];
                    before += k < warp ? c : 0;
                    tot += c;
                }
            int incl = tot;
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, incl, d);
                if (lane >= d)
                    incl += y;
            }
            const int excl = run + incl - tot;
            if (q < NC)
                slot[q] = excl + before;
            if (warp == 0 && q < n_top) {
                const Key k = keys[q];
                hough_peak pr;
                pr.theta = (uint16_t)key_theta(p, k);
                pr.rho = (uint16_t)key_rho(p, k);
                pr.votes = (int32_t)key_votes(p, k);
                pr.n_hits = tot;
                pr.hit_begin = excl;
                p.peaks[(size_t)w * p.max_peaks + q] = pr;
            }
            run += __shfl_sync(0xffffffffu, incl, 31);
        }
        __syncwarp();
        for (int base = h0; base < h1; base += 32) {
            const int i = base + lane;
            if (chunk > 32) {                // else cat and m are still the block's
                cat = -1;
                if (i < h1) {
                    if (cat_s) {
                        cat = cat_s[i];
                    } else {
                        const int v = p.hit_track[beg + i];
                        cat = v >= 0 ? v : (v == -1 ? n_top : n_top + 1);
                    }
                }
                m = __match_any_sync(0xffffffffu, cat);
            }
            const int leader = __ffs(m) - 1;
            int pos = 0;
            if (i < h1 && lane == leader) {
                pos = slot[cat];
                if (chunk > 32)
                    slot[cat] = pos + __popc(m);
            }
            pos = __shfl_sync(0xffffffffu, pos, leader);
            if (i < h1)
                p.track_hits[beg + pos + __popc(m & lt)] = i;
            __syncwarp();
        }
    }
    __syncthreads();
    // leave the scratch zero
    for (int q = threadIdx.x; q < 2 * nw * NC; q += S::threads())
        (q < nw * NC ? wcat : wpos - nw * NC)[q] = 0;
    if (cat_s)
        for (int i = threadIdx.x; i < H; i += S::threads())
            cat_s[i] = 0;
}

// A window's state before its tiles.
template <class S>
__device__ __forceinline__ void reset_window(const KParams &p, int *hist, WinScalars &ws)
{
    if (threadIdx.x == 0) {
        ws.kth = p.max_peaks > 0 ? ~0ull : 0ull;
        ws.n_top = 0;
        ws.n_buf = 0;
        ws.fail = INT_MAX;
        ws.n_sel = 0;
        ws.vk = 0;
        ws.n_found = 0;
        ws.sum = 0u;
        ws.flags = 0u;
    }
    for (int i = threadIdx.x; i < kHistBins; i += S::threads())
        hist[i] = 0;
    __syncthreads();
}

// One window in the counter width P and the key type Key: tiles, then the
// association, whose scratch is the tile (all zero after the tiles, and left
// so): the per-warp category counts and slots, then the categories if they
// fit.  False when a counter overflowed (SUM).
template <class S, int P, class Key, bool F64, bool SUM = false>
__device__ __forceinline__ bool find_window(const KParams &p, long long w, long long beg, int H, const SmemLayout &L,
                            unsigned char *smem, WinScalars &ws)
{
    const int nw = S::warps(), warp = threadIdx.x >> 5;
    uint32_t *tile = reinterpret_cast<uint32_t *>(smem + L.acc);
    int2 *stage = reinterpret_cast<int2 *>(smem + L.stage);
    int *hist = reinterpret_cast<int *>(smem + L.hist);
    int4 *pk = reinterpret_cast<int4 *>(smem + L.pk);
    const Key *keys = nullptr;
    int n_top = 0;
    reset_window<S>(p, hist, ws);
    const int nv = process_tiles<S, P, Key, F64, SUM>(
        p, beg, H, tile, stage, reinterpret_cast<uint32_t *>(smem + L.carry),
        reinterpret_cast<uint16_t *>(smem + L.list) + warp * kListCap, smem + L.buf, smem + L.sel,
        pk, hist, reinterpret_cast<int *>(smem + L.wtot), ws, w, 0, p.n_theta, keys, n_top);
    if (SUM && nv == -2)
        return false;
    const int need = nw * (n_top + 2);
    int *scr = reinterpret_cast<int *>(tile);
    const bool cats = H <= (int)(p.acc_bytes >> 2) - 2 * need;
    associate<S, Key, F64>(p, w, beg, H, n_top, keys, pk, nv == H ? stage : nullptr,
                        cats ? scr + 2 * need : nullptr, scr, scr + need);
    return true;
}

// The body of the find kernels.  F64: the FP64 variant of the bins
// (HOUGH_FLAG_FP64), a kernel of its own so that its registers do not weigh
// on the fixed-point kernel.
template <class S, bool F64>
__device__ __forceinline__ void find_body(const KParams &p)
{
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ WinScalars ws;
    const int nw = S::warps();
    const SmemLayout L = smem_layout(p.acc_bytes, p.hit_stage, p.n_b, p.kp, nw);
    // the tile and the guards of the carried row start all zero; every tile
    // and the association leave them so
    for (int i = threadIdx.x; i < (int)(p.acc_bytes >> 2); i += S::threads())
        reinterpret_cast<uint32_t *>(smem + L.acc)[i] = 0u;
    for (int i = threadIdx.x; i < 2 * (p.n_b + 2 * kGuard); i += S::threads())
        reinterpret_cast<uint32_t *>(smem + L.carry)[i] = 0u;
    long long w = blockIdx.x;
    while (w < p.n_windows) {
        long long beg = p.offsets[w], end = p.offsets[w + 1];
        bool bad = !(beg >= 0 && beg <= end && end <= p.n_hits && end - beg < (1ll << 30));
        if (bad) {
            if (threadIdx.x == 0) {
                p.status[w] = HOUGH_WIN_BAD_OFFSETS;
                p.n_peaks[w] = 0;
                if (p.n_found)
                    p.n_found[w] = 0;
            }
        } else {
            const int H = (int)(end - beg);
            // Counter width.  Windows of more hits than a byte counts still
            // run in bytes while they have few hits for the stored bins: a
            // line of 256 hits is then out of the ordinary, and its overflow
            // is found (SUM) and the window redone in 16 bits.  Half the
            // tiles, and so half the scan, the zeroing and the barriers.
            const bool key32 = H < 1 << (32 - p.tb - p.bb);
            bool done = false;
            if (p.pmax == 4) {
                if (H <= 255)
                    done = find_window<S, 4, uint32_t, F64>(p, w, beg, H, L, smem, ws);
                else if (key32 && !F64 && p.in_range && H <= 8 * p.n_b)
                    done = find_window<S, 4, uint32_t, F64, !F64>(p, w, beg, H, L, smem, ws);
            }
            if (!done) {
                if (key32 && H <= 65534)
                    find_window<S, 2, uint32_t, F64>(p, w, beg, H, L, smem, ws);
                else if (H <= 65534)
                    find_window<S, 2, unsigned long long, F64>(p, w, beg, H, L, smem, ws);
                else
                    find_window<S, 1, unsigned long long, F64>(p, w, beg, H, L, smem, ws);
            }
            if (threadIdx.x == 0) {
                unsigned fl = ws.flags;
                if (ws.n_found > p.max_peaks)
                    fl |= HOUGH_WIN_PEAK_OVERFLOW;
                p.status[w] = fl;
                p.n_peaks[w] = ws.n_top;
                if (p.n_found)
                    p.n_found[w] = ws.n_found;
            }
        }
        __syncthreads();
        if (threadIdx.x == 0)
            ws.next_w = (int)gridDim.x + (int)atomicAdd(p.work, 1u);
        __syncthreads();
        w = ws.next_w;
    }
    // The last CTA to finish resets the scheduling counters for the next launch.
    if (threadIdx.x == 0) {
        __threadfence();
        unsigned done = atomicAdd(p.work + 1, 1u);
        if (done == gridDim.x - 1) {
            atomicExch(p.work, 0u);
            atomicExch(p.work + 1, 0u);
            __threadfence();
        }
    }
}

// ---- one window over the CTAs of a cluster

// What a CTA of a cluster publishes of its tiles.
struct SplitOut {
    int n_top;           // its best peaks, sorted, at `keys` (shared address)
    unsigned keys;
    int found;
    unsigned flags;
    int overflow;        // a byte counter overflowed (SUM)
};

// The find kernels' static shared variables, beside the dynamic shared memory that
// the host sizes to the device's limits less kStaticSmem.
constexpr size_t kStaticSmem = 128;
static_assert(sizeof(WinScalars) <= kStaticSmem && sizeof(WinScalars) + sizeof(SplitOut) <= kStaticSmem,
              "static shared memory of the find kernels");

__device__ __forceinline__ void cluster_sync()
{
    asm volatile("barrier.cluster.arrive.release;\n barrier.cluster.wait.acquire;" ::: "memory");
}

// A word of CTA `rank`'s shared memory, at this CTA's address `addr`.
__device__ __forceinline__ uint32_t ld_cluster32(unsigned addr, unsigned rank)
{
    uint32_t r, v;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(v) : "r"(r) : "memory");
    return v;
}

// One window in the counter width P: every CTA of the cluster takes its share
// of the tiles (the first all of them if the hits do not fit in the
// stage), the first CTA merges their sorted peaks -- a peak's place is its
// place in its own list plus, by a search in each of the others, the number of
// better ones there -- and makes the association.  False (in every CTA) when a
// counter overflowed.
template <class S, int P, class Key, bool SUM>
__device__ __forceinline__ bool split_window(const KParams &p, long long w, long long beg, int H,
                                             unsigned rank, const SmemLayout &L,
                                             unsigned char *smem, SplitOut &so, WinScalars &ws)
{
    constexpr int nw = S::kThreads / 32;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int C = p.split;
    uint32_t *tile = reinterpret_cast<uint32_t *>(smem + L.acc);
    int2 *stage = reinterpret_cast<int2 *>(smem + L.stage);
    int *hist = reinterpret_cast<int *>(smem + L.hist);
    int4 *pk = reinterpret_cast<int4 *>(smem + L.pk);
    const int unit = 32 * p.pmax, units = (p.n_theta + unit - 1) / unit;
    int ta = (int)rank * units / C * unit, tb = ((int)rank + 1) * units / C * unit;
    if (H > p.hit_stage) {
        ta = 0;
        tb = rank == 0 ? units * unit : 0;
    }
    reset_window<S>(p, hist, ws);
    const Key *keys = nullptr;
    int n_top = 0, nv = 0;
    if (ta < tb)
        nv = process_tiles<S, P, Key, false, SUM>(
            p, beg, H, tile, stage, reinterpret_cast<uint32_t *>(smem + L.carry),
            reinterpret_cast<uint16_t *>(smem + L.list) + warp * kListCap, smem + L.buf,
            smem + L.sel, pk, hist, reinterpret_cast<int *>(smem + L.wtot), ws, w, ta, tb, keys,
            n_top);
    __syncthreads();
    if (threadIdx.x == 0) {
        so.overflow = SUM && nv == -2 ? 1 : 0;
        so.n_top = so.overflow ? 0 : n_top;
        so.keys = n_top > 0 ? (unsigned)__cvta_generic_to_shared(keys) : 0u;
        so.found = ws.n_found;
        so.flags = ws.flags;
    }
    cluster_sync();
    const unsigned so_at = (unsigned)__cvta_generic_to_shared(&so);
    if (SUM) {
        const unsigned bad = lane < C ? ld_cluster32(so_at + offsetof(SplitOut, overflow), lane) : 0u;
        if (__any_sync(0xffffffffu, bad != 0u)) {
            cluster_sync();                  // every CTA has read it
            return false;
        }
    }
    // lane c of every warp: CTA c's counts; the lists to this CTA's memory
    Key *lists = reinterpret_cast<Key *>(smem + L.total);
    int n_c = 0, found = 0;
    unsigned flags = 0u;
    if (rank == 0) {
        if (lane < C) {
            n_c = (int)ld_cluster32(so_at + offsetof(SplitOut, n_top), lane);
            found = (int)ld_cluster32(so_at + offsetof(SplitOut, found), lane);
            flags = ld_cluster32(so_at + offsetof(SplitOut, flags), lane);
        }
        for (int c = warp; c < C; c += nw) {
            const int n = __shfl_sync(0xffffffffu, n_c, c);
            const unsigned at = ld_cluster32(so_at + offsetof(SplitOut, keys), c);
            for (int i = lane; i < n; i += 32) {
                if constexpr (sizeof(Key) == 4)
                    lists[c * p.kp + i] = ld_cluster32(at + (unsigned)i * 4u, c);
                else
                    lists[c * p.kp + i] = (Key)ld_cluster32(at + (unsigned)i * 8u, c) |
                                          (Key)ld_cluster32(at + (unsigned)i * 8u + 4u, c) << 32;
            }
        }
    }
    cluster_sync();                          // the others may leave
    if (rank != 0)
        return true;
    const int total = (int)__reduce_add_sync(0xffffffffu, (unsigned)n_c);
    found = (int)__reduce_add_sync(0xffffffffu, (unsigned)found);
    flags = __reduce_or_sync(0xffffffffu, flags);
    n_top = min(p.max_peaks, total);
    Key *sorted = reinterpret_cast<Key *>(smem + L.sel);
    for (int x0 = 0; x0 < C * p.kp; x0 += S::kThreads) {
        const int x = x0 + (int)threadIdx.x, c = x / p.kp, i = x - c * p.kp;
        const bool in = c < C && i < __shfl_sync(0xffffffffu, n_c, min(c, 31));   // c is the warp's
        const Key key = in ? lists[x] : (Key)0;
        int r = i;
        for (int o = 0; o < C; ++o) {
            const int n = __shfl_sync(0xffffffffu, n_c, o);
            if (o == c)
                continue;
            int lo = 0, hi = n;              // better peaks of CTA o
            while (lo < hi) {
                const int mid = (lo + hi) >> 1;
                if (lists[o * p.kp + mid] < key)
                    lo = mid + 1;
                else
                    hi = mid;
            }
            r += lo;
        }
        if (in && r < n_top) {
            const int t = key_theta(p, key), b = key_rho(p, key);
            sorted[r] = key;
            pk[r] = make_int4(__ldg(p.C + t), __ldg(p.S + t),
                              (int)((unsigned)p.D - ((unsigned)(b - p.tol) << p.K)), t | b << 16);
        }
    }
    const int need = nw * (n_top + 2);
    int *scr = reinterpret_cast<int *>(tile);
    const bool cats = H <= (int)(p.acc_bytes >> 2) - 2 * need;
    associate<S, Key, false>(p, w, beg, H, n_top, sorted, pk, nv == H ? stage : nullptr,
                             cats ? scr + 2 * need : nullptr, scr, scr + need);
    if (threadIdx.x == 0) {
        if (found > p.max_peaks)
            flags |= HOUGH_WIN_PEAK_OVERFLOW;
        p.status[w] = flags;
        p.n_peaks[w] = n_top;
        if (p.n_found)
            p.n_found[w] = found;
    }
    return true;
}

// Batches of fewer windows than the SMs hold: p.split CTAs (a cluster) per
// window.
template <class S>
__device__ __forceinline__ void split_body(const KParams &p)
{
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ WinScalars ws;
    __shared__ SplitOut so;
    const SmemLayout L = smem_layout(p.acc_bytes, p.hit_stage, p.n_b, p.kp, S::kThreads / 32);
    const long long w = blockIdx.x / p.split;
    const unsigned rank = blockIdx.x % p.split;
    for (int i = threadIdx.x; i < (int)(p.acc_bytes >> 4); i += S::kThreads)
        reinterpret_cast<uint4 *>(smem + L.acc)[i] = make_uint4(0u, 0u, 0u, 0u);
    for (int i = threadIdx.x; i < 2 * (p.n_b + 2 * kGuard); i += S::kThreads)
        reinterpret_cast<uint32_t *>(smem + L.carry)[i] = 0u;
    const long long beg = p.offsets[w], end = p.offsets[w + 1];
    if (!(beg >= 0 && beg <= end && end <= p.n_hits && end - beg < (1ll << 30))) {
        if (rank == 0 && threadIdx.x == 0) {
            p.status[w] = HOUGH_WIN_BAD_OFFSETS;
            p.n_peaks[w] = 0;
            if (p.n_found)
                p.n_found[w] = 0;
        }
        return;                              // the whole cluster
    }
    const int H = (int)(end - beg);
    bool done = false;                       // the widths as in find_body
    const bool key32 = H < 1 << (32 - p.tb - p.bb);
    if (p.pmax == 4) {
        if (H <= 255)
            done = split_window<S, 4, uint32_t, false>(p, w, beg, H, rank, L, smem, so, ws);
        else if (key32 && p.in_range && H <= 8 * p.n_b)
            done = split_window<S, 4, uint32_t, true>(p, w, beg, H, rank, L, smem, so, ws);
    }
    if (!done) {
        if (key32 && H <= 65534)
            split_window<S, 2, uint32_t, false>(p, w, beg, H, rank, L, smem, so, ws);
        else if (H <= 65534)
            split_window<S, 2, unsigned long long, false>(p, w, beg, H, rank, L, smem, so, ws);
        else
            split_window<S, 1, unsigned long long, false>(p, w, beg, H, rank, L, smem, so, ws);
    }
}

// The find kernels (instances of find_body), compiled in translation units of
// their own so that they build in parallel (hough_find*.cu): find_kernel
// (fixed point, any CTA size up to 1024 threads and any tile), its instances
// for tiles of 32 word rows and CTAs of 128, 256, 512 and 1024 threads, and
// find_kernel_fp64 (HOUGH_FLAG_FP64).
__global__ void find_kernel(KParams p);
__global__ void find_kernel_128(KParams p);
__global__ void find_kernel_256(KParams p);
__global__ void find_kernel_512(KParams p);
__global__ void find_kernel_1024(KParams p);
__global__ void find_kernel_fp64(KParams p);
// One window per cluster (hough_find_split.cu).
__global__ void find_split_kernel_256(KParams p);
__global__ void find_split_kernel_512(KParams p);

}  // namespace hk
