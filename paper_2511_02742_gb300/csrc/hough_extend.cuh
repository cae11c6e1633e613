// Track extension (Section 4): a seed of three hits on consecutive vanes,
// taken from a peak's associated hits, extrapolated vane by vane forward and
// backward through the window's hits.  One warp per window; windows are
// independent.  Included by hough_api.cu after hough_kernels.cuh.
#pragma once

namespace hk {

constexpr int kExtClaimed = 512;   // tag of a claimed hit: kExtClaimed + track index

struct ExtParams {
    KParams k;          // hits, geometry, windows and the find step's outputs
    int n_vanes;        // 3..HOUGH_EXT_MAX_VANES
    int tol_z;          // 0..HOUGH_EXT_MAX_TOL, z units
    int cap;            // hits a warp holds in shared memory in this launch (<= 4096)
    long long lo;       // this launch takes the windows with lo < n_hits <= cap
    int flag_large;     // windows above cap get HOUGH_WIN_TOO_LARGE (last launch)
    int4 *ext;          // [n_windows * max_peaks]: first_vane, n_hits, hit_begin, seed_mid
    int32_t *ext_track; // [n_hits] window-local track index, -1 none
    int32_t *ext_hits;  // [n_hits] window-local hit order
    uint32_t *status;   // [n_windows]
};

// Shared memory of one warp: z[cap] int32, vane[cap] int16 (-1: takes no
// part), tag[cap] int16 (the hit's peak from the find step, -1 none, or
// kExtClaimed + track once claimed), bucket[cap] int16 (hit indices grouped
// by vane), group[cap] int16 (the find step's hits in track order),
// bstart[n_vanes + 1] and bcur[n_vanes] int32, seed[max_peaks] uint32 (the least
// bend << 12 | b of a peak's triplets before any hit was claimed, ~0 none),
// line[2 n_vanes + 4] int16 (the track being built, in vane order).
__host__ __device__ inline size_t ext_smem_bytes(int cap, int n_vanes, int max_peaks)
{
    return (size_t)cap * 12 + (size_t)(2 * n_vanes + 1 + max_peaks) * 4 + (size_t)(2 * n_vanes + 4) * 2;
}

// The smallest key of the warp, (bend << 36) | (b << 24) | (a << 12) | c with
// bend below 2^19: its upper 31 bits, then the lower 24 among the lanes that
// hold them.
__device__ __forceinline__ unsigned long long ext_warp_min(unsigned long long x)
{
    const unsigned hi = (unsigned)min(x >> 24, 0xffffffffull);
    const unsigned top = __reduce_min_sync(0xffffffffu, hi);
    if (top == 0xffffffffu)
        return ~0ull;
    const unsigned low = __reduce_min_sync(0xffffffffu, hi == top ? (unsigned)x & 0xffffffu : 0xffffffffu);
    return (unsigned long long)top << 24 | low;
}

// The unclaimed hit of bucket entries i, i + step, ... below s1 nearest to pred
// within tol, as the key (|z - pred| << 13) | (z > pred) << 12 | hit: the
// minimum is the nearest, then the lower z, then the lower index.  ~0u when
// there is none.  Z: the type that holds the prediction (7 |z|).
template <class Z>
__device__ __forceinline__ unsigned ext_nearest(const int32_t *zs, const int16_t *tag, const int16_t *bucket,
                                                int i, int s1, int step, Z pred, int tol)
{
    unsigned best = 0xffffffffu;
    for (; i < s1; i += step) {
        const int h = bucket[i];
        if (tag[h] >= kExtClaimed)
            continue;
        Z d = (Z)zs[h] - pred;
        const unsigned side = d > 0 ? 1u : 0u;
        d = d < 0 ? -d : d;
        if (d > tol)
            continue;
        const unsigned key = ((unsigned)d << 13) | (side << 12) | (unsigned)h;
        best = key < best ? key : best;
    }
    return best;
}

// Bound: the dependent chain of a window's steps (a bucket's bounds, its hits, a
// warp minimum per vane) and its instructions (5.4 k) at 29 warps per SM, 0.64
// instructions a cycle.  40001 windows of 86 hits, the first launch: 530 us ->
// 462 by staging the groups and two 32-bit minima per seed instead of ten
// shuffles, 412 by one pass for every peak's seed, 380 by predictions in 32
// bits, 354 by growing both ends at once, 332 by one look at each bucket in
// the seed pass; the launches that find no window of their size 13 + 27 -> 5 + 6
// us by looking at 32 windows together.  Not better: hits laid out in vane
// order (9% slower: more work to lay them out than the steps save), a 256-hit
// stage in front (40 warps per SM need 48 registers and spill: 26% slower).
template <class Z>
__device__ __forceinline__ void extend_body(const ExtParams &q)
{
    extern __shared__ __align__(16) unsigned char ext_sm[];
    const KParams &p = q.k;
    const int lane = threadIdx.x & 31;
    const int nv = q.n_vanes, cap = q.cap, tol = q.tol_z;
    int32_t *zs = reinterpret_cast<int32_t *>(ext_sm);
    int16_t *vs = reinterpret_cast<int16_t *>(zs + cap);
    int16_t *tag = vs + cap;
    int16_t *bucket = tag + cap;
    int16_t *group = bucket + cap;
    int32_t *bstart = reinterpret_cast<int32_t *>(group + cap);   // cap is a multiple of 8
    int32_t *bcur = bstart + nv + 1;
    unsigned *seed = reinterpret_cast<unsigned *>(bcur + nv);
    int16_t *line = reinterpret_cast<int16_t *>(seed + p.max_peaks);
    const int vstep = p.box.vane_step;

    // this warp's windows, 32 looked at together: a launch skips the windows of
    // the others' sizes
    for (long long k0 = 0; k0 * gridDim.x < p.n_windows; k0 += 32) {
        const long long wl = (k0 + lane) * gridDim.x + blockIdx.x;
        long long bl = 0, el = 0;
        if (wl < p.n_windows) {
            bl = __ldg(p.offsets + wl);
            el = __ldg(p.offsets + wl + 1);
        }
        const bool okl = bl >= 0 && bl <= el && el <= p.n_hits;
        unsigned todo = __ballot_sync(0xffffffffu, wl < p.n_windows &&
                                                       (okl ? el - bl > q.lo && (el - bl <= cap || q.flag_large)
                                                            : q.lo < 0));
        for (; todo != 0u; todo &= todo - 1u) {
            const int from = __ffs(todo) - 1;
            const long long w = (k0 + from) * gridDim.x + blockIdx.x;
            const long long beg = __shfl_sync(0xffffffffu, bl, from), end = __shfl_sync(0xffffffffu, el, from);
            if (!(beg >= 0 && beg <= end && end <= p.n_hits)) {
                if (lane == 0)                  // flagged once, by the first launch
                    q.status[w] = HOUGH_WIN_BAD_OFFSETS;
                continue;
            }
            const long long n = end - beg;
            const int np = min(max(p.n_peaks[w], 0), p.max_peaks);
            int4 *ext = q.ext + w * (long long)p.max_peaks;
            if (n > cap) {
                for (int i = lane; i < np; i += 32)
                    ext[i] = make_int4(-1, 0, 0, -1);
                for (long long i = lane; i < n; i += 32) {
                    q.ext_track[beg + i] = -1;
                    q.ext_hits[beg + i] = (int)i;
                }
                if (lane == 0)
                    q.status[w] = HOUGH_WIN_TOO_LARGE;
                continue;
            }
            const int H = (int)n;

            // ---- stage the window's hits and group them by vane
            for (int v = lane; v < nv; v += 32)
                bcur[v] = 0;
            __syncwarp();
            for (int i = lane; i < H; i += 32) {
                int phi, z;
                const bool ok = load_hit(p, beg + i, phi, z);
                const int ht = p.hit_track[beg + i];
                int v = -1;
                if (ok && ht != -2) {
                    // an address whose phi wraps into the box (and would be no
                    // index) counts as its encoded phi does
                    if (p.box.raw)
                        v = __ldg(p.a + beg + i);
                    if ((unsigned)v >= (unsigned)nv)
                        v = phi % vstep == 0 ? phi / vstep : -1;
                }
                zs[i] = z;
                vs[i] = (int16_t)v;
                tag[i] = (int16_t)(ht >= 0 && ht < kExtClaimed ? ht : -1);
                const int gi = p.track_hits[beg + i];
                group[i] = (int16_t)((unsigned)gi < (unsigned)H ? gi : -1);
                if (v >= 0)
                    atomicAdd(&bcur[v], 1);
            }
            __syncwarp();
            {
                // exclusive prefix over the vanes: lane l sums vanes [l k, l k + k)
                const int k = (nv + 31) >> 5;
                const int v0 = min(lane * k, nv), v1 = min(v0 + k, nv);
                int s = 0;
                for (int v = v0; v < v1; ++v)
                    s += bcur[v];
                int incl = s;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int y = __shfl_up_sync(0xffffffffu, incl, o);
                    if (lane >= o)
                        incl += y;
                }
                int run = incl - s;
                for (int v = v0; v < v1; ++v) {
                    const int c = bcur[v];
                    bstart[v] = run;
                    bcur[v] = run;
                    run += c;
                }
                if (lane == 31)
                    bstart[nv] = incl;
            }
            __syncwarp();
            for (int i = lane; i < H; i += 32) {
                const int v = vs[i];
                if (v >= 0)
                    bucket[atomicAdd(&bcur[v], 1)] = (int16_t)i;
            }
            __syncwarp();

            // ---- every peak's least triplet, a lane per place of the find's
            // lists: the seed of the peak unless an earlier track takes its hits
            const hough_peak *pk = p.peaks + w * (long long)p.max_peaks;
            for (int i = lane; i < np; i += 32)
                seed[i] = 0xffffffffu;
            __syncwarp();
            for (int j = lane; j < H; j += 32) {
                const int b = group[j];
                const int pi = b < 0 ? -1 : tag[b];
                if (pi < 0 || pi >= np || vs[b] < 0)
                    continue;
                const int hb = pk[pi].hit_begin, m = pk[pi].n_hits;
                if (hb < 0 || m < 3 || (long long)hb + m > H || j < hb || j >= hb + m)
                    continue;
                const int vb = vs[b];
                const int va = vb == 0 ? nv - 1 : vb - 1;
                const int vc = vb + 1 == nv ? 0 : vb + 1;
                const Z zb2 = 2 * (Z)zs[b];
                const int c0 = bstart[vc], c1 = bstart[vc + 1];
                // mostly one hit of the group stands on a vane
                int n_c = 0;
                Z zc = 0;
                for (int ic = c0; ic < c1; ++ic) {
                    const int c = bucket[ic];
                    if (tag[c] == pi) {
                        zc = (Z)zs[c];
                        ++n_c;
                    }
                }
                Z best = (Z)tol + 1;
                for (int ia = bstart[va], ea = n_c > 0 ? bstart[va + 1] : ia; ia < ea; ++ia) {
                    const int a = bucket[ia];
                    if (tag[a] != pi)
                        continue;
                    const Z za = (Z)zs[a];
                    Z bend = za - zb2 + zc;
                    bend = bend < 0 ? -bend : bend;
                    best = bend < best ? bend : best;
                    for (int ic = n_c > 1 ? c0 : c1; ic < c1; ++ic) {
                        const int c = bucket[ic];
                        bend = za - zb2 + zs[c];
                        bend = bend < 0 ? -bend : bend;
                        if (tag[c] == pi && bend < best)
                            best = bend;
                    }
                }
                if (best <= tol)
                    atomicMin(&seed[pi], (unsigned)best << 12 | (unsigned)b);
            }
            __syncwarp();

            // ---- the peaks in order
            int pos = 0;
            for (int p0 = 0; p0 < np; p0 += 32) {
                const unsigned mine32 = p0 + lane < np ? seed[p0 + lane] : 0xffffffffu;
                unsigned todo_p = __ballot_sync(0xffffffffu, mine32 != 0xffffffffu);
                int done_p = 0;                     // peaks of these 32 whose entries are written
                for (;;) {
                    const int kp = todo_p != 0u ? __ffs(todo_p) - 1 : 32;
                    if (lane >= done_p && lane < kp && p0 + lane < np)      // no seed
                        ext[p0 + lane] = make_int4(-1, 0, pos, -1);
                    if (kp == 32)
                        break;
                    todo_p &= todo_p - 1u;
                    done_p = kp + 1;
                    const int pi = p0 + kp;
                    const unsigned first_seed = __shfl_sync(0xffffffffu, mine32, kp);
                    int a, b = (int)(first_seed & 4095u), c;
                    unsigned ac = 0xffffffffu;      // the least a << 12 | c of that bend
                    if (tag[b] == pi) {
                        const int vb = vs[b];
                        const int va = vb == 0 ? nv - 1 : vb - 1;
                        const int vc = vb + 1 == nv ? 0 : vb + 1;
                        const Z zb2 = 2 * (Z)zs[b], least = (Z)(first_seed >> 12);
                        const int c0 = bstart[vc], c1 = bstart[vc + 1];
                        for (int ia = bstart[va] + lane, ea = bstart[va + 1]; ia < ea; ia += 32) {
                            const int x = bucket[ia];
                            if (tag[x] != pi)
                                continue;
                            const Z za = (Z)zs[x];
                            for (int ic = c0; ic < c1; ++ic) {
                                const int y = bucket[ic];
                                const Z bend = za - zb2 + zs[y];
                                if (tag[y] == pi && (bend == least || bend == -least))
                                    ac = min(ac, (unsigned)x << 12 | (unsigned)y);
                            }
                        }
                        ac = __reduce_min_sync(0xffffffffu, ac);
                    }
                    if (ac != 0xffffffffu) {
                        a = (int)(ac >> 12);
                        c = (int)(ac & 4095u);
                    } else {
                        // a hit of it is claimed: the least of the triplets left
                        const int hb = pk[pi].hit_begin, m = pk[pi].n_hits;
                        unsigned long long best = ~0ull;
                        for (int j = lane; j < m; j += 32) {
                            const int b = group[hb + j];
                            if (b < 0 || tag[b] != pi)
                                continue;
                            const int vb = vs[b];
                            if (vb < 0)
                                continue;
                            const int va = vb == 0 ? nv - 1 : vb - 1;
                            const int vc = vb + 1 == nv ? 0 : vb + 1;
                            const Z zb2 = 2 * (Z)zs[b];
                            const int c0 = bstart[vc], c1 = bstart[vc + 1];
                            for (int ia = bstart[va], ea = bstart[va + 1]; ia < ea; ++ia) {
                                const int a = bucket[ia];
                                if (tag[a] != pi)
                                    continue;
                                const Z za = (Z)zs[a];
                                for (int ic = c0; ic < c1; ++ic) {
                                    const int c = bucket[ic];
                                    if (tag[c] != pi)
                                        continue;
                                    Z bend = za - zb2 + zs[c];
                                    bend = bend < 0 ? -bend : bend;
                                    if (bend > tol)
                                        continue;
                                    const unsigned long long key = ((unsigned long long)bend << 36) |
                                                                   ((unsigned long long)b << 24) |
                                                                   ((unsigned long long)a << 12) |
                                                                   (unsigned long long)c;
                                    best = key < best ? key : best;
                                }
                            }
                        }
                        best = ext_warp_min(best);
                        if (best == ~0ull) {
                            if (lane == 0)
                                ext[pi] = make_int4(-1, 0, pos, -1);
                            continue;
                        }
                        b = (int)((best >> 24) & 4095u);
                        a = (int)((best >> 12) & 4095u);
                        c = (int)(best & 4095u);
                    }
                    const int16_t mine = (int16_t)(kExtClaimed + pi);
                    int lo = nv + 1, hi = nv + 4;
                    if (lane == 0) {
                        tag[a] = tag[b] = tag[c] = mine;
                        line[lo] = (int16_t)a;
                        line[lo + 1] = (int16_t)b;
                        line[lo + 2] = (int16_t)c;
                    }
                    __syncwarp();
                    // both ways at once, lanes 0 to 15 forward and 16 to 31 backward: the
                    // parabola through the last three hits, one vane on.  The two
                    // never meet while two vanes are free, so the hits are those of
                    // going forward first.
                    const int dir = lane >> 4;
                    bool any = true;
                    {
                        Z z0 = zs[dir ? c : a], z1 = zs[b], z2 = zs[dir ? a : c];
                        int tv = vs[dir ? a : c];
                        bool more = true;
                        while (any && hi - lo + 2 <= nv) {
                            tv = dir ? (tv == 0 ? nv - 1 : tv - 1) : (tv + 1 == nv ? 0 : tv + 1);
                            const unsigned best = ext_nearest<Z>(zs, tag, bucket, bstart[tv] + (lane & 15),
                                                                 more ? bstart[tv + 1] : 0, 16, 3 * z2 - 3 * z1 + z0, tol);
                            const unsigned kf = __reduce_min_sync(0xffffffffu, dir ? 0xffffffffu : best);
                            const unsigned kb = __reduce_min_sync(0xffffffffu, dir ? best : 0xffffffffu);
                            const unsigned key = dir ? kb : kf;
                            hi += kf != 0xffffffffu ? 1 : 0;
                            lo -= kb != 0xffffffffu ? 1 : 0;
                            more = key != 0xffffffffu;
                            if (more) {
                                const int h = (int)(key & 4095u);
                                if ((lane & 15) == 0) {
                                    tag[h] = mine;
                                    line[dir ? lo : hi - 1] = (int16_t)h;
                                }
                                z0 = z1;
                                z1 = z2;
                                z2 = zs[h];
                            }
                            any = (kf & kb) != 0xffffffffu;
                            __syncwarp();
                        }
                    }
                    if (any) {
                        // they may meet: given back, and forward first
                        for (int j = lo + lane; j < hi; j += 32)
                            if (j < nv + 1 || j >= nv + 4) {
                                const int h = line[j], ht = p.hit_track[beg + h];
                                tag[h] = (int16_t)(ht >= 0 && ht < kExtClaimed ? ht : -1);
                            }
                        lo = nv + 1;
                        hi = nv + 4;
                        __syncwarp();
                        // forward: the parabola through the last three hits, one vane on
                        {
                            Z z0 = zs[a], z1 = zs[b], z2 = zs[c];
                            int v2 = vs[c];
                            while (hi - lo < nv) {
                                const int tv = v2 + 1 == nv ? 0 : v2 + 1;
                                const unsigned key = __reduce_min_sync(
                                    0xffffffffu, ext_nearest<Z>(zs, tag, bucket, bstart[tv] + lane, bstart[tv + 1], 32,
                                                                3 * z2 - 3 * z1 + z0, tol));
                                if (key == 0xffffffffu)
                                    break;
                                const int h = (int)(key & 4095u);
                                if (lane == 0) {
                                    tag[h] = mine;
                                    line[hi] = (int16_t)h;
                                }
                                ++hi;
                                z0 = z1;
                                z1 = z2;
                                z2 = zs[h];
                                v2 = tv;
                                __syncwarp();
                            }
                        }
                        // backward, from the seed's first hit
                        {
                            Z z0 = zs[c], z1 = zs[b], z2 = zs[a];
                            int v2 = vs[a];
                            while (hi - lo < nv) {
                                const int tv = v2 == 0 ? nv - 1 : v2 - 1;
                                const unsigned key = __reduce_min_sync(
                                    0xffffffffu, ext_nearest<Z>(zs, tag, bucket, bstart[tv] + lane, bstart[tv + 1], 32,
                                                                3 * z2 - 3 * z1 + z0, tol));
                                if (key == 0xffffffffu)
                                    break;
                                const int h = (int)(key & 4095u);
                                --lo;
                                if (lane == 0) {
                                    tag[h] = mine;
                                    line[lo] = (int16_t)h;
                                }
                                z0 = z1;
                                z1 = z2;
                                z2 = zs[h];
                                v2 = tv;
                                __syncwarp();
                            }
                        }
                    }
                    __syncwarp();
                    const int cnt = hi - lo;
                    for (int j = lane; j < cnt; j += 32)
                        q.ext_hits[beg + pos + j] = line[lo + j];
                    if (lane == 0)
                        ext[pi] = make_int4(vs[line[lo]], cnt, pos, b);
                    pos += cnt;
                    __syncwarp();
                }
            }

            // ---- per-hit track and the unclaimed hits in index order
            for (int base = 0; base < H; base += 32) {
                const int i = base + lane;
                const int t = i < H ? tag[i] : 0;
                const bool un = i < H && t < kExtClaimed;
                if (i < H)
                    q.ext_track[beg + i] = un ? -1 : t - kExtClaimed;
                const unsigned m = __ballot_sync(0xffffffffu, un);
                if (un)
                    q.ext_hits[beg + pos + __popc(m & ((1u << lane) - 1u))] = i;
                pos += __popc(m);
            }
            if (lane == 0)
                q.status[w] = 0u;
            __syncwarp();
        }
    }
}

// Predictions in 32 bits, and for geometries with z of 2^27 units and more.
__global__ void __launch_bounds__(32) extend_kernel(ExtParams q) { extend_body<int>(q); }
__global__ void __launch_bounds__(32) extend_kernel_wide(ExtParams q) { extend_body<long long>(q); }

}  // namespace hk
