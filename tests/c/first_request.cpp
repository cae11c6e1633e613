// The first request of every batch size on a new server, in a process that has
// run nothing before:
//   first_request <geometry file> <rows and bins>
// Prints a line per size: windows, latency of its first request and the median
// of its next nine, in us.
#include <cuda_runtime.h>

#include <algorithm>
#include <chrono>
#include <cstdio>
#include <cstdlib>
#include <vector>

#include "hough.h"

static const int MAX_W = 700, HITS = 142;

template <class T>
static T *pinned(size_t n)
{
    void *p = nullptr;
    if (cudaHostAlloc(&p, n * sizeof(T), cudaHostAllocDefault) != cudaSuccess)
        exit(2);
    return static_cast<T *>(p);
}

int main(int argc, char **argv)
{
    if (argc != 3)
        return 1;
    hough_geometry g;
    FILE *f = fopen(argv[1], "rb");
    if (!f || fread(&g, sizeof g, 1, f) != 1)
        return 1;
    fclose(f);
    const int n = atoi(argv[2]);
    hough_thresholds th{};
    th.vote_threshold = 5;
    th.assoc_tol_bins = 1;
    th.max_peaks = 64;
    hough_ctx *ctx = nullptr;
    hough_server *s = nullptr;
    hough_server_config c{};
    c.n_slots = 1;
    c.raw_hits = 1;
    c.slot_windows = MAX_W;
    c.slot_hits = MAX_W * HITS;
    c.max_queued = 4;
    if (hough_create(&g, n, n, &th, &ctx) != HOUGH_OK || hough_server_create(ctx, &c, &s) != HOUGH_OK)
        return 3;
    int32_t *vane = pinned<int32_t>(MAX_W * HITS), *strip = pinned<int32_t>(MAX_W * HITS);
    std::vector<int64_t> offsets(MAX_W + 1);
    for (int i = 0; i < MAX_W * HITS; ++i) {         // ten lines of fourteen hits a window
        const int t = i % HITS / 14;
        vane[i] = (7 * t + i) % g.n_vanes;
        strip[i] = (100 + 180 * t + 4 * (t % 5) * vane[i] + i % 7) % g.n_z_strips;
    }
    for (int w = 0; w <= MAX_W; ++w)
        offsets[w] = (int64_t)w * HITS;
    hough_request r{};
    r.in0 = vane;
    r.in1 = strip;
    r.window_offsets = offsets.data();
    r.out.peaks = pinned<hough_peak>(MAX_W * 64);
    r.out.n_peaks = pinned<int32_t>(MAX_W);
    r.out.n_found = pinned<int32_t>(MAX_W);
    r.out.window_status = pinned<uint32_t>(MAX_W);
    r.out.hit_track = pinned<int32_t>(MAX_W * HITS);
    r.out.track_hits = pinned<int32_t>(MAX_W * HITS);
    for (int w : {1, 60, 200, 350, 700}) {
        r.n_windows = w;
        std::vector<double> us;
        for (int i = 0; i < 10; ++i) {
            const auto t0 = std::chrono::steady_clock::now();
            uint64_t ticket = 0;
            hough_request_result res{};
            if (hough_server_submit(s, &r, &ticket) != HOUGH_OK ||
                hough_server_wait(s, ticket, 60000, &res) != HOUGH_OK || res.status != HOUGH_OK)
                return 4;
            us.push_back(std::chrono::duration<double, std::micro>(std::chrono::steady_clock::now() - t0).count());
        }
        std::sort(us.begin() + 1, us.end());
        std::printf("%d %.1f %.1f\n", w, us[0], us[5]);
    }
    hough_server_destroy(s);
    hough_destroy(ctx);
    return 0;
}
