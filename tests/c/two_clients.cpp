// Clients of one server, each waiting for its result before it sends its next
// request of 20 windows:
//   two_clients <geometry file> <clients> <requests>
// Prints the median time, in ns, from a request's arrival to the launch of its batch.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdio>
#include <cstdlib>
#include <thread>
#include <vector>

#include "hough.h"

static const int W = 20, HITS = 142;

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
    if (argc != 4)
        return 1;
    hough_geometry g;
    FILE *f = fopen(argv[1], "rb");
    if (!f || fread(&g, sizeof g, 1, f) != 1)
        return 1;
    fclose(f);
    const int clients = atoi(argv[2]), requests = atoi(argv[3]);
    hough_thresholds th{};
    th.vote_threshold = 5;
    th.assoc_tol_bins = 1;
    th.max_peaks = 64;
    hough_ctx *ctx = nullptr;
    hough_server *s = nullptr;
    hough_server_config c{};
    c.n_slots = clients;
    c.raw_hits = 1;
    c.slot_windows = 256;
    c.slot_hits = 1 << 17;
    c.max_queued = 64;
    if (hough_create(&g, 512, 512, &th, &ctx) != HOUGH_OK || hough_server_create(ctx, &c, &s) != HOUGH_OK)
        return 3;
    std::vector<std::vector<int64_t>> waits(clients);
    auto client = [&](int k) {
        int32_t *vane = pinned<int32_t>(W * HITS), *strip = pinned<int32_t>(W * HITS);
        std::vector<int64_t> offsets(W + 1);
        for (int i = 0; i < W * HITS; ++i) {         // ten lines of fourteen hits a window
            const int t = i % HITS / 14;
            vane[i] = (7 * t + i) % g.n_vanes;
            strip[i] = (100 + 180 * t + 4 * (t % 5) * vane[i] + 31 * k + i % 7) % g.n_z_strips;
        }
        for (int w = 0; w <= W; ++w)
            offsets[w] = (int64_t)w * HITS;
        hough_request r{};
        r.in0 = vane;
        r.in1 = strip;
        r.window_offsets = offsets.data();
        r.n_windows = W;
        r.out.peaks = pinned<hough_peak>(W * 64);
        r.out.n_peaks = pinned<int32_t>(W);
        r.out.n_found = pinned<int32_t>(W);
        r.out.window_status = pinned<uint32_t>(W);
        r.out.hit_track = pinned<int32_t>(W * HITS);
        r.out.track_hits = pinned<int32_t>(W * HITS);
        for (int i = 0; i < requests; ++i) {
            uint64_t ticket = 0;
            hough_request_result res{};
            if (hough_server_submit(s, &r, &ticket) != HOUGH_OK ||
                hough_server_wait(s, ticket, 60000, &res) != HOUGH_OK || res.status != HOUGH_OK)
                exit(4);
            waits[k].push_back(res.launch_ns - res.arrival_ns);
        }
    };
    std::vector<std::thread> threads;
    for (int k = 0; k < clients; ++k)
        threads.emplace_back(client, k);
    for (std::thread &t : threads)
        t.join();
    hough_server_destroy(s);
    hough_destroy(ctx);
    std::vector<int64_t> all;
    for (const auto &v : waits)
        all.insert(all.end(), v.begin(), v.end());
    std::sort(all.begin(), all.end());
    std::printf("%lld\n", (long long)all[all.size() / 2]);
    return 0;
}
