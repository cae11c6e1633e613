// The request loop's rule for holding requests back (hough_gather.h), run
// against a clock of one microsecond a step.
//   gather <slots> <slot_windows> <request_windows> <clients> <gap_us> <requests>
// clients > 0: that many clients, each waiting for its last request before it
// sends the next; 0: a request every gap_us, its result collected at once; -1: a
// request every gap_us, results left unread.  A batch takes 90 us.
// Prints: batches, requests of the largest batch, and the mean time, in ns, that
// requests waited while a slot was free.
#include <cstdio>
#include <cstdlib>
#include <deque>
#include <vector>

#include "hough_gather.h"

struct Request {
    int64_t at;
    bool soon;
    int client;
};

int main(int argc, char **argv)
{
    if (argc != 7)
        return 1;
    const int slots = atoi(argv[1]), slot_windows = atoi(argv[2]), windows = atoi(argv[3]);
    const int clients = atoi(argv[4]), gap = atoi(argv[5]), requests = atoi(argv[6]);
    Gather g(152, slot_windows, 1 << 20);
    std::deque<Request> queue;
    std::vector<std::vector<Request>> slot(slots);
    std::vector<int64_t> done(slots, -1);            // -1: free
    std::vector<int64_t> next(clients > 0 ? clients : 1);
    for (size_t c = 0; c < next.size(); ++c)
        next[c] = 37 * (int64_t)c;
    int sent = 0, served = 0, batches = 0, largest = 0;
    int64_t waited = 0;
    for (int64_t t = 0; served < requests; ++t) {
        const int64_t ns = 1000 * t;
        for (size_t c = 0; c < next.size(); ++c)
            if (sent < requests && next[c] >= 0 && t >= next[c]) {
                queue.push_back({ns, g.queued(ns, windows, 0), (int)c});
                next[c] = clients > 0 ? -1 : next[c] + gap;
                ++sent;
            }
        bool busy = false;
        for (int k = 0; k < slots; ++k) {
            if (done[k] >= 0 && t >= done[k]) {
                for (const Request &r : slot[k])
                    if (clients > 0)
                        next[r.client] = t + 1;
                served += (int)slot[k].size();
                done[k] = -1;
            }
            busy = busy || done[k] >= 0;
        }
        for (int k = 0; k < slots && !queue.empty(); ++k) {
            if (done[k] >= 0)
                continue;
            int waiting = 0;
            for (const int64_t n : next)
                waiting += clients > 0 && n < 0;
            if (g.hold(ns, queue.front().at, queue.front().soon, busy, clients < 0 ? served : 0, waiting)) {
                waited += 1000 * (int64_t)queue.size();
                break;
            }
            slot[k].clear();
            int w = 0;
            while (!queue.empty() && (slot[k].empty() || w + windows <= slot_windows)) {
                w += windows;
                slot[k].push_back(queue.front());
                queue.pop_front();
            }
            g.taken(w, 0);
            batches += 1;
            largest = largest > (int)slot[k].size() ? largest : (int)slot[k].size();
            done[k] = t + 90;
            busy = true;
        }
        if (t > 1000000)
            return 2;                                // never served
    }
    std::printf("%d %d %lld\n", batches, largest, (long long)(waited / requests));
    return 0;
}
