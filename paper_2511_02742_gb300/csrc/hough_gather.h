// hough_gather.h -- when the request loop (hough_server.cpp) holds requests back
// although a slot is free, so that others may join their batch.  Host code
// without CUDA.
#pragma once

#include <algorithm>
#include <cstdint>

// How long a request may be held.  About the time of a small batch, so that
// requests that keep coming one after the other (39 us apart and less) are
// served by few batches, not by one batch (ten copies and a launch) each.
constexpr int64_t kGatherNs = 60'000;

// Results that lie there unread before requests are held.
constexpr int64_t kGatherUnread = 4;

// Holding costs every client that looks at its results time and gains it none
// (requests of 20 windows, mean latency held and not: two clients that wait for
// their results 121 and 76 us, four 145 and 109, a request every 39 us whose
// results are polled 102 and 67; the rates are those of the clients, or lower
// held).  So requests are held only while nobody looks:
//  - no thread waits for a result (wait, drain), and results lie there unread:
//    the client sends many requests before it collects; and
//  - a batch is on the GPU (else a request starts at once), and the request
//    came less than kGatherNs after the one before it (a lone one has nobody to
//    join), less than kGatherNs ago; and
//  - the queue leaves room: fewer windows than the GPU has SMs, and than a slot
//    takes, and fewer hits than a slot takes.
class Gather {
public:
    Gather(int64_t full_windows, int64_t slot_windows, int64_t slot_hits)
        : full_(std::min(full_windows, slot_windows)), hits_full_(slot_hits) {}

    // A request was queued; returns whether it came soon after the one before.
    bool queued(int64_t now, int64_t windows, int64_t hits)
    {
        const bool soon = any_ && now - last_ < kGatherNs;
        any_ = true;
        last_ = now;
        windows_ += windows;
        hits_ += hits;
        return soon;
    }

    // A batch was taken from the queue.
    void taken(int64_t windows, int64_t hits)
    {
        windows_ -= windows;
        hits_ -= hits;
    }

    // Whether to hold the queue, whose oldest request came at `queued` (`soon`:
    // what queued() said of it).  busy: a batch is on the GPU; unread: completed
    // results not yet delivered; waiting: threads in wait or drain.
    bool hold(int64_t now, int64_t queued, bool soon, bool busy, int64_t unread, int waiting) const
    {
        return busy && soon && waiting == 0 && unread >= kGatherUnread && windows_ < full_ &&
               hits_ < hits_full_ && now - queued < kGatherNs;
    }

private:
    int64_t full_, hits_full_;
    int64_t windows_ = 0, hits_ = 0;     // queued
    int64_t last_ = 0;                   // when the last request was queued
    bool any_ = false;
};
