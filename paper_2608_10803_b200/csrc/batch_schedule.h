// Order of the launches of adapt_matmul_batch: which calls leave together, on which stream, and which streams wait for which.
// Plain C++ (no device code): the launches, and the waits of one stream for another, are the caller's `Ops`.
#pragma once

#include <cstddef>
#include <cstdint>
#include <algorithm>
#include <vector>

#include "group_plan.h"

namespace adapt {

struct Range { uintptr_t lo, hi; };
inline bool hits(const std::vector<Range>& v, const Range& x)
{
    bool any = false;
    for (const Range& r : v) any |= (x.lo < r.hi) & (r.lo < x.hi);
    return any;
}

// One call of the list, as far as the order matters.
struct BatchCall {
    Range a, b, c;              // what it reads (A, B) and writes (C)
    bool unsound;               // null, misaligned or overlapping operands: most likely refused, so the calls before it leave first
    bool groupable;             // may join a grouped launch
    bool workspace;             // needs the workspace of the stream it runs on
    bool alone;                 // nothing may run beside it (stream-K: its CTAs wait for one another and must all be resident)
    double us;                  // predicted time
};
constexpr int kBatchInternalMax = 4;                        // internal streams
constexpr int kBatchLanesMax = 1 + kBatchInternalMax;       // ... and the caller's

// Internal streams for a list of `count` calls of which `singles` are launched by themselves, `with_workspace` of them over a workspace:
// none for a short list, else no more than `limit` and no more than there are launches to overlap (the caller's stream takes part).
inline int batch_internal_lanes(int64_t count, int64_t singles, int64_t with_workspace, int limit)
{
    if (count < 8 || limit < 2) return 0;
    const int64_t launches = singles + (singles < count ? 1 : 0);
    return (int)std::max<int64_t>(0, std::min<int64_t>(std::min(limit, kBatchInternalMax), std::max(with_workspace, launches - 1)));
}

// The calls 0 .. count-1 of call_of(i), with the result of running them in that order.
//
// Groupable calls are collected and leave together in grouped launches; the others are launched as they come.  A call is only
// collected, and another only launched past the collected ones, while none of its buffers meets theirs in a way that order would
// matter.
//
// Lanes are streams that run beside each other; lane 0 is the caller's stream.  A call that needs a workspace goes to one of the others
// where there are any: theirs are kept from list to list, whatever stream the caller names, so a list that has run once runs without
// growing one on every stream, also in a capture on a stream that has not been used before.  A launch goes to the lane with the least predicted work queued, so that the
// launch gaps and the tail of one call fill with the next call's work.  A launch whose output overlaps what another lane still reads
// or writes, or whose inputs overlap what it writes, first waits for that lane; a lane remembers the buffers of its last 16 calls,
// and when that memory is full all other lanes are made to wait for it.
//
// Ops: adapt_status_t single(int64_t i, int lane), group(const std::vector<int64_t>& calls, int lane), and wait(int lane, int other):
// `lane` continues after everything queued on `other`.
template <class CallOf, class Ops>
adapt_status_t run_batch(int64_t count, int lanes, CallOf call_of, Ops& ops)
{
    constexpr size_t kLaneMemory = 32;
    std::vector<Range> reads[kBatchLanesMax], writes[kBatchLanesMax];
    double queued[kBatchLanesMax] = {};

    // Chooses the lane of a launch that reads and writes the given buffers and makes it wait for the lanes it depends on.
    auto enter = [&](const Range* rd, size_t n_rd, const Range* wr, size_t n_wr, bool alone, bool workspace, int* out) -> adapt_status_t {
        int lane = workspace && lanes > 1 ? 1 : 0;
        for (int l = lane + 1; l < lanes; ++l) if (queued[l] < queued[lane]) lane = l;
        *out = lane;
        for (int o = 0; o < lanes; ++o) {
            if (o == lane) continue;
            bool dep = alone;
            for (size_t j = 0; j < n_wr && !dep; ++j) dep = hits(reads[o], wr[j]) || hits(writes[o], wr[j]);
            for (size_t j = 0; j < n_rd && !dep; ++j) dep = hits(writes[o], rd[j]);
            // everything lane o has queued comes first; what o did before is then ordered before all of this lane's
            // later calls as well, but the other lanes still have to see it: keep o's memory
            if (dep) { const adapt_status_t r = ops.wait(lane, o); if (r != ADAPT_OK) return r; }
        }
        if (lanes > 1 && reads[lane].size() >= kLaneMemory) {
            // this lane's memory is full: every other lane waits for it, and it starts a new memory
            for (int o = 0; o < lanes; ++o)
                if (o != lane) { const adapt_status_t r = ops.wait(o, lane); if (r != ADAPT_OK) return r; }
            reads[lane].clear();
            writes[lane].clear();
        }
        return ADAPT_OK;
    };
    auto leave = [&](int lane, const Range* rd, size_t n_rd, const Range* wr, size_t n_wr, double us) {
        queued[lane] += std::max(1.0, us);
        if (lanes == 1) return;
        reads[lane].insert(reads[lane].end(), rd, rd + n_rd);
        writes[lane].insert(writes[lane].end(), wr, wr + n_wr);
    };

    std::vector<int64_t> group;                         // the calls collected so far, independent of one another
    std::vector<Range> group_reads, group_writes;
    double group_us = 0.0;
    auto flush = [&]() -> adapt_status_t {
        if (group.empty()) return ADAPT_OK;
        int lane = 0;
        adapt_status_t r = enter(group_reads.data(), group_reads.size(), group_writes.data(), group_writes.size(), false, false, &lane);
        if (r == ADAPT_OK) r = ops.group(group, lane);
        if (r == ADAPT_OK) leave(lane, group_reads.data(), group_reads.size(), group_writes.data(), group_writes.size(), group_us);
        group.clear();
        group_reads.clear();
        group_writes.clear();
        group_us = 0.0;
        return r;
    };

    adapt_status_t status = ADAPT_OK;
    for (int64_t i = 0; i < count && status == ADAPT_OK; ++i) {
        const BatchCall k = call_of(i);
        if ((k.unsound || hits(group_writes, k.a) || hits(group_writes, k.b) || hits(group_writes, k.c) || hits(group_reads, k.c)) && (status = flush()) != ADAPT_OK) break;
        if (k.groupable && !k.unsound) {
            group.push_back(i);
            group_reads.push_back(k.a);
            group_reads.push_back(k.b);
            group_writes.push_back(k.c);
            group_us += 0.25 * k.us;
            if (group.size() >= kGroupMax) status = flush();
            continue;
        }
        const Range rd[2] = {k.a, k.b};
        int lane = 0;
        if ((status = enter(rd, 2, &k.c, 1, k.alone, k.workspace, &lane)) != ADAPT_OK) break;
        if ((status = ops.single(i, lane)) != ADAPT_OK) break;
        leave(lane, rd, 2, &k.c, 1, k.us);
        if (k.alone)
            for (int o = 0; o < lanes && status == ADAPT_OK; ++o)
                if (o != lane) status = ops.wait(o, lane);
    }
    // the calls still collected come before the one that failed: they leave in any case, and the first error is the result
    const adapt_status_t r = flush();
    return status != ADAPT_OK ? status : r;
}

}  // namespace adapt
