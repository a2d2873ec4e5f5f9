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
    int variant;                // ... of this kernel, data type and pair of layouts (0 .. kBatchKinds - 1)
    bool workspace;             // needs the workspace of the stream it runs on
    bool alone;                 // nothing may run beside it (stream-K: its CTAs wait for one another and must all be resident)
    double us;                  // predicted time
};
constexpr int kBatchVariants = 8;                           // data types and pairs of layouts
constexpr int kBatchDirect = kBatchVariants;                // ... and from here on the same for calls of one tcgen05 tile per CTA (direct_gemm.cuh)
constexpr int kBatchKinds = 2 * kBatchVariants;
constexpr int kBatchInternalMax = 4;                        // internal streams
constexpr int kBatchLanesMax = 1 + kBatchInternalMax;       // ... and the caller's

// What a second stream has to hide of a list of two launches (us) to be worth the events of its fork and join.
constexpr double kBatchForkUs = 4.0;

// Internal streams for a list of `count` calls of which `singles` are launched by themselves, `with_workspace` of them over a workspace, and the
// others in `grouped` launches: none for a short list, nor for two launches in all without a workspace of which a second stream would hide less than
// kBatchForkUs, else no more than `limit` and no more than there are calls to overlap (the caller's stream takes part).
inline int batch_internal_lanes(int64_t count, int64_t singles, int64_t with_workspace, int limit, int64_t grouped = 1, double hidden_us = 0.0)
{
    if (count < 8 || limit < 2) return 0;
    if (with_workspace == 0 && singles + (singles < count ? grouped : 0) <= 2 && hidden_us < kBatchForkUs) return 0;
    const int64_t apart = singles + (singles < count ? 1 : 0);         // the grouped launches follow one another
    return (int)std::max<int64_t>(0, std::min<int64_t>(std::min(limit, kBatchInternalMax), std::max(with_workspace, apart - 1)));
}

// What a second stream hides of a grouped launch of these entries (in group_order) and a call of `single_us`.  The launch leaves SMs idle while its
// longest chain runs: about 2 us a stage, against 3.3 us for what a CTA slot (two per SM) has to do on average.  A long call covers the launch's start
// and end.  Measured over 140 such lists of 8 to 48 calls, 128 to 1500 a side, time on two streams over time on one: where this says 4 us or more (23 lists)
// 0.68 to 1.01, 0.90 on average (15 calls to 1500 and 4096 x 4096 x 4096: 138.8 -> 107.2 us); elsewhere 1.035 on average, one stream being faster by more
// than 5 % in 51 lists (23 calls to 256 and 20000 x 64 x 64: 15.5 and 17.7) and slower in 15.
inline double batch_hidden_us(const GroupEntry* e, size_t n, int n_sm, double single_us)
{
    double work = 0.0;
    int longest = 0;
    for (size_t j = 0; j < n; ++j) {
        work += (double)(e[j].item.tiles << e[j].item.share_log2) * e[j].chain;
        longest = std::max(longest, e[j].chain);
    }
    const double idle = 2.0 * longest - 3.3 * work / (2.0 * n_sm);
    return std::max(std::min(idle, single_us), 0.05 * single_us);
}

// The calls 0 .. count-1 of call_of(i), with the result of running them in that order.
//
// Groupable calls are collected per variant, up to kGroupMax of one, and leave together in one grouped launch; the others are launched
// as they come.  A call is only collected, and another only launched past the collected ones, while none of its buffers meets theirs
// in a way that order would matter.
//
// Lanes are streams that run beside each other; lane 0 is the caller's stream.  A call that needs a workspace goes to one of the others
// where there are any: theirs are kept from list to list, whatever stream the caller names, so a list that has run once runs without
// growing one on every stream, also in a capture on a stream that has not been used before.  A launch goes to the lane with the least predicted work queued, so that the
// launch gaps and the tail of one call fill with the next call's work.  A launch whose output overlaps what another lane still reads
// or writes, or whose inputs overlap what it writes, first waits for that lane; a lane remembers the buffers of its last 16 calls,
// and when that memory is full all other lanes are made to wait for it.
//
// Ops: adapt_status_t single(int64_t i, int lane), group(const std::vector<int64_t>& calls, int lane) with calls of one variant, independent
// of one another, and wait(int lane, int other):
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

    struct Pending {                                    // the calls of one variant collected so far; those of all variants are independent
        std::vector<int64_t> calls;
        std::vector<Range> reads, writes;
        double us = 0.0;
    } pending[kBatchKinds];
    auto flush = [&](Pending& g) -> adapt_status_t {
        if (g.calls.empty()) return ADAPT_OK;
        int lane = 0;
        adapt_status_t r = enter(g.reads.data(), g.reads.size(), g.writes.data(), g.writes.size(), false, false, &lane);
        if (r == ADAPT_OK) r = ops.group(g.calls, lane);
        if (r == ADAPT_OK) leave(lane, g.reads.data(), g.reads.size(), g.writes.data(), g.writes.size(), g.us);
        g.calls.clear();
        g.reads.clear();
        g.writes.clear();
        g.us = 0.0;
        return r;
    };
    unsigned collected = 0;                             // the kinds that have any (a list of small calls asks for them at every call)
    auto flush_all = [&]() -> adapt_status_t {          // every kind leaves, also after one that failed; the first error
        adapt_status_t first = ADAPT_OK;
        for (int v = 0; collected >> v; ++v) {
            const adapt_status_t r = flush(pending[v]);
            if (first == ADAPT_OK) first = r;
        }
        collected = 0;
        return first;
    };
    auto meets_pending = [&](const BatchCall& k) -> bool {
        for (int v = 0; collected >> v; ++v) {
            const Pending& g = pending[v];
            if (!g.calls.empty() && (hits(g.writes, k.a) || hits(g.writes, k.b) || hits(g.writes, k.c) || hits(g.reads, k.c))) return true;
        }
        return false;
    };

    adapt_status_t status = ADAPT_OK;
    for (int64_t i = 0; i < count && status == ADAPT_OK; ++i) {
        const BatchCall k = call_of(i);
        if ((k.unsound || meets_pending(k)) && (status = flush_all()) != ADAPT_OK) break;
        if (k.groupable && !k.unsound) {
            Pending& g = pending[k.variant];
            if (g.calls.empty()) {                      // (growing them call by call is a tenth of what a list of small calls takes the host)
                g.calls.reserve(kGroupMax);
                g.reads.reserve(2 * kGroupMax);
                g.writes.reserve(kGroupMax);
            }
            collected |= 1u << k.variant;
            g.calls.push_back(i);
            g.reads.push_back(k.a);
            g.reads.push_back(k.b);
            g.writes.push_back(k.c);
            g.us += 0.25 * k.us;
            if (g.calls.size() >= kGroupMax) status = flush(g);
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
    const adapt_status_t r = flush_all();
    return status != ADAPT_OK ? status : r;
}

}  // namespace adapt
