// How a strided batch runs: the host rules, free of device code.
#pragma once

#include <cstddef>
#include <cstdint>
#include <algorithm>

#include "group_plan.h"

namespace adapt {

// Re-pitched copies of a batch's operands are held for this many bytes of entries at a time (the stream keeps that workspace; a batch
// whose copies are larger goes in several launches).  Each further launch drains and fills the chip once more, about 8 us: with 64 MB at a
// time 200 x (520 x 1003 x 331), 200 MB of copies, took 279 us against 249 in one launch, and keeping the copies in L2 gave nothing back.
constexpr int64_t kBatchCopyBytes = (int64_t)256 << 20;

// An operand of a strided batch as the tensor-core kernel reads it: in place, or (rows or entries off 16-byte boundaries, narrow
// rows) over one re-pitched copy of all entries, which takes entries that lie back to back.
struct BatchOperand {
    const void* src;
    int64_t inner, outer, entries, stride;     // of the caller's matrices (entries = 1: shared by the batch)
    bool shared, copy, ok;
    int64_t pitch, entry_stride;               // of what TMA reads
    BatchOperand(const void* p, int64_t in, int64_t out, int64_t batch, int64_t st)
        : src(p), inner(in), outer(out), entries(st == 0 ? 1 : batch), stride(st == 0 ? in * out : st), shared(st == 0)
    {
        copy = !tma_friendly(inner) || ((uintptr_t)p & 15) != 0 || (entries > 1 && stride % 8 != 0);
        ok = !copy || stride == inner * outer;
        pitch = copy ? padded_pitch(inner) : inner;
        entry_stride = copy || entries == 1 ? pitch * outer : stride;
    }
    int64_t entry_bytes() const { return copy ? outer * pitch * 2 : 0; }                    // of the copy of one entry
    size_t bytes() const { return (size_t)round_up(entries * entry_bytes(), 256); }         // of the copy
    // entries first .. first + count - 1 of the batch
    BatchOperand part(int64_t first, int64_t count) const
    {
        BatchOperand o = *this;
        if (shared) return o;
        o.src = (const unsigned short*)src + first * stride;
        o.entries = count;
        return o;
    }
};

// The entries of one launch: as many as keep the copies of both operands within `limit` bytes (0: not even one entry does).
inline int64_t batch_chunk(const BatchOperand& a, const BatchOperand& b, int64_t batch, int64_t limit)
{
    const int64_t shared = (a.shared ? a.entry_bytes() : 0) + (b.shared ? b.entry_bytes() : 0);
    const int64_t each = (a.shared ? 0 : a.entry_bytes()) + (b.shared ? 0 : b.entry_bytes());
    const int64_t room = limit - 512 - shared;                         // 512: each copy ends on a 256-byte boundary
    if (shared + each == 0) return batch;
    if (room < each) return 0;
    return each == 0 ? batch : std::min(batch, room / each);
}

// Entry by entry, or in one launch on the grouped kernel's or in one or several on the tensor-core kernel's tiles.
enum { kBatchLoop = 0, kBatchGroup, kBatchUmma };
struct BatchRoute { int kind, BN; int64_t chunk; };

// The estimates behind the choice (us).  Grouped kernel: rounds of two CTAs per SM, 1.5 us and 0.6 us per stage of a group of warps.
// Tensor-core kernel: rounds of one CTA per SM, k-blocks of 0.25 to 0.42 us (64 to 256 columns) or the tile's drain, whichever is
// longer, a copy of operands that TMA cannot read in place, 4 us around it.  Entry by entry: the plan's prediction less the
// microsecond that consecutive launches overlap.
inline BatchRoute batch_route(const Shape& s, const Config& c, const Machine& m, int64_t batch, bool group_ok, bool umma_ok, const BatchOperand& a,
                              const BatchOperand& b, bool tma_store)
{
    BatchRoute best = {kBatchLoop, 0, batch};
    double us = (double)batch * std::max(1.5, c.predicted_us - 1.0);
    if (group_ok) {
        const double rounds = (double)ceil_div(batch * ceil_div(s.M, 64) * ceil_div(s.N, 64), 2 * (int64_t)m.n_sm);
        const double chain = c.family == ADAPT_FAM_SIMT ? 1.0 : (double)ceil_div(s.K, 2 * kClusterKS);
        const double t = 3.0 + rounds * (1.5 + 0.6 * chain);
        if (t < us) { us = t; best = {kBatchGroup, 0, batch}; }
    }
    const int64_t chunk = umma_ok && a.ok && b.ok ? batch_chunk(a, b, batch, std::min(kBatchCopyBytes, m.workspace_limit)) : 0;
    if (chunk > 0) {
        for (int BN : {64, 128, 256}) {
            if (BN > 64 && s.N <= BN / 2) continue;
            const double t_kb = BN == 64 ? 0.25 : BN == 128 ? 0.30 : 0.42;
            const double kb = 2.0 * std::min<double>(128.0, (double)s.M) * BN / 1024.0;
            const double drain = tma_store ? 0.25 + 0.0275 * kb : 1.4 + 0.031 * kb;
            auto launch_us = [&](int64_t n) -> double {
                const double na = a.shared ? 1.0 : (double)n, nb = b.shared ? 1.0 : (double)n;
                const double copies = ((a.copy ? na * a.outer * (a.inner + a.pitch) : 0.0) + (b.copy ? nb * b.outer * (b.inner + b.pitch) : 0.0)) * 2.0;
                const double traffic = 2.0 * (na * s.M * s.K + nb * s.K * s.N + (double)n * s.M * s.N);
                const double rounds = (double)ceil_div(n * ceil_div(s.M, 128) * ceil_div(s.N, BN), m.n_sm);
                return std::max(rounds * std::max((double)ceil_div(s.K, 64) * t_kb, drain), traffic / 5.5e6) + 4.0 + (copies > 0 ? 0.5 + copies / 5.5e6 : 0.0);
            };
            const double t = (double)(batch / chunk) * launch_us(chunk) + (batch % chunk ? launch_us(batch % chunk) : 0.0);
            if (t < us) { us = t; best = {kBatchUmma, BN, chunk}; }
        }
    }
    return best;
}

}  // namespace adapt
