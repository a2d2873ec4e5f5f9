// tcgen05 GEMM on tall pair tiles: 512 x 256 outputs per SM pair, all 512 TMEM columns as the two accumulators of ONE tile.
//
// The 256 x 256 pair tile (umma_gemm.cuh) brings 32 KB per k-block and SM for 512 cycles of MMA: when this kernel was written, that loop was bound by its loads
// (8192^3 with zero operands, where power does not interfere, cycles per k-block: 685 in full, 587 with the MMAs alone, 638 with the loads
// alone; six or seven stages change nothing), and with data in the operands the same traffic is the energy the power cap takes out of the
// clock.  Here a CTA takes 256 rows and half of 256 columns: 48 KB per 1024 cycles of MMA, a quarter less per flop.
// Measured by itself in a row of calls, 256 x 256 pair tiles -> this kernel, bf16 with random operands under the power cap: 8192^3 920 -> 801 us,
// 16384 x 16384 x 4096 2167 -> 1560, 2048 x 14336 x 4096 207 -> 183, 2048 x 4096 x 4096 59 -> 52, 4096 x 4096 x 2048 64 -> 55, 12288 x 688 x 16991 (row
// classes) 305 -> 258.  A 2048-token training step of a 4096 x 4096 layer makes the fourth of these twice and the fifth once: one after the other, with
// operands from DRAM and 64 tiles on 74 pairs, they take 193 -> 186 us in all.  Short k ranges gain little: 8192 x 4096 x 512 36.6 -> 34.6,
// 10000 x 1024 x 1024 23.5 -> 23.0, and row classes lose there (20000 x 512 x 333: 17.1, 15.6 on 1-CTA tiles).  8192^3 with zero operands: 601 -> 523 us
// = 2.1 PFLOP/s.  Profiled on 8192 x 8192 x 4096: tensor pipe 88 % busy (78), 3.6 GB through L2 (5.3).
//
// The two accumulators are the halves of one tile, so there is no spare buffer to hide the drain of a tile behind the next one's MMAs.
// Instead the halves are a few k-blocks apart at the ends of a tile: the upper half's MMAs of the first kTallLag k-blocks are issued before
// the lower half's, and so are those of the last: the epilogue empties the upper accumulator while the lower one is finished, and the
// lower one while the next tile's upper half has begun.  The epilogue packs its share of both halves into registers, hands the accumulators
// back, and lets the packed values leave through one TMA store box per warp (the ring takes 192 KB) beside the next tile's MMAs.
// (Stored from the registers, 32 rows of 32 bytes an instruction, a tile took 8 us instead of 4.)
//
// Tiles that would leave most of the last wave idle are cut into their 256-row halves (tall_schedule).  k runs in one order (no rotation by tile).
#pragma once

#include "umma_gemm.cuh"

namespace adapt {

constexpr int kTallLag = 3;          // k-blocks between the halves of a tile at its ends (held in the ring meanwhile: below kTallStages)
static_assert(kTallLag < kTallStages, "the held k-blocks are part of the ring");

struct TallParams {
    int M, N;
    int kb_total;                    // k-blocks
    TallWork work;
    int dtype;
    uint32_t idesc;
    int a_sigma[8];                  // row classes: shift (elements) of class j against its 16-byte aligned base
    int c_hint;                      // C (rows on 32-byte boundaries) is stored with an evict-first L2 policy
    int prefetch;                    // ask L2 for the first boxes ahead of the dependency wait
    ReduceEpilogue ep;
    unsigned int* status;
};

template <bool A_MN, bool B_MN, bool CLS, bool EPI>
__global__ void __launch_bounds__(kUmmaThreads, 1)
tall_gemm_kernel(const __grid_constant__ TmapPackT<CLS ? 1 : 0> maps, const __grid_constant__ TallParams p)
{
    static_assert(!CLS || (!A_MN && B_MN), "row classes: K-major A, row-major B");
    constexpr int S = kTallStages;
    constexpr int A_HALF = 128 * kUmmaBK * 2;                  // this CTA's rows of one half
    constexpr int B_BYTES = 128 * kUmmaBK * 2;                 // this CTA's columns
    constexpr int STAGE_BYTES = 2 * A_HALF + B_BYTES;
    static_assert(STAGE_BYTES == kTallStageBytes, "stage layout");

    extern __shared__ uint8_t smem_raw[];
    const uint32_t smem_base = (ptx::smem_u32(smem_raw) + 1023u) & ~1023u;
    uint8_t* gen_base = smem_raw + (smem_base - ptx::smem_u32(smem_raw));
    const uint32_t bar_base = smem_base + (uint32_t)S * STAGE_BYTES;
    // barrier block: full[S], empty[S], "this CTA's A boxes have landed"[S], "the peer's A rows are ready"[S], tmem_full[2], tmem_empty[2],
    // the TMEM pointer, the abort flag
    const uint32_t full_bar = bar_base, empty_bar = bar_base + 8u * S, afull_bar = bar_base + 16u * S, aready_bar = bar_base + 24u * S;
    const uint32_t tfull_bar = bar_base + 32u * S, tempty_bar = tfull_bar + 16u, tmem_slot = tempty_bar + 16u;
    uint8_t* bar_gen = gen_base + (size_t)S * STAGE_BYTES;
    volatile uint32_t* tmem_slot_ptr = reinterpret_cast<volatile uint32_t*>(bar_gen + 32 * S + 32);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(bar_gen + 32 * S + 36);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t cta_rank = ptx::cluster_ctarank();
    const bool leader = cta_rank == 0;
    const int slot = (int)(blockIdx.x >> 1), n_slots = (int)(gridDim.x >> 1);

    if (threadIdx.x == 0) {
        *abort_flag = 0;
        for (int s = 0; s < S; ++s) {
            ptx::mbar_init(full_bar + 8u * s, 1);
            ptx::mbar_init(empty_bar + 8u * s, 1);
            ptx::mbar_init(afull_bar + 8u * s, 1);
            ptx::mbar_init(aready_bar + 8u * s, 1);
        }
        for (int h = 0; h < 2; ++h) {
            ptx::mbar_init(tfull_bar + 8u * h, 1);
            ptx::mbar_init(tempty_bar + 8u * h, kUmmaEpilogueWarps * 2);       // one arrive per epilogue warp of the pair
        }
        ptx::fence_barrier_init();
        ptx::fence_proxy_async_smem();
        TallItem w;
        if (tall_item<CLS>(p.work, slot, n_slots, 0, w)) {
            ptx::prefetch_tensormap(&maps.a[CLS ? (w.blk0 & 7) : 0]);
            ptx::prefetch_tensormap(&maps.c[CLS ? (w.blk0 & 7) : 0]);
        }
        ptx::prefetch_tensormap(&maps.b[0]);
    }
    if (warp == 1) {
        ptx::tmem_alloc<2>(tmem_slot, 512);
        ptx::tmem_relinquish<2>();
        pdl_launch_dependents();                               // (umma_gemm.cuh says why not before)
    }
    ptx::tc_fence_before();
    ptx::cluster_sync_all();                                   // the peer's barriers exist
    ptx::tc_fence_after();
    const uint32_t tmem_base = *tmem_slot_ptr;

    // The TMA requests of a k-block: A's boxes of the upper half, of the lower half, then B's.
    constexpr int A_BOXES = A_MN ? 2 : 1;                      // per half: one of 64 k x 128 rows, or two of 64 rows x 64 k
    constexpr int B_BOXES = B_MN ? 2 : 1;
    constexpr int NREQ = 2 * A_BOXES + B_BOXES;
    const bool is_a = lane < 2 * A_BOXES;
    const int half_of = lane / A_BOXES, ja = lane % A_BOXES, jb = lane - 2 * A_BOXES;
    auto row_of = [&](int blk) -> int {                        // this CTA's first row of a block: of A, or of the class's view
        return (CLS ? (blk >> 3) : blk) * 256 + (int)cta_rank * 128;
    };

    if (warp == 0 && lane < NREQ && p.prefetch) {              // hints only, ahead of the wait for the kernel before this one
        TallItem w;
        if (tall_item<CLS>(p.work, slot, n_slots, 0, w) && (w.two || !is_a || half_of == 0)) {
            const int kshift = CLS ? p.a_sigma[w.blk0 & 7] : 0;
            for (int kb = 0; kb < min(S, p.kb_total); ++kb) {
                const int k0 = kb * kUmmaBK;
                if (is_a) {
                    const int row = row_of(half_of ? w.blk1 : w.blk0) + (A_MN ? 64 * ja : 0);
                    ptx::tma_prefetch_2d(&maps.a[CLS ? (w.blk0 & 7) : 0], A_MN ? row : k0, A_MN ? k0 : row);
                } else {
                    const int col = w.nb * 256 + (int)cta_rank * 128 + (B_MN ? 64 * jb : 0);
                    ptx::tma_prefetch_2d(&maps.b[0], B_MN ? col : k0, B_MN ? k0 - kshift : col);
                }
            }
        }
    }
    pdl_wait();

    if (warp == 0) {
        // ------------------------------ producer -----------------------------------------------
        // (one elected thread: umma_gemm.cuh's producer says why)
        if (ptx::elect_one()) {
            int stage = 0;
            uint32_t phase = 0;
            uint32_t full_leader, afull_own;                   // cluster addresses: the leader's barriers, this CTA's own
            asm volatile("mapa.shared::cluster.u32 %0, %1, 0;" : "=r"(full_leader) : "r"(full_bar));
            asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(afull_own) : "r"(afull_bar), "r"(cta_rank));
            bool ok = true;
            TallItem w;
            for (int it = 0; ok && tall_item<CLS>(p.work, slot, n_slots, it, w); ++it) {
                const int cls = CLS ? (w.blk0 & 7) : 0;
                const int kshift = CLS ? p.a_sigma[cls] : 0;       // B's k-rows lag A's by sigma
                const CUtensorMap* tmA = &maps.a[cls];
                const int a_bytes = w.two ? 2 * A_HALF : A_HALF;
                const int rows[2] = {row_of(w.blk0), row_of(w.blk1)}, col = w.nb * 256 + (int)cta_rank * 128;
                for (int kb = 0; kb < p.kb_total; ++kb) {
                    if (!ptx::mbar_wait(empty_bar + 8u * stage, phase ^ 1u, abort_flag)) { ok = false; break; }
                    const bool heads = CLS && kb == 0 && kshift > 0;       // A's first k-block has row heads to zero: it reports to its own CTA
                    if (heads) ptx::mbar_arrive_expect_tx(afull_bar + 8u * stage, (uint32_t)a_bytes);
                    if (leader) ptx::mbar_arrive_expect_tx(full_bar + 8u * stage, (uint32_t)(2 * (B_BYTES + (heads ? 0 : a_bytes))));
                    const int k0 = kb * kUmmaBK;
                    const uint32_t at = smem_base + (uint32_t)stage * STAGE_BYTES, fb = full_leader + 8u * stage;
                    const uint32_t ab = heads ? afull_own + 8u * stage : fb;
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        if (h == 1 && !w.two) break;
#pragma unroll
                        for (int j = 0; j < A_BOXES; ++j)
                            ptx::tma_load_2d_pair(at + (uint32_t)(h * A_HALF + j * 8192), tmA, ab, A_MN ? rows[h] + 64 * j : k0, A_MN ? k0 : rows[h]);
                    }
#pragma unroll
                    for (int j = 0; j < B_BOXES; ++j)
                        ptx::tma_load_2d_pair(at + (uint32_t)(2 * A_HALF + j * 8192), &maps.b[0], fb, B_MN ? col + 64 * j : k0 - kshift, B_MN ? k0 - kshift : col);
                    if (++stage == S) { stage = 0; phase ^= 1u; }
                }
            }
        }
    } else if (warp == 1) {
        // ------------------------------ MMA issuer ---------------------------------------------
        // Row classes: the sigma elements in front of each row of a unit's first k-block belong to the previous row of A; the warp
        // zeroes them in its own CTA before the tensor core reads them, the peer's warp 1 tells the leader when its half is done.
        auto zero_row_heads = [&](int stage, int sigma, bool two) {
            uint8_t* genA = gen_base + (size_t)stage * STAGE_BYTES;
            uint32_t keep[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) keep[i] = (2 * i >= sigma ? 0x0000ffffu : 0u) | (2 * i + 1 >= sigma ? 0xffff0000u : 0u);
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                if (h == 1 && !two) break;
                uint4 v[4];
#pragma unroll
                for (int t = 0; t < 4; ++t) {
                    const int r = lane + 32 * t;
                    v[t] = *reinterpret_cast<const uint4*>(genA + h * A_HALF + r * 128 + ((r & 7) << 4));
                }
#pragma unroll
                for (int t = 0; t < 4; ++t) {
                    const int r = lane + 32 * t;
                    *reinterpret_cast<uint4*>(genA + h * A_HALF + r * 128 + ((r & 7) << 4)) =
                        make_uint4(v[t].x & keep[0], v[t].y & keep[1], v[t].z & keep[2], v[t].w & keep[3]);
                }
            }
            ptx::fence_proxy_async_smem();
            __syncwarp();
        };
        int stage = 0;
        uint32_t phase = 0, aphase = 0;                        // aphase: per stage, parity of the next use of its A barriers
        TallItem w;
        if (!leader) {
            if (CLS)
                for (int it = 0; tall_item<CLS>(p.work, slot, n_slots, it, w); ++it) {
                    const int sigma = p.a_sigma[w.blk0 & 7];
                    if (sigma > 0) {
                        if (!ptx::mbar_wait_warp(afull_bar + 8u * stage, (aphase >> stage) & 1u, abort_flag)) break;
                        zero_row_heads(stage, sigma, w.two);
                        if (lane == 0) ptx::mbar_arrive_cluster(aready_bar + 8u * stage, 0);
                        aphase ^= 1u << stage;
                    }
                    stage = (stage + p.kb_total) % S;
                }
        } else {
            // One elected thread issues the MMAs and their commits; with row classes the warp comes here together for every item.
            constexpr uint32_t a_kstep = A_MN ? 2048u : 32u, b_kstep = B_MN ? 2048u : 32u;
            const uint64_t a_desc = ptx::smem_desc_sw128(smem_base, A_MN ? 8192u : 16u, 1024u);
            const uint64_t b_desc = ptx::smem_desc_sw128(smem_base + 2u * A_HALF, B_MN ? 8192u : 16u, 1024u);
            const uint32_t a_lo = (uint32_t)a_desc, a_hi = (uint32_t)(a_desc >> 32), b_lo = (uint32_t)b_desc, b_hi = (uint32_t)(b_desc >> 32), idesc = p.idesc;
            auto mma = [&](int half, int st, int acc, uint32_t more) {         // one k-block of one half; more = 0 starts its sum
                const uint32_t off = (uint32_t)st * (uint32_t)(STAGE_BYTES >> 4), ao = a_lo + off + (uint32_t)half * (uint32_t)(A_HALF >> 4), bo = b_lo + off;
#pragma unroll
                for (int k16 = 0; k16 < kUmmaBK / 16; ++k16)
                    ptx::umma_f16<2>(tmem_base + 256u * acc, ptx::smem_desc_join(ao + (k16 * a_kstep >> 4), a_hi), ptx::smem_desc_join(bo + (k16 * b_kstep >> 4), b_hi), idesc, k16 > 0 ? 1u : more);
            };
            uint32_t used = 0;                                 // bit h: parity of accumulator h's next use
            const int L = p.kb_total;
            bool heads = false;
            // an item's k-blocks, from ring position (st, ph) on
            auto contract = [&](int& st, uint32_t& ph) -> bool {
                auto next = [&]() { if (++st == S) { st = 0; ph ^= 1u; } };
                auto ready = [&]() -> bool { return ptx::mbar_wait(full_bar + 8u * st, ph, abort_flag); };      // the k-block's operands are in place
                auto enter = [&](int acc) -> bool {            // the accumulator is free
                    if (!ptx::mbar_wait(tempty_bar + 8u * acc, ((used >> acc) & 1u) ^ 1u, abort_flag)) return false;
                    used ^= 1u << acc;
                    ptx::tc_fence_after();
                    return true;
                };
                if (CLS && heads && !ptx::mbar_wait(aready_bar + 8u * st, (aphase >> st) & 1u, abort_flag)) return false;       // the peer's half too
                if (!w.two) {
                    if (!enter(w.acc)) return false;
                    for (int kb = 0; kb < L; ++kb) {
                        if (!ready()) return false;
                        mma(0, st, w.acc, kb > 0);
                        ptx::umma_commit_2(empty_bar + 8u * st);
                        next();
                    }
                    ptx::umma_commit_2(tfull_bar + 8u * w.acc);
                    return true;
                }
                // k-blocks [0, lag) and [L - lag, L): the upper half's first, then the lower half's of the same stages
                const int lag = min(kTallLag, L), tail = max(lag, L - kTallLag);
                auto apart = [&](int kb0, int kb1, bool begin, bool end) -> bool {
                    const int st0 = st;
                    if (begin && !enter(0)) return false;
                    for (int kb = kb0; kb < kb1; ++kb) {
                        if (!ready()) return false;
                        mma(0, st, 0, kb > 0);
                        next();
                    }
                    if (end) ptx::umma_commit_2(tfull_bar);
                    if (begin && !enter(1)) return false;
                    int s2 = st0;
                    for (int kb = kb0; kb < kb1; ++kb) {
                        mma(1, s2, 1, kb > 0);
                        ptx::umma_commit_2(empty_bar + 8u * s2);
                        if (++s2 == S) s2 = 0;
                    }
                    if (end) ptx::umma_commit_2(tfull_bar + 8u);
                    return true;
                };
                if (!apart(0, lag, true, lag == L)) return false;
                for (int kb = lag; kb < tail; ++kb) {
                    if (!ready()) return false;
                    mma(0, st, 0, 1u);
                    mma(1, st, 1, 1u);
                    ptx::umma_commit_2(empty_bar + 8u * st);
                    next();
                }
                return tail == L || apart(tail, L, false, true);
            };
            if (!CLS) {
                if (ptx::elect_one())
                    for (int it = 0; tall_item<CLS>(p.work, slot, n_slots, it, w) && contract(stage, phase); ++it) {}
            } else {
                for (int it = 0; tall_item<CLS>(p.work, slot, n_slots, it, w); ++it) {
                    const int sigma = p.a_sigma[w.blk0 & 7];
                    heads = sigma > 0;
                    if (heads) {
                        if (!ptx::mbar_wait_warp(afull_bar + 8u * stage, (aphase >> stage) & 1u, abort_flag)) break;
                        zero_row_heads(stage, sigma, w.two);
                    }
                    bool done = true;
                    int st = stage;
                    uint32_t ph = phase;
                    if (ptx::elect_one()) done = contract(st, ph);
                    if (!__all_sync(0xffffffffu, done)) break;
                    if (heads) aphase ^= 1u << stage;
                    const int adv = stage + L;                 // (the other lanes' copy of the ring position)
                    phase ^= (uint32_t)((adv / S) & 1);
                    stage = adv % S;
                }
            }
        }
    } else {
        // ------------------------------ epilogue -----------------------------------------------
        // Warp w reads TMEM lanes 32 (w % 4) .. + 31; the two warps of a lane quarter take 128 columns each.
        const int q = warp & 3, col0 = ((warp - 2) >> 2) * 128;
        const uint64_t policy = ptx::l2_policy_evict_first();
        uint8_t* box_gen = bar_gen + kUmmaBarrierBytes + (warp - 2) * kTallBoxBytes;   // this warp's staging box
        uint32_t used = 0;
        bool ok = true;
        TallItem w;
        for (int it = 0; ok && tall_item<CLS>(p.work, slot, n_slots, it, w); ++it) {
            const int n0 = w.nb * 256 + col0;
            auto row_at = [&](int blk) -> int {
                const int i = (int)cta_rank * 128 + q * 32 + lane;
                return CLS ? (blk >> 3) * 2048 + (blk & 7) + 8 * i : blk * 256 + i;
            };
            // Both halves wait for their stores in registers: the accumulators go back before the first store, and the stores run beside
            // the next tile's MMAs.
            uint32_t packed[2][64];                            // per half, the row's 128 columns; EPI: D's until the sums come
            if (EPI) {
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int row = row_at(h ? w.blk1 : w.blk0);
                    if (row >= p.M || (h == 1 && !w.two)) continue;
                    const unsigned short* d = p.ep.D + (p.ep.d_is_vector ? (int64_t)n0 : (int64_t)row * p.N + n0);
#pragma unroll
                    for (int v = 0; v < 16; ++v) {             // 8 columns at a time: D and its rows are aligned
                        if (n0 + 8 * v >= p.N) break;
                        const uint4 x = *reinterpret_cast<const uint4*>(d + 8 * v);
                        packed[h][4 * v] = x.x; packed[h][4 * v + 1] = x.y; packed[h][4 * v + 2] = x.z; packed[h][4 * v + 3] = x.w;
                    }
                }
            }
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                if (h == 1 && (!w.two || !ok)) break;
                const int acc = w.two ? h : w.acc;
                ok = ptx::mbar_wait(tfull_bar + 8u * acc, (used >> acc) & 1u, abort_flag);
                if (!ok) break;
                used ^= 1u << acc;
                __syncwarp();
                ptx::tc_fence_after();
                const uint32_t t_row = tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)(256 * acc + col0);
#pragma unroll
                for (int c = 0; c < 8; ++c) {                  // (16 columns at a time: 168 registers are all that ten warps leave)
                    if (n0 + 16 * c >= p.N) break;             // uniform across the warp
                    uint32_t r[16];
                    ptx::tmem_ld_32x16(t_row + (uint32_t)(16 * c), r);
                    ptx::tmem_ld_wait();
#pragma unroll
                    for (int i = 0; i < 8; ++i) {
                        float lo = __uint_as_float(r[2 * i]), hi = __uint_as_float(r[2 * i + 1]);
                        if (EPI) {
                            const uint32_t d = packed[h][8 * c + i];
                            const unsigned short d0 = (unsigned short)(d & 0xFFFFu), d1 = (unsigned short)(d >> 16);
                            lo = fmaf(p.ep.beta, load16_as_float(&d0, p.dtype), p.ep.alpha * lo);
                            hi = fmaf(p.ep.beta, load16_as_float(&d1, p.dtype), p.ep.alpha * hi);
                        }
                        packed[h][8 * c + i] = pack16(lo, hi, p.dtype);
                    }
                }
                ptx::tc_fence_before();
                __syncwarp();
                if (lane == 0) ptx::mbar_arrive_cluster(tempty_bar + 8u * acc, 0);
            }
            if (!ok) break;
            const CUtensorMap* tmC = &maps.c[CLS ? (w.blk0 & 7) : 0];
#pragma unroll
            for (int b = 0; b < 4; ++b) {                      // two boxes a half
                const int h = b >> 1, x = n0 + 64 * (b & 1);
                if (x >= p.N || (h == 1 && !w.two)) continue;  // uniform across the warp
                if (lane == 0) ptx::bulk_wait_read<0>();       // the box before has been read
                __syncwarp();
#pragma unroll
                for (int c = 0; c < 8; ++c) {
                    const uint32_t* v = packed[h] + 32 * (b & 1) + 4 * c;
                    *reinterpret_cast<uint4*>(box_gen + lane * 128 + ((c ^ (lane & 7)) << 4)) = make_uint4(v[0], v[1], v[2], v[3]);
                }
                ptx::fence_proxy_async_smem();
                __syncwarp();
                if (lane == 0) {
                    const int y = row_of(h ? w.blk1 : w.blk0) + q * 32;
                    if (p.c_hint) ptx::tma_store_2d_hint(tmC, ptx::smem_u32(box_gen), x, y, policy);
                    else ptx::tma_store_2d(tmC, ptx::smem_u32(box_gen), x, y);
                    ptx::bulk_commit();
                }
            }
        }
        if (lane == 0) ptx::bulk_wait_read<0>();
    }

    // ------------------------------ common exit ----------------------------------------------
    __syncwarp();                        // (one thread has run the producer's and the MMA issuer's loops)
    ptx::tc_fence_before();
    ptx::cluster_sync_all();                                   // no CTA leaves while its peer may still arrive on its barriers
    if (threadIdx.x == 0 && *abort_flag) atomicOr(p.status, 1u);
    if (warp == 1) {
        ptx::tc_fence_after();
        ptx::tmem_dealloc<2>(tmem_base, 512);
    }
}

}  // namespace adapt
