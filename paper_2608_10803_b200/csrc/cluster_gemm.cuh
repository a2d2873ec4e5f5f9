// Tile GEMM for small problems: ONE launch for any shape, layout and alignment.
//
// The tensor-core kernel needs 16-byte aligned rows for its TMA loads and a second launch to add
// split-K partials; on a problem of a few microseconds those extra launches are most of the time.
// Here a 64 x 64 output tile belongs to a thread-block cluster of CS CTAs (CS = 1, 2, 4, 8 or 16):
// CTA r of the cluster multiplies the r-th piece of the k range, the CS partial tiles are left in
// each CTA's shared memory, and every CTA then adds its 64 / CS rows of the tile over all ranks
// through distributed shared memory, in a fixed order (so the result does not depend on timing), rounds once
// and stores C.  No workspace.
//
// A tile whose k range is not shared with other CTAs (CS = 1, and every tile of a grouped launch) is, from K = 65 on, computed
// by two groups of four warps, each with stages, barrier and accumulators of its own: the groups take alternate stages (or, for a k range
// cut into pieces, alternate pieces), and their two sums are added at the end.  The pieces of a cluster are added the same
// way (even ones, odd ones, then the two sums), so a tile has the same bits whichever way its pieces were spread.
//
// Operands come in as 16-byte cp.async.cg copies into a ring of stages (64 x 64 of each operand per stage, kept in the
// operand's own orientation): the whole ring is in flight before the first wait.  A row is copied as the up to nine aligned
// 16-byte chunks that hold it, whatever its alignment; the copy's size operand zero-fills what lies beyond the matrix or the
// k range.  Rows off 16-byte boundaries are then shifted to the start of their line in place: a row's chunks are copied and
// shifted by eight lanes of one warp, so a warp-level barrier is enough for that.  ldmatrix (transposing when the operand's
// contiguous dimension is not k) feeds mma.sync.m16n8k16 with fp32 accumulation.
//
// What bounds it: the dependent chain of a stage (wait, shift, barrier, ldmatrix, MMAs), and for many tiles the shared-memory
// port (copy in, shift, ldmatrix).  Per-thread copy groups and no shifted stages beside the raw ones, against an mbarrier per
// stage that every thread's copies arrived on and a separate shifted buffer: 256 x 256 x 256 (CS = 4) 5.42 -> 4.60 us (3.97 with
// an SM per CTA), 64 x 1024 x 1024 7.16 -> 5.78 us; with two groups of warps in place of eight warps on one stage as well, 64 x 64 x 1024 by one CTA 19.0 -> 9.6 us.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>
#include <cuda_fp16.h>
#include <cuda_bf16.h>

#include "adapt_internal.h"
#include "aux_kernels.cuh"        // 16-bit conversions, fused-add parameters
#include "launch_pdl.cuh"
#include "ptx_sm100.cuh"
#include "skinny_gemm.cuh"      // mma_16816

namespace adapt {

constexpr int kClusterThreads = 256;
constexpr int kClusterTile = 64;        // output tile edge
constexpr int kClusterPitch = 72;       // 16-bit elements per staged row: 144 B, conflict-free for ldmatrix
constexpr int kClusterCPitch = 72;      // fp32 elements per row of the exchanged partial tile
static_assert(kClusterStageBytes == 2 * 64 * kClusterPitch * 2, "a stage is 64 rows of each operand");
static_assert(64 * kClusterCPitch * 4 <= kClusterStageBytes, "the partial tile reuses the first raw stage");

struct ClusterParams {
    const unsigned short* A;
    const unsigned short* B;
    unsigned short* C;
    int M, N, K;
    int64_t lda, ldb;            // leading dimensions in elements
    int P_n;                     // tiles along n
    int CS;                      // CTAs per cluster = pieces of the k range
    int k_per_cta;               // k values per CTA, a multiple of 16
    int share_log2, q;           // two-group tiles: the tile's pieces are shared by 2^share_log2 CTAs of a cluster, of which this is the q-th
    int ring;                    // raw stages in flight per CTA (1..kClusterMaxRing)
    int prefetch;                // L2 prefetch of the ring's stages ahead of the dependency wait
    int aligned;                 // bit 0: every row of A starts on a 16-byte boundary, bit 1: every row of B
    ReduceEpilogue ep;           // fused add (D == nullptr: none)
};

// Rows of a dense operand with `inner` contiguous elements all start on 16-byte boundaries.
__host__ __device__ inline bool rows_aligned16(const void* base, int64_t inner)
{
    return (((uintptr_t)base) & 15) == 0 && inner % 8 == 0;
}

__device__ __forceinline__ void ldmatrix_x4(uint32_t (&r)[4], uint32_t addr)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr));
}
__device__ __forceinline__ void ldmatrix_x4_trans(uint32_t (&r)[4], uint32_t addr)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr));
}
__device__ __forceinline__ uint32_t cl_rank()
{
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
// All threads of all CTAs of the cluster; release/acquire orders the shared-memory traffic around it.
__device__ __forceinline__ void cl_sync()
{
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ float4 cl_load4(uint32_t local_addr, uint32_t rank)
{
    uint32_t remote;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(remote) : "r"(local_addr), "r"(rank));
    float4 v;
    asm volatile("ld.shared::cluster.v4.f32 {%0,%1,%2,%3}, [%4];"
                 : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(remote) : "memory");
    return v;
}

// One row of an operand stage is 64 elements (128 bytes) that start `sh` bytes into a 16-byte chunk: chunk c
// of the row (c = 0..8) covers the row's bytes [16 c - sh, 16 c - sh + 16), of which those below 2 * nv exist;
// the rest is zero-filled by the copy (its size operand), so nothing needs masking later.  A chunk that holds
// an existing byte is always readable.
// A_KC: A is row-major (k contiguous); B_KC: B is column-major (k contiguous).
//
// SEQ: one CTA takes all CS pieces of the tile's k range, in two groups of warps; else it takes the piece of its cluster rank.
// SHARED: with share = 2^share_log2 > 1 CTAs to a SEQ tile, group g of CTA q takes the pieces q + share * g + 2 * share * i (i = 0, or 0 and 1) and keeps
// their sums apart; they meet in shared memory and are added over the cluster in the order of a tile of one CTA: even pieces, odd pieces, both.
template <bool A_KC, bool B_KC, bool BF16, bool SEQ, bool SHARED = false>
__device__ __forceinline__ void cluster_tile_body(const ClusterParams& p, int m0, int n0, unsigned char* s_dyn)
{
    constexpr int ROW = kClusterPitch * 2, OPND = 64 * ROW, STAGE = 2 * OPND;
    constexpr int NT = SEQ ? kClusterThreads / 2 : kClusterThreads;     // threads of a group
    constexpr int RP = NT / 8, NR = 64 / RP;                            // rows a group copies at a time; rows of an operand per thread
    constexpr int NJ = SEQ ? 4 : 2;                                     // a warp owns 32 x (8 NJ) outputs
    const int S = p.ring;
    const int tid = threadIdx.x, lane = tid & 31;
    const int grp = SEQ ? tid / NT : 0;
    const int gt = tid - grp * NT, warp = gt >> 5;
    unsigned char* ring_gen = s_dyn + grp * S * STAGE;                  // this group's ring
    const uint32_t ring0 = ptx::smem_u32(ring_gen);

    // ---- this group's stages: the first k value, the values of k left in its piece, and how both move on
    const uint32_t rank = !SEQ && p.CS > 1 ? cl_rank() : 0u;
    const int pieces = SEQ ? p.CS : 1;
    const int share_log2 = SHARED ? p.share_log2 : 0, share = 1 << share_log2, q_of_tile = SHARED ? p.q : 0;
    const bool by_stage = !SEQ || pieces == 1;                          // one piece: SEQ groups take alternate stages
    const int step_k = SEQ && by_stage ? 2 * kClusterKS : kClusterKS;
    const int spp = by_stage ? 1 : (p.k_per_cta + kClusterKS - 1) / kClusterKS;        // stages of a whole piece
    const int jump_k = 2 * share * p.k_per_cta - (spp - 1) * kClusterKS;        // from the last stage of a piece to this group's next one
    int next_piece = SEQ ? (by_stage ? 0 : ((grp << share_log2) + q_of_tile) * p.k_per_cta) : (int)rank * p.k_per_cta;
    const int k_begin = next_piece + (SEQ && by_stage ? grp * kClusterKS : 0);
    auto left_of = [&](int k) -> int { return min(p.K - k, p.k_per_cta); };             // ... of a piece that starts at k
    const int left0 = SEQ && by_stage ? p.K - k_begin : left_of(k_begin);
    auto stages_of = [&](int g) -> int {
        if (by_stage) { const int l = SEQ ? p.K - g * kClusterKS : left0; return l > 0 ? (l + step_k - 1) / step_k : 0; }
        const int first = (g << share_log2) + q_of_tile;                // first, first + 2 * share, ...; the very last piece may be short
        const int n = (pieces - first + 2 * share - 1) >> (share_log2 + 1), last = first + (n - 1) * 2 * share;
        return last == pieces - 1 ? (n - 1) * spp + (p.K - last * p.k_per_cta + kClusterKS - 1) / kClusterKS : n * spp;
    };
    const int n_stages = stages_of(grp);
    const bool al_a = p.aligned & 1, al_b = p.aligned & 2;

    // ---- copies.  Thread (r = gt / 8, c = gt % 8) copies chunk c of rows r, r + RP, ... of both operands, and, for rows off
    // 16-byte boundaries, the thread of chunk 7 also chunk 8.  RP rows and the steps between stages are multiples of 32 bytes,
    // so the misalignment is the same for all rows of a thread and in every stage.
    const int c = gt & 7, r = gt >> 3;
    const int nvs_a = min(64, p.M - m0), nvs_b = min(64, p.N - n0);    // elements of a row of an mn-contiguous stage, rows of the others
    const uintptr_t row_a = reinterpret_cast<uintptr_t>(p.A) + (uintptr_t)((A_KC ? (int64_t)(m0 + r) * p.lda + k_begin : (int64_t)(k_begin + r) * p.lda + m0) * 2);
    const uintptr_t row_b = reinterpret_cast<uintptr_t>(p.B) + (uintptr_t)((B_KC ? (int64_t)(n0 + r) * p.ldb + k_begin : (int64_t)(k_begin + r) * p.ldb + n0) * 2);
    const int sh_a = (int)(row_a & 15), sh_b = (int)(row_b & 15);
    const char* src_a = reinterpret_cast<const char*>(row_a - sh_a) + 16 * c;
    const char* src_b = reinterpret_cast<const char*>(row_b - sh_b) + 16 * c;
    const int64_t rows_a = RP * p.lda * 2, rows_b = RP * p.ldb * 2;    // bytes from a row of this thread to its next
    const int64_t unit_a = A_KC ? 2 : 2 * p.lda, unit_b = B_KC ? 2 : 2 * p.ldb;         // bytes per k value
    // bytes of chunk ch that exist in a row of nv elements
    auto chunk_bytes = [](int nv, int sh, int ch) -> int { return max(0, min(16, 2 * nv + sh - 16 * ch)); };
    // Ahead of the wait for the kernel before this one on the stream: ask L2 for the lines of the ring's stages (hints
    // only; the copies proper come after the wait), so that the trip to memory overlaps the previous kernel's tail.
    if (p.prefetch && (c == 0 || c == 7)) {
        const int ns = min(S, by_stage ? n_stages : min(n_stages, spp));
        const int64_t off_a = c == 7 ? sh_a : 0, off_b = c == 7 ? sh_b : 0;             // the row's first and its last line
#pragma unroll
        for (int j = 0; j < NR; ++j) {
            const int row = r + RP * j;
            for (int s = 0; s < ns; ++s) {
                const int left = left0 - s * step_k;
                if ((A_KC ? row < nvs_a && 8 * c < left : row < left && 8 * c < nvs_a)) ptx::prefetch_l2(src_a + j * rows_a + (int64_t)s * step_k * unit_a + off_a);
                if ((B_KC ? row < nvs_b && 8 * c < left : row < left && 8 * c < nvs_b)) ptx::prefetch_l2(src_b + j * rows_b + (int64_t)s * step_k * unit_b + off_b);
            }
        }
    }
    pdl_wait();
    auto copy16 = [](uint32_t dst, const char* from, int bytes) {
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(from), "r"(bytes) : "memory");
    };
    auto commit = []() { asm volatile("cp.async.commit_group;" ::: "memory"); };
    int is_left = left0, is_next = next_piece;                          // the stage issued next
    auto issue_stage = [&](int slot) {
        const int kv = min(64, is_left);
        const uint32_t dst = ring0 + (uint32_t)(slot * STAGE + r * ROW + 16 * c);
        auto rows = [&](bool kc, const char* src, int64_t pitch, int nvs, int sh, bool al, uint32_t d) {
            const int b = chunk_bytes(kc ? kv : nvs, sh, c), b8 = chunk_bytes(kc ? kv : nvs, sh, 8), n = kc ? nvs : kv;
#pragma unroll
            for (int j = 0; j < NR; ++j) {
                // rows beyond M or N feed outputs that are not stored and are left as they are; k rows beyond the range are zeros
                const bool exists = r + RP * j < n;
                if (kc && !exists) continue;
                copy16(d + (uint32_t)(j * RP * ROW), src + j * pitch, exists ? b : 0);
                if (!al && c == 7) copy16(d + (uint32_t)(j * RP * ROW + 16), src + j * pitch + 16, exists ? b8 : 0);
            }
        };
        rows(A_KC, src_a, rows_a, nvs_a, sh_a, al_a, dst);
        rows(B_KC, src_b, rows_b, nvs_b, sh_b, al_b, dst + (uint32_t)OPND);
        is_left -= step_k;
        int move = step_k;
        if (!by_stage && is_left <= 0) {                                // on to this group's next piece
            move = jump_k;
            is_next += 2 * share * p.k_per_cta;
            is_left = left_of(is_next);
        }
        src_a += unit_a * move;
        src_b += unit_b * move;
    };

    // ---- shift of an operand off 16-byte boundaries, in place: the 16 bytes of chunk c start sh bytes into the raw chunk; three
    // 8-byte reads from the 8-byte boundary below hold them.  All reads of a row come before its writes (the row's eight lanes
    // belong to one warp).
    auto shift_operand = [&](int op, int sh, int slot) {
        unsigned char* at = ring_gen + slot * STAGE + op * OPND + r * ROW + 16 * c;
        const bool odd = sh & 4;
        const uint32_t sel = 0x3210u + 0x1111u * (uint32_t)(sh & 3);               // byte shift 0 or 2 inside a word pair
        uint4 out[NR];
#pragma unroll
        for (int j = 0; j < NR; ++j) {
            const uint2* w = reinterpret_cast<const uint2*>(at + j * RP * ROW + (sh & 8));
            const uint2 w0 = w[0], w1 = w[1], w2 = w[2];
            const uint32_t v0 = odd ? w0.y : w0.x, v1 = odd ? w1.x : w0.y, v2 = odd ? w1.y : w1.x, v3 = odd ? w2.x : w1.y, v4 = odd ? w2.y : w2.x;
            out[j] = make_uint4(__byte_perm(v0, v1, sel), __byte_perm(v1, v2, sel), __byte_perm(v2, v3, sel), __byte_perm(v3, v4, sel));
        }
        __syncwarp();
#pragma unroll
        for (int j = 0; j < NR; ++j) *reinterpret_cast<uint4*>(at + j * RP * ROW) = out[j];
    };

    const int m_w = (warp & 1) * 32, n_w = (warp >> 1) * (8 * NJ);
    const int g = lane >> 2, t = lane & 3;
    const int lj = lane >> 3, lr = lane & 7;      // ldmatrix: this lane addresses row lr of matrix lj
    // byte offsets of this lane's ldmatrix row inside a stage, for k step 0
    // A stored [m][k]: matrices (m 0-7, k 0-7), (m 8-15, k 0-7), (m 0-7, k 8-15), (m 8-15, k 8-15); stored [k][m]: the same four, transposed
    const uint32_t off_a = A_KC ? (uint32_t)((m_w + (lj & 1) * 8 + lr) * ROW + (lj >> 1) * 16) : (uint32_t)(((lj >> 1) * 8 + lr) * ROW + (m_w + (lj & 1) * 8) * 2);
    // B stored [n][k]: matrices (n 0-7, k 0-7), (n 0-7, k 8-15), (n 8-15, k 0-7), (n 8-15, k 8-15); stored [k][n]: transposed
    const uint32_t off_b = (uint32_t)OPND + (B_KC ? (uint32_t)((n_w + (lj >> 1) * 8 + lr) * ROW + (lj & 1) * 16) : (uint32_t)(((lj & 1) * 8 + lr) * ROW + (n_w + (lj >> 1) * 8) * 2));
    float acc[2][NJ][4], tot[2][NJ][4];           // the sum of the piece at hand; SEQ: of this group's pieces before it
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < NJ; ++j)
#pragma unroll
            for (int e = 0; e < 4; ++e) acc[i][j][e] = tot[i][j][e] = 0.f;

    for (int s = 0; s < S; ++s) {
        if (s < n_stages) issue_stage(s);
        commit();
    }
    // A slot is free once the group has met again after the MMAs that read it, so its refill is issued one iteration later: S - 2
    // copy groups may still be under way when a stage is needed (a ring of one stage is never refilled).
    int slot = 0, left = left0;
    for (int s = 0; s < n_stages; ++s) {
        switch (S) {
            case 1: case 2: asm volatile("cp.async.wait_group 0;" ::: "memory"); break;
            case 3: asm volatile("cp.async.wait_group 1;" ::: "memory"); break;
            case 4: asm volatile("cp.async.wait_group 2;" ::: "memory"); break;
            case 5: asm volatile("cp.async.wait_group 3;" ::: "memory"); break;
            default: asm volatile("cp.async.wait_group 4;" ::: "memory"); break;
        }
        __syncwarp();                   // this warp's rows have landed
        if (!al_a) shift_operand(0, sh_a, slot);
        if (!al_b) shift_operand(1, sh_b, slot);
        if (!SEQ) __syncthreads();
        else if (grp == 0) asm volatile("bar.sync 1, %0;" ::"n"(NT) : "memory");
        else asm volatile("bar.sync 2, %0;" ::"n"(NT) : "memory");
        // now the whole stage is in place; every warp of the group is past the MMAs of stage s - 1
        const uint32_t base = ring0 + (uint32_t)(slot * STAGE);
        auto load_step = [&](int i, uint32_t (&fa)[2][4], uint32_t (&fb)[NJ / 2][4]) {
#pragma unroll
            for (int mi = 0; mi < 2; ++mi) {
                if (A_KC) ldmatrix_x4(fa[mi], base + off_a + (uint32_t)(16 * mi * ROW + 32 * i));
                else ldmatrix_x4_trans(fa[mi], base + off_a + (uint32_t)(32 * mi + 16 * i * ROW));
            }
#pragma unroll
            for (int nj = 0; nj < NJ / 2; ++nj) {
                if (B_KC) ldmatrix_x4(fb[nj], base + off_b + (uint32_t)(16 * nj * ROW + 32 * i));
                else ldmatrix_x4_trans(fb[nj], base + off_b + (uint32_t)(32 * nj + 16 * i * ROW));
            }
        };
        auto mma_step = [&](uint32_t (&fa)[2][4], uint32_t (&fb)[NJ / 2][4]) {
#pragma unroll
            for (int mi = 0; mi < 2; ++mi)
#pragma unroll
                for (int nj = 0; nj < NJ; ++nj)
                    mma_16816<BF16>(acc[mi][nj], fa[mi][0], fa[mi][1], fa[mi][2], fa[mi][3], fb[nj >> 1][2 * (nj & 1)], fb[nj >> 1][2 * (nj & 1) + 1]);
        };
        // the first fragments, the copies of the refill while they are under way, then the MMAs
        uint32_t fa[2][2][4], fb[2][NJ / 2][4];
        load_step(0, fa[0], fb[0]);
        if (s > 0) {
            if (s - 1 + S < n_stages) issue_stage(slot > 0 ? slot - 1 : S - 1);
            commit();
        }
        if (left >= kClusterKS) {       // a full stage: the next step's fragments are under way during a step's MMAs
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                if (i < 3) load_step(i + 1, fa[(i + 1) & 1], fb[(i + 1) & 1]);
                mma_step(fa[i & 1], fb[i & 1]);
            }
        } else {
            mma_step(fa[0], fb[0]);
            for (int i = 1; 16 * i < left; ++i) {
                load_step(i, fa[0], fb[0]);
                mma_step(fa[0], fb[0]);
            }
        }
        if (++slot == S) slot = 0;
        left -= step_k;
        if (!by_stage && left <= 0) {
            if (!SHARED || share == 1 || s + 1 < n_stages || n_stages <= spp) {     // (shared tiles: a second piece stays in acc)
#pragma unroll
                for (int i = 0; i < 2; ++i)
#pragma unroll
                    for (int j = 0; j < NJ; ++j)
#pragma unroll
                        for (int e = 0; e < 4; ++e) { tot[i][j][e] += acc[i][j][e]; acc[i][j][e] = 0.f; }
            }
            next_piece += 2 * share * p.k_per_cta;
            left = left_of(next_piece);
        }
    }
    // the fused add: alpha * sum + beta * D in fp32, before the cast
    auto finish = [&](float v, int m, int n) -> float { return fused_add(p.ep, v, m, n, p.N, BF16 ? 1 : 0); };

    // rounds and stores this thread's accumulators, or (both) the half of them that its group stores with the other group's sums
    // added from shared memory; a lane holds pairs of neighbouring columns
    auto store_direct = [&](bool both, const float* other) {
#pragma unroll
        for (int mi = 0; mi < 2; ++mi) {
            if (both && mi != grp) continue;
#pragma unroll
            for (int nj = 0; nj < NJ; ++nj)
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int row = m_w + 16 * mi + g + 8 * h, col = n_w + 8 * nj + 2 * t;
                    const int m = m0 + row, n = n0 + col;
                    if (m >= p.M || n >= p.N) continue;
                    float2 v = make_float2(acc[mi][nj][2 * h], acc[mi][nj][2 * h + 1]);
                    if (both) {
                        const float2 o = *reinterpret_cast<const float2*>(&other[row * kClusterCPitch + col]);
                        v.x += o.x;
                        v.y += o.y;
                    }
                    const unsigned short lo16 = float_to_16(finish(v.x, m, n), BF16 ? 1 : 0);
                    const unsigned short hi16 = n + 1 < p.N ? float_to_16(finish(v.y, m, n + 1), BF16 ? 1 : 0) : 0;
                    unsigned short* dst = p.C + (int64_t)m * p.N + n;
                    if (n + 1 < p.N && (reinterpret_cast<uintptr_t>(dst) & 3) == 0) {
                        *reinterpret_cast<uint32_t*>(dst) = (uint32_t)lo16 | ((uint32_t)hi16 << 16);
                    } else {
                        dst[0] = lo16;
                        if (n + 1 < p.N) dst[1] = hi16;
                    }
                }
        }
    };

    // four neighbouring outputs, rounded and stored
    auto store4 = [&](int m, int n, const float (&o)[4]) {
        unsigned short* dst = p.C + (int64_t)m * p.N + n;
        unsigned short h[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) h[j] = n + j < p.N ? float_to_16(finish(o[j], m, n + j), BF16 ? 1 : 0) : 0;
        if (n + 4 <= p.N && (reinterpret_cast<uintptr_t>(dst) & 7) == 0) {
            *reinterpret_cast<uint2*>(dst) = make_uint2((uint32_t)h[0] | ((uint32_t)h[1] << 16), (uint32_t)h[2] | ((uint32_t)h[3] << 16));
        } else {
#pragma unroll
            for (int j = 0; j < 4; ++j)
                if (n + j < p.N) dst[j] = h[j];
        }
    };

    if (SHARED && share > 1) {
        // piece q + share * g + 2 * share * i of this CTA is buffer g + 2 i: the sums of a group's first piece are in tot, a second one's in acc
        auto put = [&](int buffer, const float (&v)[2][NJ][4]) {
            float* s = reinterpret_cast<float*>(s_dyn + buffer * kClusterStageBytes);
#pragma unroll
            for (int mi = 0; mi < 2; ++mi)
#pragma unroll
                for (int nj = 0; nj < NJ; ++nj)
#pragma unroll
                    for (int h = 0; h < 2; ++h)
                        *reinterpret_cast<float2*>(&s[(m_w + 16 * mi + g + 8 * h) * kClusterCPitch + n_w + 8 * nj + 2 * t]) = make_float2(v[mi][nj][2 * h], v[mi][nj][2 * h + 1]);
        };
        __syncthreads();
        put(grp, tot);
        if (n_stages > spp) put(grp + 2, acc);
        cl_sync();
        const uint32_t base_rank = cl_rank() - (uint32_t)p.q;
        const int rows_mine = kClusterTile >> p.share_log2;
        for (int e = tid; e < rows_mine * 16; e += kClusterThreads) {
            const int row = p.q * rows_mine + (e >> 4), col = (e & 15) * 4;
            const int m = m0 + row, n = n0 + col;
            if (m >= p.M || n >= p.N) continue;
            float4 sum[2] = {make_float4(0.f, 0.f, 0.f, 0.f), make_float4(0.f, 0.f, 0.f, 0.f)};
            const uint32_t addr = ptx::smem_u32(s_dyn) + (uint32_t)(row * kClusterCPitch + col) * 4u;
            for (int pc0 = 0; pc0 < pieces; pc0 += 4) {        // four remote reads in flight (pieces: 4, 8 or 16)
                float4 v[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) v[j] = cl_load4(addr + (uint32_t)(((pc0 + j) >> p.share_log2) * kClusterStageBytes), base_rank + (uint32_t)((pc0 + j) & (share - 1)));
#pragma unroll
                for (int j = 0; j < 4; ++j) { sum[j & 1].x += v[j].x; sum[j & 1].y += v[j].y; sum[j & 1].z += v[j].z; sum[j & 1].w += v[j].w; }
            }
            const float o[4] = {sum[0].x + sum[1].x, sum[0].y + sum[1].y, sum[0].z + sum[1].z, sum[0].w + sum[1].w};
            store4(m, n, o);
        }
        cl_sync();                                             // no CTA leaves while a peer still reads its sums
        return;
    }
    if (SEQ) {
        // The two groups' sums: each group adds and stores half of its warps' rows (the 16 x 32 blocks mi = group) and hands the other
        // half over through shared memory.  With nothing on the second group's side the first one stores all.
        if (!by_stage) {
#pragma unroll
            for (int i = 0; i < 2; ++i)
#pragma unroll
                for (int j = 0; j < NJ; ++j)
#pragma unroll
                    for (int e = 0; e < 4; ++e) acc[i][j][e] = tot[i][j][e];
        }
        const bool both = stages_of(1) > 0;
        float* sC = reinterpret_cast<float*>(s_dyn);       // [64 x 72]: row blocks of 32 hold 16 rows for either group
        if (both) {
            __syncthreads();
#pragma unroll
            for (int mi = 0; mi < 2; ++mi) {
                if (mi == grp) continue;
#pragma unroll
                for (int nj = 0; nj < NJ; ++nj)
#pragma unroll
                    for (int h = 0; h < 2; ++h)
                        *reinterpret_cast<float2*>(&sC[(m_w + 16 * mi + g + 8 * h) * kClusterCPitch + n_w + 8 * nj + 2 * t]) =
                            make_float2(acc[mi][nj][2 * h], acc[mi][nj][2 * h + 1]);
            }
            __syncthreads();
        } else if (grp != 0) {
            return;
        }
        store_direct(both, sC);
        return;
    }
    if (p.CS == 1) {                    // (K <= 64: one stage, all eight warps on it)
        store_direct(false, nullptr);
        return;
    }

    // the CTA's partial tile, fp32, into its own shared memory
    float* sC = reinterpret_cast<float*>(s_dyn);
    __syncthreads();
#pragma unroll
    for (int mi = 0; mi < 2; ++mi)
#pragma unroll
        for (int nj = 0; nj < NJ; ++nj)
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int row = m_w + 16 * mi + g + 8 * h, col = n_w + 8 * nj + 2 * t;
                *reinterpret_cast<float2*>(&sC[row * kClusterCPitch + col]) = make_float2(acc[mi][nj][2 * h], acc[mi][nj][2 * h + 1]);
            }
    cl_sync();

    // rank r adds rows [r * 64 / CS, (r + 1) * 64 / CS) over the even ranks and over the odd ones, both ascending, adds the two and stores
    const int rows_mine = kClusterTile / p.CS;
    for (int e = tid; e < rows_mine * 16; e += kClusterThreads) {
        const int row = (int)rank * rows_mine + (e >> 4), col = (e & 15) * 4;
        const int m = m0 + row, n = n0 + col;
        if (m >= p.M || n >= p.N) continue;
        float4 sum[2] = {make_float4(0.f, 0.f, 0.f, 0.f), make_float4(0.f, 0.f, 0.f, 0.f)};
        const uint32_t addr = (uint32_t)__cvta_generic_to_shared(&sC[row * kClusterCPitch + col]);
        for (int q0 = 0; q0 < p.CS; q0 += 4) {             // four remote reads in flight
            float4 v[4];
#pragma unroll
            for (int q = 0; q < 4; ++q)
                if (q0 + q < p.CS) v[q] = cl_load4(addr, (uint32_t)(q0 + q));
#pragma unroll
            for (int q = 0; q < 4; ++q)
                if (q0 + q < p.CS) { sum[q & 1].x += v[q].x; sum[q & 1].y += v[q].y; sum[q & 1].z += v[q].z; sum[q & 1].w += v[q].w; }
        }
        const float o[4] = {sum[0].x + sum[1].x, sum[0].y + sum[1].y, sum[0].z + sum[1].z, sum[0].w + sum[1].w};
        store4(m, n, o);
    }
    // no CTA may leave while a peer still reads its partial tile
    cl_sync();
}

template <bool A_KC, bool B_KC, bool BF16, bool SEQ>
__global__ void __launch_bounds__(kClusterThreads, 2)
cluster_gemm_kernel(const ClusterParams p)
{
    extern __shared__ __align__(128) unsigned char s_dyn[];
    pdl_launch_dependents();
    const int tile = (int)(blockIdx.x / (unsigned)p.CS);
    cluster_tile_body<A_KC, B_KC, BF16, SEQ>(p, (tile / p.P_n) * kClusterTile, (tile % p.P_n) * kClusterTile, s_dyn);
}

typedef void (*ClusterKernel)(const ClusterParams);

template <bool SEQ>
inline ClusterKernel cluster_pick(bool a_kc, bool b_kc, bool bf16)
{
    if (bf16) {
        if (a_kc) return b_kc ? cluster_gemm_kernel<true, true, true, SEQ> : cluster_gemm_kernel<true, false, true, SEQ>;
        return b_kc ? cluster_gemm_kernel<false, true, true, SEQ> : cluster_gemm_kernel<false, false, true, SEQ>;
    }
    if (a_kc) return b_kc ? cluster_gemm_kernel<true, true, false, SEQ> : cluster_gemm_kernel<true, false, false, SEQ>;
    return b_kc ? cluster_gemm_kernel<false, true, false, SEQ> : cluster_gemm_kernel<false, false, false, SEQ>;
}

// Once per device: the launches need more than the default dynamic shared memory.
inline cudaError_t cluster_set_attributes()
{
    for (int v = 0; v < 8; ++v) {
        const ClusterKernel split = cluster_pick<false>(v & 1, v & 2, v & 4), alone = cluster_pick<true>(v & 1, v & 2, v & 4);
        cudaError_t e = cudaFuncSetAttribute(split, cudaFuncAttributeMaxDynamicSharedMemorySize, kClusterAloneBytes);
        if (e != cudaSuccess) return e;
        e = cudaFuncSetAttribute(split, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);   // clusters of 16
        if (e != cudaSuccess) return e;
        e = cudaFuncSetAttribute(alone, cudaFuncAttributeMaxDynamicSharedMemorySize, cluster_seq_smem_bytes(kClusterSeqRing));
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

// Largest cluster size (16, 8, 4, 2, 1) of which the device runs at least one cluster with an SM per CTA.
inline int cluster_max_size()
{
    for (int cs = 16; cs > 1; cs >>= 1) {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3((unsigned)cs, 1, 1);
        cfg.blockDim = dim3(kClusterThreads, 1, 1);
        cfg.dynamicSmemBytes = (size_t)kClusterAloneBytes;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = (unsigned)cs;
        attr[0].val.clusterDim.y = 1;
        attr[0].val.clusterDim.z = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        int n = 0;
        if (cudaOccupancyMaxActiveClusters(&n, (const void*)cluster_pick<false>(true, false, false), &cfg) == cudaSuccess && n >= 1) return cs;
        (void)cudaGetLastError();
    }
    return 1;
}

// Host launcher.  c.cluster = CS; c.stages = depth of the raw ring; the grid is CS CTAs per tile, the cluster spans blockIdx.x.
inline adapt_status_t launch_cluster(const Shape& s, const Config& c, const void* A, const void* B, void* C,
                                     int n_sm, cudaStream_t stream, int prefetch = 1, const ReduceEpilogue* epi = nullptr)
{
    ClusterParams p;
    p.A = (const unsigned short*)A;
    p.B = (const unsigned short*)B;
    p.C = (unsigned short*)C;
    p.M = (int)s.M; p.N = (int)s.N; p.K = (int)s.K;
    const bool a_kc = s.layoutA == ADAPT_ROW_MAJOR, b_kc = s.layoutB == ADAPT_COL_MAJOR;
    p.lda = a_kc ? s.K : s.M;
    p.ldb = b_kc ? s.K : s.N;
    p.P_n = c.P_n;
    p.CS = c.cluster;
    p.k_per_cta = (int)round_up(ceil_div(s.K, c.cluster), 16);
    const bool seq = cluster_two_groups(s.K, c.cluster);
    p.share_log2 = p.q = 0;
    p.ring = seq ? cluster_alone_ring(s.K) : c.stages;
    p.prefetch = prefetch;
    p.aligned = (rows_aligned16(A, p.lda) ? 1 : 0) | (rows_aligned16(B, p.ldb) ? 2 : 0);
    p.ep = epi ? *epi : no_epilogue();
    cudaLaunchConfig_t cfg;
    memset(&cfg, 0, sizeof(cfg));
    cfg.gridDim = dim3((unsigned)((int64_t)c.P_m * c.P_n * c.cluster), 1, 1);
    cfg.blockDim = dim3(kClusterThreads, 1, 1);
    cfg.dynamicSmemBytes = (size_t)(seq ? cluster_seq_smem_bytes(p.ring) : cluster_launch_bytes(p.ring, c.cluster, (int64_t)c.P_m * c.P_n, n_sm));
    cfg.stream = stream;
    cudaLaunchAttribute attr[2];
    pdl_attribute(&attr[0]);
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = (unsigned)c.cluster;
    attr[1].val.clusterDim.y = 1;
    attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = c.cluster > 1 ? 2 : 1;
    void* args[1] = {&p};
    const size_t arg_bytes[1] = {sizeof(p)};
    if (launch_exc(&cfg, (const void*)(seq ? cluster_pick<true>(a_kc, b_kc, s.dtype != 0) : cluster_pick<false>(a_kc, b_kc, s.dtype != 0)), args, arg_bytes, 1) != cudaSuccess) return ADAPT_ERR_CUDA;
    return ADAPT_OK;
}

}  // namespace adapt
