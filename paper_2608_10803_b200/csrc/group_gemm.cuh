// Many small GEMMs in ONE launch: the lists of adapt_matmul_batch and the entries of adapt_matmul_strided_batch.
//
// A GEMM of a few microseconds is mostly launch, first trip to memory and drain; one launch each leaves the chip idle
// between them (48 layers of 16 .. 1024 a side: 110 us on four streams, two microseconds a call, for 16 MB of operands).
// Here the 64 x 64 tiles of all entries run side by side, one per CTA.  An entry keeps the arithmetic of its own plan:
//   pieces > 0: the one-launch cluster kernel's tiles.  The CTA walks the plan's pieces of the k range and adds
//               their sums in the same order: the bits of the call made alone, where each piece has a CTA of its own.
//               The tiles with the longest chains are shared by two or four CTAs of a cluster (group_share).  (Clusters of four for
//               every tile, the pieces of one group of warps spread over them, took 53 us for those 48 layers, one CTA per tile 40 us.)
//   pieces = 0: the CUDA-core kernel's tiles (a few 16-k steps).
// The list travels in the kernel's parameters, so nothing is copied to the device and the launch can be captured.
#pragma once

#include "aux_kernels.cuh"
#include "cluster_gemm.cuh"
#include "group_plan.h"

namespace adapt {

enum { kGroupPlain = 0, kGroupShort, kGroupShared };

// What bounds it: latency with two CTAs per SM.  Those 48 layers take 31.0 us, 21.7 for the 47 that share the launch and 8.7 for the one
// with a launch of its own (each by itself); the 762 tiles are 2.6 rounds of CTAs whose longest chain is 8 stages (0.33 us per aligned 64 k
// values and group of warps, 0.6 off 16-byte boundaries).  Profiled: 13.7 warps per SM (128 registers a thread), issue slots 35 % used,
// stalls on fixed latencies and shared memory, DRAM 4 %.  The deepest entries come first and the ring is no deeper than the list needs.
// FORM kGroupShort: every item has K <= 64 in one piece (one stage): no two-group tiles, so fewer registers and three CTAs per SM instead of two
// (96 products of 128 x 128 x 64 in one launch: 6.6 us with the general kernel, 4.4 with this one, 266 as 96 launches).
// kGroupShared: clusters, with the tiles of some items shared by several CTAs (an instantiation of its own: the other lists' tiles took 4 % longer with
// this code beside theirs).
template <bool A_KC, bool B_KC, bool BF16, int FORM>
__global__ void __launch_bounds__(kClusterThreads, FORM == kGroupShort ? 3 : 2)
group_gemm_kernel(const __grid_constant__ GroupParams p)
{
    extern __shared__ __align__(128) unsigned char s_dyn[];
    pdl_launch_dependents();
    const int t_all = (int)blockIdx.x;
    GroupPlace at;
    const bool work = group_place(p, t_all, at);
    if (FORM == kGroupShared && !work) {                    // a CTA that only fills a cluster
        if (t_all < p.sync_ctas) { cl_sync(); cl_sync(); }  // ... of shared tiles: both of their barriers
        return;
    }
    const GroupItem& it = p.item[at.item];
    const int entry = at.entry, tile = at.tile;
    const int m0 = (tile / it.P_n) * kClusterTile, n0 = (tile % it.P_n) * kClusterTile;
    const unsigned short* A = it.A + entry * p.sa;
    const unsigned short* B = it.B + entry * p.sb;
    unsigned short* C = it.C + entry * p.sc;
    if (it.pieces == 0) {
        SimtParams q;
        q.M = it.M; q.N = it.N; q.K = it.K;
        q.a_sm = A_KC ? it.K : 1; q.a_sk = A_KC ? 1 : it.M;
        q.b_sk = B_KC ? 1 : it.N; q.b_sn = B_KC ? it.K : 1;
        q.P_n = it.P_n; q.P_k = 1; q.kb_per_split = (it.K + 15) / 16;
        q.Np = 0; q.dtype = BF16 ? 1 : 0; q.prefetch = 0;
        q.C = C; q.partial = nullptr; q.ep.D = nullptr;
        SimtStage* sm = reinterpret_cast<SimtStage*>(s_dyn);
        simt_tile_body<false>(A, B, q, m0, n0, 0, sm[0], sm[1]);
        return;
    }
    ClusterParams q;
    q.A = A; q.B = B; q.C = C;
    q.M = it.M; q.N = it.N; q.K = it.K;
    q.lda = A_KC ? it.K : it.M;
    q.ldb = B_KC ? it.K : it.N;
    q.P_n = it.P_n;
    q.CS = it.pieces;
    q.k_per_cta = it.k_per_piece;
    q.ring = p.ring;
    q.prefetch = p.prefetch;
    q.share_log2 = it.share_log2; q.q = at.q;
    q.aligned = (rows_aligned16(A, q.lda) ? 1 : 0) | (rows_aligned16(B, q.ldb) ? 2 : 0);
    q.ep.D = nullptr;
    cluster_tile_body<A_KC, B_KC, BF16, FORM != kGroupShort, FORM == kGroupShared>(q, m0, n0, s_dyn);
}

typedef void (*GroupKernel)(const GroupParams);

template <int FORM>
inline GroupKernel group_pick(bool a_kc, bool b_kc, bool bf16)
{
    if (bf16) {
        if (a_kc) return b_kc ? group_gemm_kernel<true, true, true, FORM> : group_gemm_kernel<true, false, true, FORM>;
        return b_kc ? group_gemm_kernel<false, true, true, FORM> : group_gemm_kernel<false, false, true, FORM>;
    }
    if (a_kc) return b_kc ? group_gemm_kernel<true, true, false, FORM> : group_gemm_kernel<true, false, false, FORM>;
    return b_kc ? group_gemm_kernel<false, true, false, FORM> : group_gemm_kernel<false, false, false, FORM>;
}

inline cudaError_t group_set_attributes()
{
    for (int v = 0; v < 8; ++v) {
        for (GroupKernel k : {group_pick<kGroupPlain>(v & 1, v & 2, v & 4), group_pick<kGroupShared>(v & 1, v & 2, v & 4)}) {
            const cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, cluster_seq_smem_bytes(kClusterSeqRing));
            if (e != cudaSuccess) return e;
        }
    }
    return cudaSuccess;
}

// One launch; p holds the items (group_add) and the strides.
inline cudaError_t launch_group(GroupParams& p, bool a_kc, bool b_kc, cudaStream_t stream)
{
    const GroupForm form = group_form(p);
    cudaLaunchConfig_t cfg;
    memset(&cfg, 0, sizeof(cfg));
    cfg.gridDim = dim3((unsigned)group_grid(p), 1, 1);
    cfg.blockDim = dim3(kClusterThreads, 1, 1);
    cfg.dynamicSmemBytes = (size_t)form.smem_bytes;
    cfg.stream = stream;
    cudaLaunchAttribute attr[2];
    pdl_attribute(&attr[0]);
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = kGroupCluster;
    attr[1].val.clusterDim.y = 1;
    attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = p.sync_ctas > 0 ? 2 : 1;
    void* args[1] = {&p};
    const size_t bytes[1] = {sizeof(p)};
    const bool bf16 = p.dtype != 0;
    const GroupKernel k = p.sync_ctas > 0 ? group_pick<kGroupShared>(a_kc, b_kc, bf16) : form.short_k ? group_pick<kGroupShort>(a_kc, b_kc, bf16)
                                                                                                     : group_pick<kGroupPlain>(a_kc, b_kc, bf16);
    return launch_exc(&cfg, (const void*)k, args, bytes, 1);
}

}  // namespace adapt
