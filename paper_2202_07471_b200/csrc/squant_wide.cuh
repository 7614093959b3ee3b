// Output channels that are too long for a group of the grouped kernel: 1x1 rows of more than 8 K weights
// get a thread block of 512 threads each, and channels that do not fit one thread block's shared memory a
// cluster of 2, 4 or 8 of them, each with a contiguous run of the channel's kernels.  What a channel needs
// as a whole travels through distributed shared memory (plain loads from the other thread blocks' shared
// memory; no multicast anywhere): absmax, error sum, the counts of SQuant-C's search and the short lists
// of its candidates, which every thread block collects for itself, so that all of them take the same
// decisions without a leader.
//
// Channels this wide can hold 2^16 and more kernels, the size from which the one element that sits on
// the edge of the clip range (|w/s| a shade above qmax) can make it into a top-k; they run the bodies
// that check every candidate against the range, as in the CPU definition: an element whose flipped code
// would leave the range is no candidate.
//
// With the bodies of squant_rows.cuh and squant_conv.cuh, two thread blocks per multiprocessor where the channel
// can be cut that small: 256 rows of 100,352, 128 of 65,541 and 64x8192x3x3 690 -> 224 us on a B200.
#pragma once

#include "squant_conv.cuh"

namespace sq {

constexpr int kWideMaxCluster = 8;
// Longest row of the row kernel (164 KB of shared memory); up to here it was laid out and compared with the staged
// body of the grouped kernel.  Longer rows that fit one thread block still take that body, which is the slower one
// there: 1024 rows of 32,772 weights 318 us against 99 in this kernel, of 40,000 480 against 116, 16 rows of 40,000 83 against 22.
constexpr int kRowBlockElems = 32768;

// Rows of more than 8 K weights, one thread block per output channel, two per multiprocessor.
__global__ void __launch_bounds__(kBlockThreads, 2)
squant_row_kernel(const __grid_constant__ LaunchTable tbl, int qmax, unsigned mode)
{
    extern __shared__ __align__(16) unsigned char smem[];
    const int item = blockIdx.x;
    int layer = 0;
#pragma unroll 1
    for (int step = tbl.top_step; step > 0; step >>= 1)
        if (layer + step < tbl.n_layers && tbl.first_item[layer + step] <= item) layer += step;
    const LayerDesc &L = tbl.layers[layer];
    Group G;
    G.g = kBlockThreads;
    G.t = threadIdx.x;
    G.bar = 0;
    SQ_DBG(row_bytes(kBlockThreads, L.off_vi, kBlock) <= static_cast<int>(dynamic_smem_bytes()), 10);
    if (L.sin) row_body<true, kBlock>(L, item - tbl.first_item[layer], G, smem, qmax, mode, true);
    else row_body<false, kBlock>(L, item - tbl.first_item[layer], G, smem, qmax, mode, true);
}

// Shared memory of one of a cluster's thread blocks that has `kpc` kernels of K weights.
__host__ __device__ inline long long wide_bytes(int kpc, int K)
{
    const long long nk = static_cast<long long>(kpc) * K;
    if (nk > (1 << 20)) return 1ll << 30;
    return K == 1 ? row_bytes(kBlockThreads, (kpc + 6) >> 2, kCluster) : conv_bytes(kBlockThreads, static_cast<int>(nk), K, kCluster);
}

// One output channel per cluster; grid = channels * cluster size.  L.off_vi = vectors of a run (1x1).
__global__ void __launch_bounds__(kBlockThreads, 2)
squant_wide_kernel(const LayerDesc L, int qmax, unsigned mode, int kpc)
{
    extern __shared__ __align__(16) unsigned char smem[];
    cg::cluster_group cluster = cg::this_cluster();
    const int C = static_cast<int>(cluster.num_blocks()), rank = static_cast<int>(cluster.block_rank());
    const int m = static_cast<int>(blockIdx.x) / C;
    const int n0 = min(rank * kpc, L.N), nloc = min(L.N - n0, kpc);   // this thread block's kernels
    Group G;
    G.g = kBlockThreads;
    G.t = threadIdx.x;
    G.bar = 0;
    SQ_DBG(wide_bytes(kpc, L.K) <= static_cast<long long>(dynamic_smem_bytes()), 11);
    const bool range = L.sin != nullptr || L.N >= 65536;   // a flip can be barred by the clip range
    if (L.K == 1) {
        if (range) row_body<true, kCluster>(L, m, G, smem, qmax, mode, true, n0, nloc);
        else row_body<false, kCluster>(L, m, G, smem, qmax, mode, true, n0, nloc);
    } else if (L.K == 9 && (mode & 2u)) {
        if (range) conv_body<9, true, kCluster>(L, m, G, smem, qmax, mode, n0, nloc);
        else conv_body<9, false, kCluster>(L, m, G, smem, qmax, mode, n0, nloc);
    } else {
        if (range) conv_body<0, true, kCluster>(L, m, G, smem, qmax, mode, n0, nloc);
        else conv_body<0, false, kCluster>(L, m, G, smem, qmax, mode, n0, nloc);
    }
    cluster.sync();   // no thread block leaves while another may still read its shared memory
}

}  // namespace sq
