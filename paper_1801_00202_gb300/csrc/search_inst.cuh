// Launch wrappers for one instantiation (words per lane) of the search kernel;
// each search_kN.cu instantiates one so the library compiles in parallel.
#pragma once

#include "search_impl.cuh"

namespace mce {

// The instance for blocks of `threads` threads (listing has the short one).
template <int K, int PIVOT, bool LIST>
auto search_kernel_for(unsigned threads)
{
    if constexpr (LIST) return search_kernel<K, PIVOT, true, kShortThreads>;
    else
        return threads <= kShortThreads ? search_kernel<K, PIVOT, false, kShortThreads>
                                        : search_kernel<K, PIVOT, false, kLaunchThreads>;
}

template <int K, int PIVOT, bool LIST>
cudaError_t run_search_t(const SearchParams &prm, const LaunchShape &sh, cudaStream_t s)
{
    cudaError_t e = cudaSuccess;
    if (!prm.prepared) {
        const unsigned *rp = nullptr;
        if (PIVOT == MCE_PIVOT_TOMITA && prm.n > 0) {
            unsigned *dst = &prm.ctl->pad4[0];
            root_tomita_pivot_kernel<0><<<1, 1024, 0, s>>>(prm.rows, prm.n, prm.wp, dst);
            rp = dst;
        }
        search_init_kernel<0><<<64, 256, 0, s>>>(prm);
        e = cudaGetLastError();
        if (e != cudaSuccess) return e;
        e = prm.part ? launch_part_frames(prm, rp, s) : launch_seed_children(prm, rp, s);
        if (e != cudaSuccess) return e;
    }
    auto kernel = search_kernel_for<K, PIVOT, LIST>(sh.threads);
    e = kernel_smem_setup((const void *)kernel, sh.threads <= kShortThreads);
    if (e != cudaSuccess) return e;
    kernel<<<sh.blocks, sh.threads, sh.smem, s>>>(prm);
    return cudaGetLastError();
}

template <int K, int PIVOT, bool LIST>
cudaError_t occupancy_t(int threads, size_t smem, int *blocks_per_sm)
{
    auto kernel = search_kernel_for<K, PIVOT, LIST>((unsigned)threads);
    cudaError_t e = kernel_smem_setup((const void *)kernel, (unsigned)threads <= kShortThreads);
    if (e != cudaSuccess) return e;
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, kernel, threads, smem);
}

// The instance for batch blocks of `threads` threads.  Blocks of up to 256 run
// several to an SM and want the smaller register count: three of 256 threads
// instead of two (the outer loop's subproblems, G(10000, 0.005) in all 6.3 ->
// 5.8 ms).
template <int K, int PIVOT>
auto batch_kernel_for(unsigned threads)
{
    return threads > kShortThreads / 2u && threads <= kShortThreads ? batch_kernel<K, PIVOT, kShortThreads>
                                                                   : batch_kernel<K, PIVOT, kLaunchThreads>;
}

template <int K, int PIVOT>
cudaError_t run_batch_t(const BatchParams &bp, const LaunchShape &sh, cudaStream_t s)
{
    batch_kernel_for<K, PIVOT>(sh.threads)<<<sh.blocks, sh.threads, sh.smem, s>>>(bp);
    return cudaGetLastError();
}

template <int K, int PIVOT>
cudaError_t batch_occupancy_t(int threads, size_t smem, int *blocks_per_sm)
{
    auto kernel = batch_kernel_for<K, PIVOT>((unsigned)threads);
    cudaError_t e = kernel_smem_setup((const void *)kernel);
    if (e != cudaSuccess) return e;
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, kernel, threads, smem);
}

// The listing variant (LIST) has no batched form.
template <int K, int PIVOT, bool LIST>
SearchImpl impl_t()
{
    if constexpr (LIST)
        return {run_search_t<K, PIVOT, true>, occupancy_t<K, PIVOT, true>, nullptr, nullptr};
    else
        return {run_search_t<K, PIVOT, false>, occupancy_t<K, PIVOT, false>, run_batch_t<K, PIVOT>,
                batch_occupancy_t<K, PIVOT>};
}

template <int K, bool LIST>
SearchImpl pick(int pivot)
{
    switch (pivot) {
    case MCE_PIVOT_GREEDY: return impl_t<K, MCE_PIVOT_GREEDY, LIST>();
    case MCE_PIVOT_GREEDY_TX: return impl_t<K, MCE_PIVOT_GREEDY_TX, LIST>();
    case MCE_PIVOT_TOMITA: return impl_t<K, MCE_PIVOT_TOMITA, LIST>();
    default: return {nullptr, nullptr, nullptr, nullptr};
    }
}

}  // namespace mce

#define MCE_DEFINE_SEARCH(K) \
    namespace mce { SearchImpl search_impl_##K(int pivot) { return pick<K, false>(pivot); } }
#define MCE_DEFINE_SEARCH_LIST(K) \
    namespace mce { SearchImpl search_list_impl_##K(int pivot) { return pick<K, true>(pivot); } }
