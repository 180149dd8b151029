// zc_kdec.cu -- width scan (decode-tile offsets) and decompression kernels.
#define ZC_DECODE_KERNELS
#include "zc_launch.h"

namespace zc {

cudaError_t launch_wscan(const Launch& P, unsigned grid, cudaStream_t s)
{
    return launch_after(k_wscan, grid, NTHREADS, 0, s, P);
}

cudaError_t launch_tile_map(const Item* items, unsigned n_items, unsigned total_tiles,
                            unsigned* map, cudaStream_t s, bool by_chunk, bool dependent)
{
    const unsigned grid = (total_tiles + NTHREADS - 1) / NTHREADS;
    if (dependent) return launch_after(k_tile_map, grid, NTHREADS, 0, s, items, n_items, total_tiles, map, by_chunk ? 1 : 0);
    k_tile_map<<<grid, NTHREADS, 0, s>>>(items, n_items, total_tiles, map, by_chunk ? 1 : 0);
    return cudaGetLastError();
}

cudaError_t launch_group(Item* items, unsigned n_items, unsigned* part, unsigned* map,
                         cudaStream_t s)
{
    const unsigned nblk = (n_items + GROUP_T - 1) / GROUP_T;
    const cudaError_t e1 = launch_after(k_group_count, nblk, GROUP_T, 0, s, (const Item*)items, n_items, part);
    if (e1 != cudaSuccess) return e1;
    const cudaError_t e2 = launch_after(k_group_scan, 1, 1024, 0, s, part, nblk);
    if (e2 != cudaSuccess) return e2;
    return launch_after(k_group_place, nblk, GROUP_T, 0, s, items, n_items, (const unsigned*)part, map);
}

template <int DU>
static cudaError_t decompress_u(const Launch& P, unsigned grid, cudaStream_t s, bool after_wscan)
{
    if (P.items != nullptr) {
        const cudaError_t e = smem_limit<k_decompress<true, true, DU>>(DEC_SMEM_BYTES);
        if (e != cudaSuccess) return e;
        return launch_after(k_decompress<true, true, DU>, grid, NTHREADS, DEC_SMEM_BYTES, s, P);
    }
    if (!after_wscan) {  // (small streams only: 64-row units)
        const cudaError_t e = smem_limit<k_decompress<false, true, DEC_U>>(DEC_SMEM_BYTES);
        if (e != cudaSuccess) return e;
        return launch_after(k_decompress<false, true, DEC_U>, grid, NTHREADS, DEC_SMEM_BYTES, s, P);
    }
    const cudaError_t e = smem_limit<k_decompress<false, false, DU>>(DEC_SMEM_BYTES);
    if (e != cudaSuccess) return e;
    // launched dependent on the width scan just before it on the stream: its
    // CTAs read their headers while the scan still runs
    return launch_after(k_decompress<false, false, DU>, grid, NTHREADS, DEC_SMEM_BYTES, s, P);
}

cudaError_t launch_decompress(const Launch& P, unsigned grid, cudaStream_t s, bool after_wscan)
{
    return P.urows == DEC_U_LARGE ? decompress_u<DEC_U_LARGE>(P, grid, s, after_wscan)
                                  : decompress_u<DEC_U>(P, grid, s, after_wscan);
}

}  // namespace zc
