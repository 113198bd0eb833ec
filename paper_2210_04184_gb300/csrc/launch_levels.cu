// Launchers of the latent pass on the compact state (k_levels.cuh) and of the conversions between
// its levels and the entry form: every (T, WT, K) instantiation, K = 1, 2.
#define FUSE_LAUNCH_DEFINITIONS
#include "launch.cuh"

namespace fuse {

template <typename F>
static void with_grid_k(int K, F&& f) {
    if (K == 1) f(std::integral_constant<int, 1>{});
    else f(std::integral_constant<int, 2>{});
}

template <typename T, typename WT>
void levels_launch(const LevelArgs<T, WT>& a, int K, dim3 grid, unsigned threads, size_t smem, cudaStream_t s) {
    with_grid_k(K, [&](auto k) { latent_levels_kernel<T, WT, decltype(k)::value><<<grid, threads, smem, s>>>(a); });
}

template <typename T, typename WT>
void levels_init_launch(const LevelArgs<T, WT>& a, int K, int kept, cudaStream_t s) {
    const size_t n = (size_t)a.H * a.W;
    const dim3 grid((unsigned)((n + 127) / 128), (unsigned)kept);
    with_grid_k(K, [&](auto k) {
        levels_init_kernel<T, decltype(k)::value><<<grid, 128, 0, s>>>(a.rec, a.masks, a.e, a.tab, n, a.Ls);
    });
}

template <typename T, typename WT>
void levels_batch_launch(const LevelArgs<T, WT>* args, const Segment* seg, int nseg, int K, unsigned blocks,
                         unsigned threads, size_t smem, cudaStream_t s) {
    with_grid_k(K, [&](auto k) {
        latent_levels_batch_kernel<T, WT, decltype(k)::value><<<blocks, threads, smem, s>>>(args, seg, nseg);
    });
}

template <typename T, typename WT>
void points_batch_launch(const LevelArgs<T, WT>* args, const Segment* seg, int nseg, int first, unsigned blocks,
                         cudaStream_t s) {
    points_batch_kernel<T, WT><<<blocks, 256, 0, s>>>(args, seg, nseg, first);
}

template <typename T, typename WT>
void points_launch(const LevelArgs<T, WT>& a, int first, cudaStream_t s) {
    const int rows = a.H * a.Ls;
    points_kernel<T><<<(unsigned)((rows + 7) / 8), 256, 0, s>>>(a.X, const_cast<LevelPoint<T>*>(a.pt), rows, a.W, a.S,
                                                               a.grid, first);
}

template <typename T, typename WT>
void levels_convert_launch(const LevelArgs<T, WT>& a, int K, int kept, int to_levels, int check, int* bad,
                           cudaStream_t s) {
    const dim3 grid((unsigned)(((size_t)a.H * a.W + 127) / 128), (unsigned)kept);
    with_grid_k(K, [&](auto k) {
        constexpr int KK = decltype(k)::value;
        if (to_levels) entries_to_levels_kernel<T, WT, KK><<<grid, 128, 0, s>>>(a, check, bad);
        else levels_to_entries_kernel<T, WT, KK><<<grid, 128, 0, s>>>(a);
    });
}

template <typename T, typename WT>
void level_table_launch(const WT* omega, code_t<T>* tab, int H, int W, int K, int S, int half, int kept, T coef,
                        const LatentGrid<T>* grid, cudaStream_t s) {
    const dim3 blocks((unsigned)(((size_t)H * W + 127) / 128), (unsigned)kept);
    with_grid_k(K, [&](auto k) {
        level_table_kernel<T, WT, decltype(k)::value><<<blocks, 128, 0, s>>>(omega, tab, H, W, S, half, coef, grid);
    });
}

template <typename T, typename WT>
void wmax_launch(const WT* w, size_t n, LatentGrid<T>* grid, T coef, cudaStream_t s) {
    wmax_kernel<T, WT><<<608, 256, 0, s>>>(w, n, grid);
    grid_kernel<T><<<1, 1, 0, s>>>(grid, coef);
}

template <typename T, typename WT>
cudaError_t levels_set_smem(int K, int bytes) {
    cudaError_t e = cudaSuccess;
    with_grid_k(K, [&](auto k) {
        constexpr int KK = decltype(k)::value;
        const auto A = cudaFuncAttributeMaxDynamicSharedMemorySize;
        e = cudaFuncSetAttribute(latent_levels_kernel<T, WT, KK>, A, bytes);
        if (e == cudaSuccess) e = cudaFuncSetAttribute(latent_levels_batch_kernel<T, WT, KK>, A, bytes);
        // 164 KB of shared memory per SM (72%), the rest L1: the events' scattered reads of the table and
        // the points gain more from L1 than the pass from two more blocks (24 tiles of 96 to 384, 40
        // iterations: 2.75 ms per pass, 2.91 with 196 or 228 KB, 4.0 with 132 KB)
        const auto P = cudaFuncAttributePreferredSharedMemoryCarveout;
        if (e == cudaSuccess) e = cudaFuncSetAttribute(latent_levels_kernel<T, WT, KK>, P, 72);
        if (e == cudaSuccess) e = cudaFuncSetAttribute(latent_levels_batch_kernel<T, WT, KK>, P, 72);
    });
    return e;
}

#define FUSE_LEVELS_INST(T, WT)                                                                                 \
    template void levels_launch<T, WT>(const LevelArgs<T, WT>&, int, dim3, unsigned, size_t, cudaStream_t);      \
    template void levels_batch_launch<T, WT>(const LevelArgs<T, WT>*, const Segment*, int, int, unsigned,        \
                                             unsigned, size_t, cudaStream_t);                                  \
    template void levels_init_launch<T, WT>(const LevelArgs<T, WT>&, int, int, cudaStream_t);                   \
    template void points_batch_launch<T, WT>(const LevelArgs<T, WT>*, const Segment*, int, int, unsigned,        \
                                             cudaStream_t);                                                    \
    template void points_launch<T, WT>(const LevelArgs<T, WT>&, int, cudaStream_t);                             \
    template void levels_convert_launch<T, WT>(const LevelArgs<T, WT>&, int, int, int, int, int*, cudaStream_t); \
    template void level_table_launch<T, WT>(const WT*, code_t<T>*, int, int, int, int, int, int, T,              \
                                            const LatentGrid<T>*, cudaStream_t);                               \
    template void wmax_launch<T, WT>(const WT*, size_t, LatentGrid<T>*, T, cudaStream_t);                                       \
    template cudaError_t levels_set_smem<T, WT>(int, int);

FUSE_LEVELS_INST(float, float)
FUSE_LEVELS_INST(float, __nv_bfloat16)
FUSE_LEVELS_INST(double, double)

}  // namespace fuse
