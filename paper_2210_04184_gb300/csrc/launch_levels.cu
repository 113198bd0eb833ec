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
void levels_init_launch(const LevelArgs<T, WT>& a, int K, int kept, int clear, cudaStream_t s) {
    const size_t n = (size_t)a.H * a.W;
    const dim3 grid((unsigned)((n + 127) / 128), (unsigned)kept);
    with_grid_k(K, [&](auto k) {
        levels_init_kernel<T, decltype(k)::value><<<grid, 128, 0, s>>>(a.rec, a.masks, a.e, a.tab, n, a.Ls, clear,
                                                                        a.ctl);
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
                                                               a.grid, first, a.ctl);
}

// Runs of pixels over the kept offsets, and blocks of a launch over them: as many as fit the device at
// once, `resident` per SM, so that a launch that finds nothing to do ends in microseconds.
template <typename T, typename WT>
static int window_runs(const LevelArgs<T, WT>& a, int kept, int run) {
    return kept * (int)(((size_t)a.H * a.W + run - 1) / run);
}
static unsigned window_blocks(int runs, int nsm, int resident) {
    return (unsigned)(runs < resident * nsm ? runs : resident * nsm);
}

template <typename T, typename WT>
void levels_to_entries_launch(const LevelArgs<T, WT>& now, const LevelArgs<T, WT>& old, int K, int kept, int nsm, int want,
                              cudaStream_t s) {
    with_grid_k(K, [&](auto k) {
        constexpr int KK = decltype(k)::value;
        constexpr int R = window_run<T, KK>();
        const int runs = window_runs(now, kept, R);
        const unsigned blocks = window_blocks(runs, nsm, window_resident<T, KK>());
        levels_to_entries_kernel<T, WT, KK><<<blocks, R, 0, s>>>(now, old, runs, want);
    });
}

template <typename T, typename WT>
void save_entries_launch(const LevelArgs<T, WT>& now, const LevelArgs<T, WT>& old, T* out, int K, int kept, int nsm,
                         cudaStream_t s) {
    with_grid_k(K, [&](auto k) {
        constexpr int KK = decltype(k)::value;
        constexpr int R = window_run<T, KK>();
        const int runs = window_runs(now, kept, R);
        const unsigned blocks = window_blocks(runs, nsm, window_resident<T, KK>());
        const size_t words = (size_t)kept * (2 * KK + 1) * (2 * KK + 1) * now.Ls * now.H * now.W;
        save_entries_kernel<T, WT, KK><<<blocks, R, 0, s>>>(now, old, out,
                                                                                                        words, runs);
    });
}

template <typename T, typename WT>
void entries_check_launch(const LevelArgs<T, WT>& a, int K, int kept, int nsm, cudaStream_t s) {
    with_grid_k(K, [&](auto k) {
        constexpr int KK = decltype(k)::value;
        constexpr int R = window_run<T, KK>();
        const int runs = window_runs(a, kept, R);
        const unsigned blocks = window_blocks(runs, nsm, window_resident<T, KK>());
        entries_check_kernel<T, WT, KK><<<blocks, R, 0, s>>>(a, runs);
    });
}

template <typename T, typename WT>
void entries_to_levels_launch(const LevelArgs<T, WT>& a, int K, int kept, int nsm, cudaStream_t s) {
    with_grid_k(K, [&](auto k) {
        constexpr int KK = decltype(k)::value;
        constexpr int R = window_run<T, KK>();
        const int runs = window_runs(a, kept, R);
        const unsigned blocks = window_blocks(runs, nsm, window_resident<T, KK>());
        entries_to_levels_kernel<T, WT, KK><<<blocks, R, 0, s>>>(a, runs);
    });
}

template <typename T, typename WT>
void level_table_launch(const LevelArgs<T, WT>& a, int K, int kept, int nsm, cudaStream_t s) {
    const int runs = window_runs(a, kept, 128);
    with_grid_k(K, [&](auto k) {
        level_table_kernel<T, WT, decltype(k)::value><<<window_blocks(runs, nsm, 16), 128, 0, s>>>(
            a.omega, const_cast<code_t<T>*>(a.tab), a.H, a.W, a.S, a.half, a.coef, a.grid, runs, a.ctl);
    });
}

template <typename T>
void weights_change_launch(const void* omega, void* was, size_t bytes, LatentGrid<T>* grid, LatentCtl* ctl, int nsm,
                           cudaStream_t s) {
    const size_t words = was ? bytes / 16 : 0, need = (words + 1023) / 1024;
    const unsigned blocks = (unsigned)(need < 1 ? 1 : need < (size_t)4 * nsm ? need : (size_t)4 * nsm);
    weights_change_kernel<T><<<blocks, 256, 0, s>>>((const uint4*)omega, (uint4*)was, words, grid, ctl);
}

template <typename T>
void latent_begin_launch(const BeginArgs<T>* a, int n, cudaStream_t s) {
    for (int i = 0; i < n; i += BeginBatch<T>::kMost) {
        BeginBatch<T> batch;
        const int m = n - i < BeginBatch<T>::kMost ? n - i : BeginBatch<T>::kMost;
        int blocks = 1;
        for (int j = 0; j < m; ++j) {
            batch.a[j] = a[i + j];
            const int k = begin_blocks(a[i + j].count);
            blocks = k > blocks ? k : blocks;
        }
        latent_begin_kernel<T><<<dim3((unsigned)blocks, (unsigned)m), 1024, 0, s>>>(batch);
    }
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
    template void levels_init_launch<T, WT>(const LevelArgs<T, WT>&, int, int, int, cudaStream_t);              \
    template void points_batch_launch<T, WT>(const LevelArgs<T, WT>*, const Segment*, int, int, unsigned,        \
                                             cudaStream_t);                                                    \
    template void points_launch<T, WT>(const LevelArgs<T, WT>&, int, cudaStream_t);                             \
    template void levels_to_entries_launch<T, WT>(const LevelArgs<T, WT>&, const LevelArgs<T, WT>&, int, int, int, \
                                                  int, cudaStream_t);                                          \
    template void save_entries_launch<T, WT>(const LevelArgs<T, WT>&, const LevelArgs<T, WT>&, T*, int, int, int, \
                                             cudaStream_t);                                                    \
    template void entries_check_launch<T, WT>(const LevelArgs<T, WT>&, int, int, int, cudaStream_t);            \
    template void entries_to_levels_launch<T, WT>(const LevelArgs<T, WT>&, int, int, int, cudaStream_t);        \
    template void level_table_launch<T, WT>(const LevelArgs<T, WT>&, int, int, int, cudaStream_t);              \
    template void wmax_launch<T, WT>(const WT*, size_t, LatentGrid<T>*, T, cudaStream_t);                                       \
    template cudaError_t levels_set_smem<T, WT>(int, int);

FUSE_LEVELS_INST(float, float)
FUSE_LEVELS_INST(float, __nv_bfloat16)
FUSE_LEVELS_INST(double, double)
template void weights_change_launch<float>(const void*, void*, size_t, LatentGrid<float>*, LatentCtl*, int, cudaStream_t);
template void latent_begin_launch<float>(const BeginArgs<float>*, int, cudaStream_t);
template void latent_begin_launch<double>(const BeginArgs<double>*, int, cudaStream_t);
template void weights_change_launch<double>(const void*, void*, size_t, LatentGrid<double>*, LatentCtl*, int, cudaStream_t);

}  // namespace fuse
