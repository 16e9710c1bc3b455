// sgf_block_fwd.cu -- forward passes of the block convolutions (sgf_block.cuh).
#include "sgf_block_pass.cuh"

namespace sgf {
#define SGF_BLK_FWD(T, PASS)                                                                                       \
    template cudaError_t blk_prepare_pass<T, PASS, false>();                                                      \
    template cudaError_t blk_prepare_pass<T, PASS, true>();                                                       \
    template cudaError_t blk_launch<T, PASS, false>(int, const SolveArgs<T> &, const BlkArgs<T> &,                 \
                                                    const BlkBatch<T> &, cudaStream_t);                           \
    template cudaError_t blk_launch<T, PASS, true>(int, const SolveArgs<T> &, const BlkArgs<T> &,                  \
                                                   const BlkBatch<T> &, cudaStream_t);
SGF_BLK_FWD(float, BLK_ROWS)
SGF_BLK_FWD(float, BLK_COLS)
SGF_BLK_FWD(double, BLK_ROWS)
SGF_BLK_FWD(double, BLK_COLS)
}  // namespace sgf
