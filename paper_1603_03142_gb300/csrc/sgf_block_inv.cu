// sgf_block_inv.cu -- inverse passes of the block convolutions (sgf_block.cuh).
#include "sgf_block_pass.cuh"

namespace sgf {
#define SGF_BLK_INV(T, PASS)                                                                                       \
    template cudaError_t blk_prepare_pass<T, PASS, false>();                                                      \
    template cudaError_t blk_prepare_pass<T, PASS, true>();                                                       \
    template cudaError_t blk_launch<T, PASS, false>(int, const SolveArgs<T> &, const BlkArgs<T> &,                 \
                                                    const BlkBatch<T> &, cudaStream_t);                           \
    template cudaError_t blk_launch<T, PASS, true>(int, const SolveArgs<T> &, const BlkArgs<T> &,                  \
                                                   const BlkBatch<T> &, cudaStream_t);
SGF_BLK_INV(float, BLK_ICOLS)
SGF_BLK_INV(float, BLK_IROWS)
SGF_BLK_INV(double, BLK_ICOLS)
SGF_BLK_INV(double, BLK_IROWS)
}  // namespace sgf
