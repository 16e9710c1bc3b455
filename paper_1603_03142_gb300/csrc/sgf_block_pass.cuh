// sgf_block_pass.cuh -- the block-convolution passes as kernels (one instance
// per pass, element type and single / batch form; included by sgf_block_fwd.cu
// and sgf_block_inv.cu).
#pragma once
#include "sgf_block.cuh"

namespace sgf {

template <typename T>
struct BlkBatch {
    const SolveArgs<T> *args;
    const BlkArgs<T> *blk;
    const int *prefix, *index;  // first CTA of every plan; its index in args and blk
    int plans;
    int round;  // of the inverse rows (single solves too)
};

template <typename T, int PASS, int LOGB>
__device__ __forceinline__ void blk_body(const SolveArgs<T> &a, const BlkArgs<T> &k, const BlkStage &s, int target,
                                         int blk, unsigned char *smem)
{
    if constexpr (PASS == BLK_ROWS)
        blk_rows_body<T, LOGB>(a, k, s, blk, (int)blockIdx.y, gridDim.y == 3 ? 1 : 3, smem);
    else if constexpr (PASS == BLK_COLS)
        blk_cols_body<T, LOGB>(k, s, blk, smem);
    else if constexpr (PASS == BLK_ICOLS)
        blk_icols_body<T, LOGB>(k, s, a.ncomp, blk, smem);
    else
        blk_irows_body<T, LOGB>(a, k, s, target, blk, smem);
}

// B from 16 (the smallest the host sends here) to 2048 (FP64: 1024).  One kernel
// for every B: the stages of a solve then share a launch per pass, and its 256
// threads hold 16 values each at every B.
template <typename T, int PASS, bool BATCH>
__global__ void __launch_bounds__(kBlkThreads, sizeof(T) == 8 ? 1 : 3)
    k_blk(const __grid_constant__ SolveArgs<T> a0, const __grid_constant__ BlkArgs<T> k0, BlkBatch<T> bt)
{
    extern __shared__ __align__(32) unsigned char smem_blk[];
    int blk = (int)blockIdx.x;
    const int pl = BATCH ? blk_plan<T>(bt.prefix, bt.plans, blk) : 0;
    if (BATCH)
        blk -= bt.prefix[pl];
    const int at = BATCH ? bt.index[pl] : 0;
    const SolveArgs<T> &a = BATCH ? bt.args[at] : a0;
    const BlkArgs<T> &k = BATCH ? bt.blk[at] : k0;
    int stage = 0, target = 0;
    if constexpr (PASS == BLK_IROWS) {
        int g = 0;
        while (g + 1 < k.segs[bt.round] && blk >= k.seg[bt.round][g + 1].blk)
            ++g;
        stage = k.seg[bt.round][g].stage;
        target = k.seg[bt.round][g].ti;
        blk -= k.seg[bt.round][g].blk;
    } else {
        stage = blk_stage<T>(k, PASS, blk);
    }
    const BlkStage &s = k.st[stage];
    switch (s.logB) {
    case 4: blk_body<T, PASS, 4>(a, k, s, target, blk, smem_blk); break;
    case 5: blk_body<T, PASS, 5>(a, k, s, target, blk, smem_blk); break;
    case 6: blk_body<T, PASS, 6>(a, k, s, target, blk, smem_blk); break;
    case 7: blk_body<T, PASS, 7>(a, k, s, target, blk, smem_blk); break;
    case 8: blk_body<T, PASS, 8>(a, k, s, target, blk, smem_blk); break;
    case 9: blk_body<T, PASS, 9>(a, k, s, target, blk, smem_blk); break;
    case 10: blk_body<T, PASS, 10>(a, k, s, target, blk, smem_blk); break;
    case 11:
        if constexpr (sizeof(T) == 4)
            blk_body<T, PASS, 11>(a, k, s, target, blk, smem_blk);
        break;
    default: break;
    }
}

// Dynamic shared memory of a pass: the largest over the block sizes.
template <typename T, int LOGB>
constexpr size_t blk_smem_b(int pass)
{
    using C = typename Cx<T>::C;
    const size_t tw = (((size_t)tw_layout(F16<LOGB>::twlen, 1 << LOGB).entries) * sizeof(C) + 15) & ~(size_t)15;
    return tw + blk_xbuf_bytes<T, LOGB>() + (pass == BLK_IROWS ? 2 * kBlkCells * sizeof(T) : 0) +
           (pass == BLK_ROWS || pass == BLK_IROWS ? BShape<LOGB>::G * sizeof(BlkSeq) : 0);
}
template <typename T>
constexpr size_t blk_smem(int pass)
{
    size_t m = 0;
    const size_t v[] = {blk_smem_b<T, 4>(pass), blk_smem_b<T, 5>(pass), blk_smem_b<T, 6>(pass),  blk_smem_b<T, 7>(pass),
                        blk_smem_b<T, 8>(pass), blk_smem_b<T, 9>(pass), blk_smem_b<T, 10>(pass), sizeof(T) == 4 ? blk_smem_b<T, 11>(pass) : 0};
    for (size_t x : v)
        m = x > m ? x : m;
    return m;
}

template <typename T, int PASS, bool BATCH>
cudaError_t blk_prepare_pass()
{
    return cudaFuncSetAttribute(k_blk<T, PASS, BATCH>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)blk_smem<T>(PASS));
}

template <typename T, int PASS, bool BATCH>
cudaError_t blk_launch(int blocks, const SolveArgs<T> &a, const BlkArgs<T> &k, const BlkBatch<T> &bt, cudaStream_t st)
{
    if (blocks <= 0)
        return cudaSuccess;
    // forward rows: the three fields of a CTA's rows one after the other, or a CTA each where the
    // launch would leave SMs without one (3 resident CTAs on each)
    const dim3 grid(blocks, PASS == BLK_ROWS && blocks < 3 * kSMs ? 3 : 1);
    k_blk<T, PASS, BATCH><<<grid, kBlkThreads, blk_smem<T>(PASS), st>>>(a, k, bt);
    return cudaGetLastError();
}

#define SGF_BLK_EXTERN(T, PASS)                                                                                    \
    extern template cudaError_t blk_prepare_pass<T, PASS, false>();                                               \
    extern template cudaError_t blk_prepare_pass<T, PASS, true>();                                                \
    extern template cudaError_t blk_launch<T, PASS, false>(int, const SolveArgs<T> &, const BlkArgs<T> &,          \
                                                           const BlkBatch<T> &, cudaStream_t);                    \
    extern template cudaError_t blk_launch<T, PASS, true>(int, const SolveArgs<T> &, const BlkArgs<T> &,           \
                                                          const BlkBatch<T> &, cudaStream_t);
SGF_BLK_EXTERN(float, BLK_ROWS)
SGF_BLK_EXTERN(float, BLK_COLS)
SGF_BLK_EXTERN(float, BLK_ICOLS)
SGF_BLK_EXTERN(float, BLK_IROWS)
SGF_BLK_EXTERN(double, BLK_ROWS)
SGF_BLK_EXTERN(double, BLK_COLS)
SGF_BLK_EXTERN(double, BLK_ICOLS)
SGF_BLK_EXTERN(double, BLK_IROWS)
#undef SGF_BLK_EXTERN

}  // namespace sgf
