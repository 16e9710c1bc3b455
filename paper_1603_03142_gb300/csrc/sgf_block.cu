// sgf_block.cu -- the products of the block convolutions (see sgf_block.cuh)
// and the host side of their launches.
#include "sgf_block_pass.cuh"

namespace sgf {

// ------------------------------------------------------------------- mac
// Y_q,r(k) = sum over terms, units p and fields f of K_pq,f(k) X_p,f,r(k).  A
// warp takes 32 consecutive 16-byte pieces of the frequencies, QG target units
// and R right-hand sides (sources that share the kernel spectra), all sums in
// registers; the warps of a CTA are neighbouring target groups of the same
// frequencies, so the sources' values come from L1 after the first.  Every
// kernel value is read once per R right-hand sides, straight into registers:
// the kernel spectra are the traffic, and enough independent 16-byte loads are
// in flight to stream them.  The sum's order (term, p, f) does not depend on QG
// or R, and its multiply-adds are written out, so a nest gives the same forces
// alone and in a batch.
__device__ __forceinline__ void mac_add(float4 &s, const float4 &k, const float4 &x)
{
    s.x = fmaf(k.x, x.x, fmaf(-k.y, x.y, s.x));
    s.y = fmaf(k.x, x.y, fmaf(k.y, x.x, s.y));
    s.z = fmaf(k.z, x.z, fmaf(-k.w, x.w, s.z));
    s.w = fmaf(k.z, x.w, fmaf(k.w, x.z, s.w));
}
__device__ __forceinline__ void mac_add(double2 &s, const double2 &k, const double2 &x)
{
    s.x = fma(k.x, x.x, fma(-k.y, x.y, s.x));
    s.y = fma(k.x, x.y, fma(k.y, x.x, s.y));
}
__device__ __forceinline__ float4 ld_stream(const float4 *p)
{
    float4 v;
    asm("ld.global.nc.L1::no_allocate.v4.f32 {%0, %1, %2, %3}, [%4];"
        : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
        : "l"(p));
    return v;
}
__device__ __forceinline__ double2 ld_stream(const double2 *p)
{
    double2 v;
    asm("ld.global.nc.L1::no_allocate.v2.f64 {%0, %1}, [%2];" : "=d"(v.x), "=d"(v.y) : "l"(p));
    return v;
}

template <typename T> struct MacVec;
template <> struct MacVec<float> { using V = float4; static constexpr int E = 2; };
template <> struct MacVec<double> { using V = double2; static constexpr int E = 1; };

template <typename T>
struct MacArgs {
    const MacItem *items;
    const MacTerm *terms;
    const size_t *xo, *ao;
    const typename Cx<T>::C *spec, *x;
    typename Cx<T>::C *acc;
    int nitems;
};

template <typename T, int NC, int QG, int R>
__device__ __forceinline__ void mac_body(const MacArgs<T> &m, const MacItem &it, int tile, int q0, int lane)
{
    using V = typename MacVec<T>::V;
    constexpr int E = MacVec<T>::E;
    const int fv = tile * 32 + lane, FV = it.F / E;
    if (fv >= FV)
        return;
    V acc[QG][NC][R];
#pragma unroll
    for (int q = 0; q < QG; ++q)
#pragma unroll
        for (int c = 0; c < NC; ++c)
#pragma unroll
            for (int r = 0; r < R; ++r)
                acc[q][c][r] = V{};
    for (int tm = 0; tm < it.term_count; ++tm) {
        const MacTerm te = m.terms[it.term_begin + tm];
        const V *kb = reinterpret_cast<const V *>(m.spec + te.k_off + (size_t)q0 * te.sq) + fv;
        const V *xb[R];
#pragma unroll
        for (int r = 0; r < R; ++r)
            xb[r] = reinterpret_cast<const V *>(m.x + m.xo[te.x_begin + r]) + fv;
        const size_t sp = te.sp / E, sq = te.sq / E;
#pragma unroll (QG * R <= 2 ? 2 : 1)
        for (int p = 0; p < it.m2; ++p) {
#pragma unroll
            for (int f = 0; f < 3; ++f) {
                V xv[R];
#pragma unroll
                for (int r = 0; r < R; ++r)
                    xv[r] = __ldg(xb[r] + (size_t)(p * 3 + f) * FV);
#pragma unroll
                for (int q = 0; q < QG; ++q)
#pragma unroll
                    for (int c = 0; c < NC; ++c) {
                        const V kv = ld_stream(kb + p * sp + q * sq + (size_t)(c * 3 + f) * FV);
#pragma unroll
                        for (int r = 0; r < R; ++r)
                            mac_add(acc[q][c][r], kv, xv[r]);
                    }
            }
        }
    }
#pragma unroll
    for (int r = 0; r < R; ++r) {
        V *dst = reinterpret_cast<V *>(m.acc + m.ao[it.a_begin + r]) + fv;
#pragma unroll
        for (int q = 0; q < QG; ++q)
#pragma unroll
            for (int c = 0; c < NC; ++c)
                dst[(size_t)((q0 + q) * NC + c) * FV] = acc[q][c][r];
    }
}

template <typename T, int NC>
__global__ void __launch_bounds__(kBlkThreads, 2) k_blk_mac(MacArgs<T> m)
{
    int lo = 0, hi = m.nitems;  // the CTA's item
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (m.items[mid].blk_begin <= (int)blockIdx.x)
            lo = mid;
        else
            hi = mid;
    }
    const MacItem it = m.items[lo];
    const int lane = threadIdx.x & 31;
    const int w = ((int)blockIdx.x - it.blk_begin) * (kBlkThreads / 32) + (threadIdx.x >> 5);
    const int tile = w / it.nqg, q0 = (w - tile * it.nqg) * it.qg;
    if (tile >= it.tiles)
        return;
    if (it.rhs == 1) {
        if (it.qg == 4)
            mac_body<T, NC, 4, 1>(m, it, tile, q0, lane);
        else if (it.qg == 2)
            mac_body<T, NC, 2, 1>(m, it, tile, q0, lane);
        else
            mac_body<T, NC, 1, 1>(m, it, tile, q0, lane);
    } else if (it.rhs == 2) {
        if (it.qg == 2)
            mac_body<T, NC, 2, 2>(m, it, tile, q0, lane);
        else
            mac_body<T, NC, 1, 2>(m, it, tile, q0, lane);
    } else if (it.rhs == 3) {
        mac_body<T, NC, 1, 3>(m, it, tile, q0, lane);
    } else {
        mac_body<T, NC, 1, 4>(m, it, tile, q0, lane);
    }
}

template <typename T>
cudaError_t launch_blk_mac(int blocks, const MacItem *items, int nitems, const MacTerm *terms, const size_t *xo,
                           const size_t *ao, const void *spec, const void *x, void *acc, int ncomp, cudaStream_t st)
{
    using C = typename Cx<T>::C;
    if (blocks <= 0)
        return cudaSuccess;
    const MacArgs<T> m{items, terms, xo, ao, static_cast<const C *>(spec), static_cast<const C *>(x),
                       static_cast<C *>(acc), nitems};
    if (ncomp == 2)
        k_blk_mac<T, 2><<<blocks, kBlkThreads, 0, st>>>(m);
    else
        k_blk_mac<T, 1><<<blocks, kBlkThreads, 0, st>>>(m);
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_blk_pass(int pass, int round, int blocks, const SolveArgs<T> &a, const BlkArgs<T> &k,
                            cudaStream_t st)
{
    BlkBatch<T> bt{};
    bt.round = round;
    switch (pass) {
    case BLK_ROWS: return blk_launch<T, BLK_ROWS, false>(blocks, a, k, bt, st);
    case BLK_COLS: return blk_launch<T, BLK_COLS, false>(blocks, a, k, bt, st);
    case BLK_ICOLS: return blk_launch<T, BLK_ICOLS, false>(blocks, a, k, bt, st);
    case BLK_IROWS: return blk_launch<T, BLK_IROWS, false>(blocks, a, k, bt, st);
    default: return cudaErrorInvalidValue;
    }
}

template <typename T>
cudaError_t launch_blk_pass_batch(int pass, int round, int blocks, int plans, const int *prefix,
                                  const int *index, const SolveArgs<T> *da, const BlkArgs<T> *dk, cudaStream_t st)
{
    const BlkBatch<T> bt{da, dk, prefix, index, plans, round};
    const SolveArgs<T> a{};
    const BlkArgs<T> k{};
    switch (pass) {
    case BLK_ROWS: return blk_launch<T, BLK_ROWS, true>(blocks, a, k, bt, st);
    case BLK_COLS: return blk_launch<T, BLK_COLS, true>(blocks, a, k, bt, st);
    case BLK_ICOLS: return blk_launch<T, BLK_ICOLS, true>(blocks, a, k, bt, st);
    case BLK_IROWS: return blk_launch<T, BLK_IROWS, true>(blocks, a, k, bt, st);
    default: return cudaErrorInvalidValue;
    }
}

template <typename T>
cudaError_t blk_prepare()
{
    cudaError_t e;
    if ((e = blk_prepare_pass<T, BLK_ROWS, false>()) != cudaSuccess ||
        (e = blk_prepare_pass<T, BLK_ROWS, true>()) != cudaSuccess ||
        (e = blk_prepare_pass<T, BLK_COLS, false>()) != cudaSuccess ||
        (e = blk_prepare_pass<T, BLK_COLS, true>()) != cudaSuccess ||
        (e = blk_prepare_pass<T, BLK_ICOLS, false>()) != cudaSuccess ||
        (e = blk_prepare_pass<T, BLK_ICOLS, true>()) != cudaSuccess ||
        (e = blk_prepare_pass<T, BLK_IROWS, false>()) != cudaSuccess ||
        (e = blk_prepare_pass<T, BLK_IROWS, true>()) != cudaSuccess)
        return e;
    return cudaSuccess;
}

int blk_blocks(int pass, const BlkStage &s, int ncomp)
{
    const long long B = 1LL << s.logB, m2 = (long long)s.m * s.m, G = kBlkThreads / (2 * (B / 16));
    long long seqs = 0;
    switch (pass) {
    case BLK_ROWS: seqs = s.src_count * m2 * (B / 2); break;
    case BLK_COLS: seqs = s.src_count * m2 * 3 * (B + 1); break;
    case BLK_ICOLS: seqs = (s.tgt_count[0] + s.tgt_count[1]) * m2 * ncomp * (B + 1); break;
    case BLK_IROWS: seqs = m2 * ncomp * (B / 2); break;
    default: break;
    }
    return (int)((seqs + G - 1) / G);
}

#define SGF_BLK_INST(T)                                                                                            \
    template cudaError_t launch_blk_pass<T>(int, int, int, const SolveArgs<T> &, const BlkArgs<T> &, cudaStream_t);     \
    template cudaError_t launch_blk_pass_batch<T>(int, int, int, int, const int *, const int *,                \
                                                  const SolveArgs<T> *, const BlkArgs<T> *, cudaStream_t);         \
    template cudaError_t launch_blk_mac<T>(int, const MacItem *, int, const MacTerm *, const size_t *,             \
                                           const size_t *, const void *, const void *, void *, int, cudaStream_t); \
    template cudaError_t blk_prepare<T>();
SGF_BLK_INST(float)
SGF_BLK_INST(double)

}  // namespace sgf
