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

// Products of pairs that are mirror-symmetric in x, y or both.  A kernel block at the
// mirrored units is, per frequency, the loaded one at the mirrored ky, its conjugate
// there, or its own conjugate (y, x, both axes), times the table's parity.  So a
// lane takes a frequency (kx, ky) and its mirror (kx, -ky), and every kernel value
// serves its 2 or 4 mirror images: targets run over one half (quarter) of the units,
// and half (a quarter) of the spectra are read.  Centred nests, the most common kind,
// are symmetric in both axes: 1024^2 3 levels 627 -> 290 us for the products (5.2 of
// 6.8 TB/s, held by load latency at 16 warps per SM: 128 registers, 8 bytes spilled),
// 256^2, symmetric in y, 52 -> 38.
// FP32: in FP64 the multiply-adds bound the products, not the spectra.
template <int NC>
__device__ constexpr bool mac_odd(bool y, int c, int f)
{
    // tables (K0x, Kxx, Kxy), (K0y, Kyx, Kyy): odd in x where u or v - v_c times x enters
    // once, likewise y; potential (P0, Px, Py)
    return NC == 1 ? (y ? f == 2 : f == 1) : y ? (c == 0 ? f == 2 : f != 2) : (c == 0 ? f != 1 : f == 1);
}
template <bool CONJ, bool NEG, typename C>
__device__ __forceinline__ void mac_img(C &s, const C &k, const C &x)
{
    const auto kr = NEG ? -k.x : k.x;
    const auto ki = NEG != CONJ ? -k.y : k.y;
    s.x = fma(kr, x.x, fma(-ki, x.y, s.x));
    s.y = fma(kr, x.y, fma(ki, x.x, s.y));
}
// Image (MX, MY) of kernel values ka at (kx, ky), kb at (kx, -ky) for table (c, f).
template <int NC, bool MX, bool MY, typename C>
__device__ __forceinline__ void mac_pair(C &sa, C &sb, const C &ka, const C &kb, const C &xa, const C &xb, int c, int f)
{
    const bool neg = (MX && mac_odd<NC>(false, c, f)) != (MY && mac_odd<NC>(true, c, f));
    // mirrored ky on one axis alone; conjugate where x is mirrored
    const C &k1 = MX != MY ? kb : ka, &k2 = MX != MY ? ka : kb;
    if (neg) {
        mac_img<MX, true>(sa, k1, xa);
        mac_img<MX, true>(sb, k2, xb);
    } else {
        mac_img<MX, false>(sa, k1, xa);
        mac_img<MX, false>(sb, k2, xb);
    }
}
__device__ __forceinline__ float2 ld_stream(const float2 *p)
{
    float2 v;
    asm("ld.global.nc.L1::no_allocate.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "l"(p));
    return v;
}

template <typename T, int NC, int SYM, int R>
__device__ __forceinline__ void mac_sym_body(const MacArgs<T> &m, const MacItem &it, int tile, int unit, int lane)
{
    using C = typename Cx<T>::C;
    constexpr bool SX = (SYM & kMirrorX) != 0, SY = (SYM & kMirrorY) != 0;
    constexpr int IM = (SX ? 2 : 1) * (SY ? 2 : 1);
    const int B = 1 << it.logB, mm = 1 << it.logm, idx = tile * 32 + lane;
    if (idx >= (B + 1) * (B + 1))
        return;
    // pair j of column kx: ky = 2 j (j <= B/2) or 2 j' + 1, and its mirror within the same parity half
    const int kx = idx / (B + 1), j = idx - kx * (B + 1);
    const int odd = j > B / 2 ? 1 : 0, ja = odd ? j - (B / 2 + 1) : j;
    const size_t fa = (size_t)kx * (2 * B) + odd * B + ja;
    const size_t fb = (size_t)kx * (2 * B) + odd * B + (odd ? B - 1 - ja : (B - ja) & (B - 1));
    const size_t F = (size_t)it.F;
    // unit u mirrored by image e (bit 0: x if SX, else y; bit 1: y)
    auto mirror = [&](int u, int e) {
        const int x = u & (mm - 1), y = u >> it.logm;
        const bool mx = SX && (e & 1), my = SY && (SX ? (e & 2) != 0 : (e & 1) != 0);
        return ((my ? mm - 1 - y : y) << it.logm) + (mx ? mm - 1 - x : x);
    };
    const int lq = SX ? it.logm - 1 : it.logm;  // base units: the lower half in the mirrored axes
    const int q = ((unit >> lq) << it.logm) + (unit & ((1 << lq) - 1));
    C sa[IM][NC][R], sb[IM][NC][R];
#pragma unroll
    for (int e = 0; e < IM; ++e)
#pragma unroll
        for (int c = 0; c < NC; ++c)
#pragma unroll
            for (int r = 0; r < R; ++r)
                sa[e][c][r] = sb[e][c][r] = hmk<C>(T(0), T(0));
    for (int tm = 0; tm < it.term_count; ++tm) {
        const MacTerm te = m.terms[it.term_begin + tm];
        const C *xb0[R];
#pragma unroll
        for (int r = 0; r < R; ++r)
            xb0[r] = m.x + m.xo[te.x_begin + r];
#pragma unroll (R == 1 ? 2 : 1)
        for (int p = 0; p < it.m2; ++p) {
            const C *kp = m.spec + te.k_off + (size_t)p * te.sp + (size_t)q * te.sq;
#pragma unroll
            for (int f = 0; f < 3; ++f) {
                C xa[IM][R], xb[IM][R];
#pragma unroll
                for (int e = 0; e < IM; ++e)
#pragma unroll
                    for (int r = 0; r < R; ++r) {
                        const C *x = xb0[r] + ((size_t)mirror(p, e) * 3 + f) * F;
                        xa[e][r] = __ldg(x + fa);
                        xb[e][r] = __ldg(x + fb);
                    }
#pragma unroll
                for (int c = 0; c < NC; ++c) {
                    const C *kk = kp + (size_t)(c * 3 + f) * F;
                    const C ka = ld_stream(kk + fa), kb = ld_stream(kk + fb);
#pragma unroll
                    for (int r = 0; r < R; ++r) {
                        mac_pair<NC, false, false>(sa[0][c][r], sb[0][c][r], ka, kb, xa[0][r], xb[0][r], c, f);
                        if constexpr (SX)
                            mac_pair<NC, true, false>(sa[1][c][r], sb[1][c][r], ka, kb, xa[1][r], xb[1][r], c, f);
                        if constexpr (SY)
                            mac_pair<NC, false, true>(sa[IM / 2][c][r], sb[IM / 2][c][r], ka, kb, xa[IM / 2][r],
                                                      xb[IM / 2][r], c, f);
                        if constexpr (SX && SY)
                            mac_pair<NC, true, true>(sa[3][c][r], sb[3][c][r], ka, kb, xa[3][r], xb[3][r], c, f);
                    }
                }
            }
        }
    }
#pragma unroll
    for (int r = 0; r < R; ++r) {
        C *dst = m.acc + m.ao[it.a_begin + r];
#pragma unroll
        for (int e = 0; e < IM; ++e)
#pragma unroll
            for (int c = 0; c < NC; ++c) {
                C *o = dst + ((size_t)mirror(q, e) * NC + c) * F;
                o[fa] = sa[e][c][r];
                o[fb] = sb[e][c][r];  // ky = 0 and the Nyquist bin: the same value again
            }
    }
}

// The CTA's item, and the warp's share of it.
template <typename T>
__device__ __forceinline__ bool mac_locate(const MacArgs<T> &m, MacItem &it, int &tile, int &q0)
{
    int lo = 0, hi = m.nitems;
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (m.items[mid].blk_begin <= (int)blockIdx.x)
            lo = mid;
        else
            hi = mid;
    }
    it = m.items[lo];
    const int w = ((int)blockIdx.x - it.blk_begin) * (kBlkThreads / 32) + (threadIdx.x >> 5);
    tile = w / it.nqg;
    q0 = (w - tile * it.nqg) * it.qg;
    return tile < it.tiles;
}

template <typename T, int NC>
__global__ void __launch_bounds__(kBlkThreads, 2) k_blk_mac(MacArgs<T> m)
{
    MacItem it;
    int tile, q0;
    if (!mac_locate(m, it, tile, q0))
        return;
    const int lane = threadIdx.x & 31;
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

template <typename T, int NC>
__global__ void __launch_bounds__(kBlkThreads, 2) k_blk_mac_sym(MacArgs<T> m)
{
    MacItem it;
    int tile, q0;
    if (!mac_locate(m, it, tile, q0))
        return;
    const int lane = threadIdx.x & 31;
    // one unit and its images a warp (mac_qg), one or two right-hand sides
    if (it.sym == (kMirrorX | kMirrorY)) {
        if (it.rhs == 2)
            mac_sym_body<T, NC, kMirrorX | kMirrorY, 2>(m, it, tile, q0, lane);
        else
            mac_sym_body<T, NC, kMirrorX | kMirrorY, 1>(m, it, tile, q0, lane);
    } else if (it.sym == kMirrorX) {
        if (it.rhs == 2)
            mac_sym_body<T, NC, kMirrorX, 2>(m, it, tile, q0, lane);
        else
            mac_sym_body<T, NC, kMirrorX, 1>(m, it, tile, q0, lane);
    } else {
        if (it.rhs == 2)
            mac_sym_body<T, NC, kMirrorY, 2>(m, it, tile, q0, lane);
        else
            mac_sym_body<T, NC, kMirrorY, 1>(m, it, tile, q0, lane);
    }
}

template <typename T>
cudaError_t launch_blk_mac(const MacLaunch &l, const MacItem *items, const MacTerm *terms, const size_t *xo,
                           const size_t *ao, const void *spec, const void *x, void *acc, int ncomp, cudaStream_t st)
{
    using C = typename Cx<T>::C;
    MacArgs<T> m{items, terms, xo, ao, static_cast<const C *>(spec), static_cast<const C *>(x), static_cast<C *>(acc),
                 l.sym_items};
    if constexpr (sizeof(T) == 4) {
        if (l.sym_blocks > 0) {  // the mirror-symmetric items come first
            if (ncomp == 2)
                k_blk_mac_sym<T, 2><<<l.sym_blocks, kBlkThreads, 0, st>>>(m);
            else
                k_blk_mac_sym<T, 1><<<l.sym_blocks, kBlkThreads, 0, st>>>(m);
        }
    }
    m.items += l.sym_items;
    m.nitems = l.items;
    if (l.blocks > 0) {
        if (ncomp == 2)
            k_blk_mac<T, 2><<<l.blocks, kBlkThreads, 0, st>>>(m);
        else
            k_blk_mac<T, 1><<<l.blocks, kBlkThreads, 0, st>>>(m);
    }
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
    template cudaError_t launch_blk_mac<T>(const MacLaunch &, const MacItem *, const MacTerm *, const size_t *,    \
                                           const size_t *, const void *, const void *, void *, int, cudaStream_t); \
    template cudaError_t blk_prepare<T>();
SGF_BLK_INST(float)
SGF_BLK_INST(double)

}  // namespace sgf
