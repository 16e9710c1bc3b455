// sgf_block.cuh -- cross-level pairs (Cases 2 and 3 of Sec. 2.2) as block
// convolutions: the kernels and the index algebra.
//
// A pair of patches m = 2^d apart couples the m^2 phases of the finer patch
// (every m-th cell, B = N/m cells a side) with the coarser patch.  The coarser
// patch is cut into m^2 blocks of B x B cells, so that every elementary
// convolution is one of B x B cells with B x B cells, zero-padded to 2B:
//   Case 2 (finer source):   target block q = sum over source phases p,
//   Case 3 (coarser source): target phase q = sum over source blocks p,
// both   Y_q^(k) = sum_p sum_f K_pq,f^(k) X_p,f^(k)   per frequency k, with
// m^2 transforms of 2B points a side in and m^2 out, where whole-grid
// convolutions take m^2 transforms of 2N points a side.  The kernel spectra
// (m^4 blocks of (B + 1) x 2B, six tables) are as many values as m^2 sets of
// (N + 1) x 2N, read once per solve: the stage is bound by streaming them.
//
// Measured (FP32, GB300, us per solve; whole-grid passes -> this, with symmetric
// products and the small solves' side stream): centred 1024^2 3 levels 2027 -> 952,
// 2048^2 2 levels off centre 2208 -> 1751, 256^2 3 levels 278 -> 119, six 256^2
// tiles and two refined patches 593 -> 305, 20 nests of 128 ... 1024 cells 3365 ->
// 1628; the 2048^2 and the 20 nests' figures hold 81 us and 18 us of the column
// pass's own gain (k_col_w).
//
// Passes of a solve, each one launch over every stage (one stage per m):
//   k_blk_rows   cells -> (sigma, dx, dy) of a source unit (phase or block),
//                two rows per complex sequence, B-point parity halves (even
//                bins from x[n], odd bins from x[n] W_2B^n), Hermitian unpack
//   k_blk_cols   columns of the same, in place (B rows in, 2B bins out)
//   k_blk_mac    the products per frequency, summed over p and f in registers
//   k_blk_icols  columns back, the parity halves folded, in place
//   k_blk_irows  rows back, added to the forces at the unit's cells
// Layout of a unit's field: [kx 0..B][half 0..1][k 0..B) complex (kx, ky = 2k +
// half); its first B values per kx hold the B rows between the row and the
// column pass.  A CTA of 256 threads runs 128/(B/16) sequences of B points
// (both halves of each), whatever B: 16 values per thread.
#pragma once
#include "sgf_block.h"
#include "sgf_kernels.cuh"

namespace sgf {

template <int LOGB>
struct BShape {
    static constexpr int B = 1 << LOGB, Q = B >> 4;
    static constexpr int G = kBlkThreads / (2 * Q);  // sequences per CTA
    static constexpr int SP = B + Q + 1;             // exchange buffer of one half
    static constexpr int HALF = B / 2 + 1;           // bins of one parity, 0..B
    static constexpr int F = (B + 1) * 2 * B;        // frequencies of a unit's field
};

// Shared memory of a CTA: twiddles | exchange buffers (or the gathered bins) | inverse
// rows: the real rows to add, and the forces they are added to | row passes: one BlkSeq
// per sequence.
template <typename T, int LOGB>
__host__ __device__ constexpr size_t blk_xbuf_bytes()
{
    using C = typename Cx<T>::C;
    using S = BShape<LOGB>;
    const size_t x = (size_t)S::G * 2 * S::SP * sizeof(C), g = (size_t)S::G * 2 * S::HALF * 2 * sizeof(C);
    return ((x > g ? x : g) + 15) & ~(size_t)15;
}
constexpr int kBlkCells = 16 * kBlkThreads;  // real values of a CTA's sequences (two rows of B each)
// A sequence of a row pass: the rows j and first column i0 of its cells, the covered
// columns [xa, xb) of each row (xa < 0: several rectangles, ask covered()), and where
// its bins lie (complex offset of its row pair at kx = 0; -1: no sequence).
struct BlkSeq {
    long long off;
    int j[2], i0, comp;
    int xa[2], xb[2];
};
// Covered columns of row jj of a patch.
template <typename T>
__device__ __forceinline__ void blk_cover(const SolveArgs<T> &a, int patch, int jj, int &xa, int &xb)
{
    xa = xb = 0;
    int n = 0;
    for (int k = a.cover_begin[patch]; k < a.cover_begin[patch + 1]; ++k) {
        const CoverRect &r = a.cover[k];
        if (jj >= r.y0 && jj < r.y1) {
            xa = r.x0;
            xb = r.x1;
            ++n;
        }
    }
    if (n > 1)
        xa = -1;
}
__device__ __forceinline__ void st4(float *p, const float (&r)[4])
{
    *reinterpret_cast<float4 *>(p) = make_float4(r[0], r[1], r[2], r[3]);
}
__device__ __forceinline__ void st4(double *p, const double (&r)[4])
{
    reinterpret_cast<double2 *>(p)[0] = make_double2(r[0], r[1]);
    reinterpret_cast<double2 *>(p)[1] = make_double2(r[2], r[3]);
}

template <typename T>
__device__ __noinline__ bool blk_covered_any(const SolveArgs<T> &a, int patch, int jj, int i)
{
    return covered(a, patch, jj, i);
}
template <typename T>
__device__ __forceinline__ bool blk_covered(const SolveArgs<T> &a, int patch, int jj, int i, int xa, int xb)
{
    return xa < 0 ? blk_covered_any(a, patch, jj, i) : i >= xa && i < xb;
}

// Cell of element (r, c) of a unit: kind 0 = phase (every m-th cell), 1 = block of B x B cells.
__device__ __forceinline__ int blk_cell(int kind, int m, int B, int u, int r) { return kind == 0 ? m * r + u : u * B + r; }

// Element e of a CTA's cells in the order of the patch's rows: its sequence and its
// column there (2^lmm units of a row pair: phases interleave, blocks follow one another).
struct BlkElem {
    int gg, c;
};
template <int LOGB>
__device__ __forceinline__ BlkElem blk_elem(int e, int lmm, int kind)
{
    const int w = e & ((1 << (LOGB + lmm)) - 1), pr = e >> (LOGB + lmm);
    const int ux = kind == 0 ? w & ((1 << lmm) - 1) : w >> LOGB;
    return BlkElem{(pr << lmm) + ux, kind == 0 ? w >> lmm : w & ((1 << LOGB) - 1)};
}

// ------------------------------------------------------------------ rows
// The sequences of a CTA are the m units of one row pair (their columns together
// are the pair's whole rows; N = 4096: half of them), for 2048/N row pairs: a
// phase's values are every m-th cell, so the other phases' loads find the same
// sectors in L1.  `fields` of the three fields run one after the other.
template <typename T, int LOGB>
__device__ __forceinline__ void blk_rows_body(const SolveArgs<T> &a, const BlkArgs<T> &k, const BlkStage &s, int lb,
                                              int f0, int fields, unsigned char *smem)
{
    using C = typename Cx<T>::C;
    using C2 = typename Cx<T>::C2;
    using S = BShape<LOGB>;
    constexpr int B = S::B, Q = S::Q, G = S::G, SP = S::SP;
    C *tw = reinterpret_cast<C *>(smem);
    unsigned char *body = smem + tw_bytes<C>(s.tw_entries);
    C *sbuf = reinterpret_cast<C *>(body);
    BlkSeq *seq = reinterpret_cast<BlkSeq *>(body + blk_xbuf_bytes<T, LOGB>());
    const int t = threadIdx.x;
    const int m = s.m, lm = __ffs(m) - 1, m2 = m * m, N = a.N, nl = a.n_log;
    const int lmm = __ffs(m < G ? m : G) - 1;           // 2^lmm units of a row pair in this CTA
    const int pairs = G >> lmm, lp = __ffs(pairs) - 1;  // row pairs
    const TwLayout tl = tw_layout(F16<LOGB>::twlen, B);
    cp_block(tw, k.tw + s.tw_off, tw_bytes<C>(s.tw_entries));
    cp_commit();
    // sequence sd: source, unit row uy, row pair rp, unit column ux; a source has N/2 row pairs, so
    // those of a CTA are of one source
    const int per = m2 * (B / 2);
    const int si = lb * G / per;
    if (si >= s.src_count)
        return;  // no sequence in this CTA
    const BlkUnit un = k.src[s.src_begin + si];
    const T *src = a.src[un.patch];
    for (int g = t; g < G; g += kBlkThreads) {
        const int sd = lb * G + g - si * per;
        const int ux = sd & (m - 1), rp = (sd >> lm) & (B / 2 - 1), uy = sd >> (lm + LOGB - 1);
        BlkSeq q;
        q.off = (long long)(s.x_off + (size_t)(si * m2 + uy * m + ux) * 3 * S::F + 2 * rp);
        q.i0 = un.kind == 0 ? ux : ux * B;
        q.comp = 0;
        for (int h = 0; h < 2; ++h) {
            q.j[h] = blk_cell(un.kind, m, B, uy, 2 * rp + h);
            blk_cover(a, un.patch, q.j[h], q.xa[h], q.xb[h]);
        }
        seq[g] = q;
    }
    const int g = t / (2 * Q), b = (t / Q) & 1, j = t & (Q - 1);
    const int st = un.kind == 0 ? m : 1;
    cp_wait<0>();
    __syncthreads();
#pragma unroll 1
    for (int f = f0; f < f0 + fields; ++f) {
        // field f of the CTA's cells, the two rows of a pair as one complex value, element c of
        // sequence gg at sbuf[2 gg SP + pad16(c)]; in the order of the patch's rows, so that loads
        // coalesce, and loaded whether used or not (at clamped cells), so that those of four
        // elements are in flight at once (1024^2 3 levels: 134 -> 121 us)
#pragma unroll 1
        for (int e0 = t; e0 < G * B; e0 += 4 * kBlkThreads) {
            T hi[4][2], lo[4][2];
#pragma unroll
            for (int w = 0; w < 4; ++w) {
                const BlkElem el = blk_elem<LOGB>(e0 + w * kBlkThreads, lmm, un.kind);
                const BlkSeq &q = seq[el.gg];
                const int i = min(q.i0 + st * el.c, nl - 1);
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int jj = min(q.j[h], nl - 1);
                    const T *r = src + (size_t)jj * N + i;
                    // central difference, one-sided on the patch's first and last cell
                    const int at = f == 1 ? i : jj, step = f == 0 ? 0 : f == 1 ? 1 : N;
                    hi[w][h] = __ldg(at < nl - 1 ? r + step : r);
                    lo[w][h] = f == 0 ? T(0) : __ldg(at > 0 ? r - step : r);
                }
            }
#pragma unroll
            for (int w = 0; w < 4; ++w) {
                const BlkElem el = blk_elem<LOGB>(e0 + w * kBlkThreads, lmm, un.kind);
                const BlkSeq &q = seq[el.gg];
                const int i = q.i0 + st * el.c;
                T x[2];
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int jj = q.j[h], at = f == 1 ? i : jj;
                    const bool live = i < nl && jj < nl && !blk_covered(a, un.patch, jj, i, q.xa[h], q.xb[h]);
                    T d = hi[w][h];
                    if (f != 0) {
                        d -= lo[w][h];
                        if (at > 0 && at < nl - 1)
                            d *= T(0.5);
                    }
                    x[h] = live ? d : T(0);
                }
                sbuf[2 * el.gg * SP + pad16(el.c)] = hmk<C>(x[0], x[1]);
            }
        }
        __syncthreads();
        C v[1][16];
#pragma unroll
        for (int u = 0; u < 16; ++u) {
            const C z = sbuf[2 * g * SP + pad16(j + u * Q)];
            v[0][u] = b ? hmul(z, twist(tw, tl, j, u)) : z;
        }
        if constexpr (F16<LOGB>::NST == 1)
            __syncthreads();  // no exchange follows: the unpack's stores would meet other threads' reads
        fft_ct<C, false, LOGB, 1, false, 0>(v, sbuf + (2 * g + b) * SP, SP, j, true, tw);
        __syncthreads();
#pragma unroll
        for (int u = 0; u < 16; ++u)
            sbuf[(2 * g + b) * SP + pad16(j + u * Q)] = v[0][u];
        __syncthreads();
        // X_a = (Z + conj Z~)/2, X_b = (Z - conj Z~)/(2i); neighbouring lanes take neighbouring row pairs
        C *xf = k.x + (size_t)f * S::F;
        for (int e = t; e < G * (B + 1); e += kBlkThreads) {
            const int pr = e & (pairs - 1), r = e >> lp;
            const int uxl = r / (B + 1), kx = r - uxl * (B + 1);
            const int gg = (pr << lmm) + uxl;
            const int bb = kx & 1, kk = kx >> 1;
            const int km = (B - bb - kk) & (B - 1);
            const C Z = sbuf[(2 * gg + bb) * SP + pad16(kk)];
            const C Zm = sbuf[(2 * gg + bb) * SP + pad16(km)];
            C2 o;
            o.x = T(0.5) * (Z.x + Zm.x);
            o.y = T(0.5) * (Z.y - Zm.y);
            o.z = T(0.5) * (Z.y + Zm.y);
            o.w = T(-0.5) * (Z.x - Zm.x);
            *reinterpret_cast<C2 *>(xf + seq[gg].off + (size_t)kx * (2 * B)) = o;
        }
        if (f + 1 < f0 + fields)
            __syncthreads();  // the exchange buffers are read
    }
}

// ------------------------------------------------------------------ cols
template <typename T, int LOGB>
__device__ __forceinline__ void blk_cols_body(const BlkArgs<T> &k, const BlkStage &s, int lb, unsigned char *smem)
{
    using C = typename Cx<T>::C;
    using S = BShape<LOGB>;
    constexpr int B = S::B, Q = S::Q, G = S::G, SP = S::SP;
    C *tw = reinterpret_cast<C *>(smem);
    C *sbuf = reinterpret_cast<C *>(smem + tw_bytes<C>(s.tw_entries));
    const TwLayout tl = tw_layout(F16<LOGB>::twlen, B);
    cp_block(tw, k.tw + s.tw_off, tw_bytes<C>(s.tw_entries));
    cp_commit();
    const int t = threadIdx.x;
    const int g = t / (2 * Q), b = (t / Q) & 1, j = t & (Q - 1);
    const long long total = (long long)s.src_count * s.m * s.m * 3 * (B + 1);
    const long long sid = (long long)lb * G + g;  // column of the stage's fields, which lie one after the other
    const bool valid = sid < total;
    C *col = k.x + s.x_off + (valid ? sid : 0) * (2 * B);
    C v[1][16];
    if (valid) {
#pragma unroll
        for (int u = 0; u < 16; ++u)
            v[0][u] = col[j + u * Q];
    }
    cp_wait<0>();
    __syncthreads();
    if (valid && b) {
#pragma unroll
        for (int u = 0; u < 16; ++u)
            v[0][u] = hmul(v[0][u], twist(tw, tl, j, u));
    }
    fft_ct<C, false, LOGB, 1, false, 0>(v, sbuf + (2 * g + b) * SP, SP, j, valid, tw);
    if constexpr (LOGB >= 8) {  // 16 threads or more write 128 contiguous bytes
        __syncthreads();        // every read of the column (its first B values) is done
        if (valid) {
#pragma unroll
            for (int u = 0; u < 16; ++u)
                col[b * B + j + u * Q] = v[0][u];
        }
    } else {
        __syncthreads();
        if (valid) {
#pragma unroll
            for (int u = 0; u < 16; ++u)
                sbuf[(2 * g + b) * SP + pad16(j + u * Q)] = v[0][u];
        }
        __syncthreads();
        C *base = k.x + s.x_off + (size_t)lb * G * (2 * B);
        for (int e = t; e < G * 2 * B; e += kBlkThreads) {
            const int seq = e >> LOGB, kk = e & (B - 1);  // seq = 2 column + half
            if ((long long)lb * G + (seq >> 1) < total)
                base[e] = sbuf[seq * SP + pad16(kk)];
        }
    }
}

// ----------------------------------------------------------------- icols
template <typename T, int LOGB>
__device__ __forceinline__ void blk_icols_body(const BlkArgs<T> &k, const BlkStage &s, int ncomp, int lb,
                                               unsigned char *smem)
{
    using C = typename Cx<T>::C;
    using S = BShape<LOGB>;
    constexpr int B = S::B, Q = S::Q, G = S::G, SP = S::SP;
    C *tw = reinterpret_cast<C *>(smem);
    C *sbuf = reinterpret_cast<C *>(smem + tw_bytes<C>(s.tw_entries));
    const TwLayout tl = tw_layout(F16<LOGB>::twlen, B);
    cp_block(tw, k.tw + s.tw_off, tw_bytes<C>(s.tw_entries));
    cp_commit();
    const int t = threadIdx.x;
    const int g = t / (2 * Q), b = (t / Q) & 1, j = t & (Q - 1);
    const long long total = (long long)(s.tgt_count[0] + s.tgt_count[1]) * s.m * s.m * ncomp * (B + 1);
    const long long sid = (long long)lb * G + g;
    const bool valid = sid < total;
    C *col = k.acc + s.a_off + (valid ? sid : 0) * (2 * B);
    C v[1][16];
    if (valid) {
#pragma unroll
        for (int u = 0; u < 16; ++u)
            v[0][u] = col[b * B + j + u * Q];
    }
    cp_wait<0>();
    __syncthreads();
    fft_ct<C, true, LOGB, 1, false, 0>(v, sbuf + (2 * g + b) * SP, SP, j, valid, tw);
    __syncthreads();
    // y[n] = even[n] + W_2B^{-n} odd[n]
    if (valid && b) {
#pragma unroll
        for (int u = 0; u < 16; ++u)
            sbuf[(2 * g + 1) * SP + pad16(j + u * Q)] = hmulc(v[0][u], twist(tw, tl, j, u));
    }
    __syncthreads();
    if (valid && b == 0) {
#pragma unroll
        for (int u = 0; u < 16; ++u)
            col[j + u * Q] = hadd(v[0][u], sbuf[(2 * g + 1) * SP + pad16(j + u * Q)]);
    }
}

// ----------------------------------------------------------------- irows
// One target: of Case 2 (kind 0, blocks of the coarser patch) or of Case 3 (kind
// 1, phases of the finer patch).  The sequences of a CTA are consecutive row
// pairs of a block, or the m phases of a row pair (as in the forward row pass), so
// that the phases interleave in shared memory and runs of whole rows are added.
// The bins come in as asynchronous copies, all in flight at once: loaded into
// registers one after the other their latency was most of the pass (1024^2 3
// levels: two launches of 65 us, now 51; 2048^2 2 levels 167 -> 113).
template <typename T, int LOGB>
__device__ __forceinline__ void blk_irows_body(const SolveArgs<T> &a, const BlkArgs<T> &k, const BlkStage &s,
                                               int target, int lb, unsigned char *smem)
{
    using C = typename Cx<T>::C;
    using C2 = typename Cx<T>::C2;
    using S = BShape<LOGB>;
    constexpr int B = S::B, Q = S::Q, G = S::G, SP = S::SP, HALF = S::HALF;
    C *tw = reinterpret_cast<C *>(smem);
    unsigned char *body = smem + tw_bytes<C>(s.tw_entries);
    C *sbuf = reinterpret_cast<C *>(body);
    C2 *stg = reinterpret_cast<C2 *>(body);  // [sequence][kx & 1][kx >> 1], then the exchange buffers
    T *rows = reinterpret_cast<T *>(body + blk_xbuf_bytes<T, LOGB>());  // [sequence][row][B]
    T *old = rows + kBlkCells;  // the forces at the CTA's cells, in the order they are added to
    BlkSeq *seq = reinterpret_cast<BlkSeq *>(old + kBlkCells);
    const TwLayout tl = tw_layout(F16<LOGB>::twlen, B);
    cp_block(tw, k.tw + s.tw_off, tw_bytes<C>(s.tw_entries));
    cp_commit();
    const int t = threadIdx.x;
    const int m = s.m, lm = __ffs(m) - 1, m2 = m * m, nc = a.ncomp, N = a.N;
    const BlkUnit tg = k.tgt[s.tgt_begin + target];
    const int kind = tg.kind, patch = tg.patch, per = m2 * (B / 2), total = per * nc;
    const int lmm = kind == 0 ? 0 : __ffs(m < G ? m : G) - 1;  // 2^lmm phases of a row pair interleave in this CTA
    const int pairs = G >> lmm, lp = __ffs(pairs) - 1;
    for (int g = t; g < G; g += kBlkThreads) {
        const int sd = lb * G + g;
        BlkSeq q;
        q.off = -1;
        if (sd < total) {
            q.comp = sd >= per ? 1 : 0;
            const int r = sd - q.comp * per;
            const int ux = kind == 0 ? (r >> (LOGB - 1)) & (m - 1) : r & (m - 1);
            const int rp = kind == 0 ? r & (B / 2 - 1) : (r >> lm) & (B / 2 - 1);
            const int uy = r >> (lm + LOGB - 1);
            q.off = (long long)(s.a_off + ((size_t)(target * m2 + uy * m + ux) * nc + q.comp) * S::F + 2 * rp);
            q.i0 = kind == 0 ? ux * B : ux;
            for (int h = 0; h < 2; ++h) {
                q.j[h] = blk_cell(1 - kind, m, B, uy, 2 * rp + h);
                blk_cover(a, patch, q.j[h], q.xa[h], q.xb[h]);
            }
        }
        seq[g] = q;
    }
    __syncthreads();
    // element e of the CTA's cells in the order of the patch's rows: its sequence, row and column
    auto cell_of = [&](int e, int &gg, int &h, int &c) {
        const int q = e >> lmm;
        c = q & (B - 1);
        h = (q >> LOGB) & 1;
        gg = ((q >> (LOGB + 1)) << lmm) + (e & ((1 << lmm) - 1));
    };
    T *ox = a.fx[patch], *oy = nc == 2 ? a.fy[patch] : nullptr;
    const int st = kind == 0 ? 1 : m;
    const bool whole = kind == 0 || m <= G;  // runs of cells one after the other (all phases of a row pair)
    for (int e = t; e < G * (B + 1); e += kBlkThreads) {
        const int pr = e & (pairs - 1), r = e >> lp;
        const int uxl = r / (B + 1), kx = r - uxl * (B + 1);
        const int gg = (pr << lmm) + uxl;
        const long long off = seq[gg].off;
        if (off >= 0) {
            C *dst = reinterpret_cast<C *>(stg + (gg * 2 + (kx & 1)) * HALF + (kx >> 1));
            const C *col = k.acc + off + (size_t)kx * (2 * B);
            cp16(dst, col);
            if constexpr (sizeof(T) == 8)
                cp16(dst + 1, col + 1);
        }
    }
    cp_commit();
    // the forces the CTA adds to: copied in behind the transforms where they lie one after the other
    if (whole) {
        constexpr int V = 16 / (int)sizeof(T);
        for (int e = V * t; e < kBlkCells; e += V * kBlkThreads) {
            int gg, h, c;
            cell_of(e, gg, h, c);
            if (seq[gg].off >= 0)
                cp16(old + e, (seq[gg].comp ? oy : ox) + (size_t)seq[gg].j[h] * N + seq[gg].i0 + st * c);
        }
    }
    cp_commit();
    cp_wait<1>();  // twiddles and bins; the forces may still be on their way
    __syncthreads();
    const int g = t / (2 * Q), b = (t / Q) & 1, j = t & (Q - 1);
    const bool valid = seq[g].off >= 0;
    C v[1][16];
    if (valid) {
#pragma unroll
        for (int u = 0; u < 16; ++u) {
            const int kx = 2 * (j + u * Q) + b;
            const int k2 = kx <= B ? kx : 2 * B - kx;  // same parity
            const C2 p = stg[(g * 2 + b) * HALF + (k2 >> 1)];
            // Z = A + iB from the stored half (kx <= B) or its conjugate mirror
            v[0][u] = kx <= B ? hmk<C>(p.x - p.w, p.y + p.z) : hmk<C>(p.x + p.w, p.z - p.y);
        }
    }
    __syncthreads();  // the gathered bins are read: the exchange buffers overwrite them
    fft_ct<C, true, LOGB, 1, false, 0>(v, sbuf + (2 * g + b) * SP, SP, j, valid, tw);
    __syncthreads();
    if (valid && b) {
#pragma unroll
        for (int u = 0; u < 16; ++u)
            sbuf[(2 * g + 1) * SP + pad16(j + u * Q)] = hmulc(v[0][u], twist(tw, tl, j, u));
    }
    __syncthreads();
    if (valid && b == 0) {
#pragma unroll
        for (int u = 0; u < 16; ++u) {
            const int n = j + u * Q;
            const C y = hadd(v[0][u], sbuf[(2 * g + 1) * SP + pad16(n)]);
            rows[(g * 2) * B + n] = y.x;
            rows[(g * 2 + 1) * B + n] = y.y;
        }
    }
    cp_wait<0>();
    __syncthreads();
    // add, four neighbouring cells at a time; covered cells keep their 0
#pragma unroll 1
    for (int w = 0; w < 4; ++w) {
        const int e = 4 * (t + w * kBlkThreads);
        int gg, h, c;
        cell_of(e, gg, h, c);
        const BlkSeq &sq = seq[gg];
        if (sq.off < 0)
            continue;
        T *o = (sq.comp ? oy : ox) + (size_t)sq.j[h] * N;
        T r[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            int gq, hq, cq;
            cell_of(e + q, gq, hq, cq);
            const int i = seq[gq].i0 + st * cq;
            r[q] = old[e + q];
            if (!whole)
                r[q] = o[i];
            if (!blk_covered(a, patch, sq.j[h], i, sq.xa[h], sq.xb[h]))
                r[q] += rows[(gq * 2 + hq) * B + cq];
            if (!whole)
                o[i] = r[q];
        }
        if (whole)
            st4(o + sq.i0 + st * c, r);
    }
}

// ------------------------------------------------- block -> plan, stage
// prefix: first block of every plan of the launch (batches), count + 1 entries.
template <typename T>
__device__ __forceinline__ int blk_plan(const int *prefix, int count, int blk)
{
    int lo = 0, hi = count;  // prefix[lo] <= blk < prefix[hi]
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (prefix[mid] <= blk)
            lo = mid;
        else
            hi = mid;
    }
    return lo;
}

// Stage of a plan's block: blocks[pass] holds the first block of each stage.
template <typename T>
__device__ __forceinline__ int blk_stage(const BlkArgs<T> &k, int pass, int &blk)
{
    int st = 0;
    while (st + 1 < k.stages && blk >= k.blocks[pass][st + 1])
        ++st;
    blk -= k.blocks[pass][st];
    return st;
}

}  // namespace sgf
