// sgf_block.h -- data structures of the block convolutions (the cross-level
// pairs of Cases 2 and 3; see sgf_block.cuh) and their launchers.
#pragma once
#include "sgf_internal.h"

namespace sgf {

constexpr int kBlkThreads = 256;
constexpr int kSMs = 152;  // of a GB300, for the rules that weigh a launch's CTAs or warps against them
constexpr int kMaxStages = kMaxLevels - 1;
enum : int { BLK_ROWS = 0, BLK_COLS = 1, BLK_ICOLS = 2, BLK_PASSES = 3, BLK_IROWS = 3 };

// A patch as the source (kind 0: its m^2 phases, Case 2; 1: its m^2 blocks, Case
// 3) or the target (kind 0: its blocks, Case 2; 1: its phases, Case 3) of a stage.
struct BlkUnit {
    int patch, kind;
};

// Everything m apart: sources src[src_begin ..), targets tgt[tgt_begin ..), those of
// Case 2 first.  x_off, a_off: complex offsets of its fields in BlkArgs::x and ::acc
// (source or target, unit, field or component, then F = (B + 1) 2B values).
struct BlkStage {
    int m, logB;
    int src_begin, src_count;
    int tgt_begin, tgt_count[2];
    int tw_off, tw_entries, pad;  // twiddle area (tw_layout of B) in BlkArgs::tw
    size_t x_off, a_off;
};

// One target of one stage in a round of the inverse rows (target ti of the stage).
struct BlkSeg {
    int stage, ti, blk;  // blk: its first CTA
};

template <typename T>
struct BlkArgs {
    using C = typename std::conditional<sizeof(T) == 8, double2, float2>::type;
    int stages;
    int blocks[BLK_PASSES][kMaxStages + 1];  // first block of each stage, per pass; the total last
    // Inverse rows: round r adds, for every patch, the pair with one other level, so
    // that no two CTAs of a launch add to one cell (and the sums have a fixed order)
    int rounds, segs[kMaxStages];
    BlkSeg seg[kMaxStages][kMaxPatches + 1];  // blk of the one after the last: the round's CTAs
    BlkStage st[kMaxStages];
    const BlkUnit *src, *tgt;
    const C *tw;
    C *x, *acc;
};

// One product of a target: kernel block (p, q, table) at k_off + p sp + q sq + table F
// (complex elements of the spectra), sources x[x_begin + r] for right-hand side r.
struct MacTerm {
    size_t k_off, sp, sq;
    int x_begin, pad;
};

// Targets with the same terms (the same kernel spectra), R right-hand sides each:
// fields read at MacPtrs x[..], results written at a[a_begin + r].
struct MacItem {
    int term_begin, term_count, a_begin, rhs;
    int m2, F, qg, nqg;       // units, frequencies, targets per warp, target groups
    int tiles, blk_begin;     // frequency tiles of a warp; the item's first CTA
    int logm, logB, sym, pad; // sym: mirror symmetry of the pairs (kMirrorX | kMirrorY)
};

// A pair whose finer patch is centred in the coarser one along an axis (A = N (m - 1)/2)
// has mirror-symmetric kernels on that axis: the block (p, q) with both units mirrored is the
// block itself at the mirrored offsets, up to each table's parity.
enum : int { kMirrorX = 1, kMirrorY = 2 };

// GenSet::cas of a set stored as the m^2 blocks of a block convolution (Case 2, Case 3),
// and above it the mirror symmetry every use of the set has: the products then read the
// lower half of the target units in the mirrored axes alone, and the other blocks of a
// Case 2 set (the whole set of such a phase in Case 3) are not generated.
constexpr int kBlkCase2 = 5, kBlkCase3 = 6, kBlkSymShift = 4;
inline __host__ __device__ int gen_case(const GenSet &g) { return g.cas & ((1 << kBlkSymShift) - 1); }
inline __host__ __device__ int gen_sym(const GenSet &g) { return g.cas >> kBlkSymShift; }
inline __host__ __device__ bool gen_blk(const GenSet &g) { return gen_case(g) == kBlkCase2 || gen_case(g) == kBlkCase3; }

// A pass of the block convolutions.  Single solve: a, k by value (plans = 1, prefix NULL);
// batch: da, dk on the device, `plans` of them, prefix[pass] on the device.
template <typename T>
cudaError_t launch_blk_pass(int pass, int round, int blocks, const SolveArgs<T> &a, const BlkArgs<T> &k,
                            cudaStream_t st);
template <typename T>
cudaError_t launch_blk_pass_batch(int pass, int round, int blocks, int plans, const int *prefix,
                                  const int *index, const SolveArgs<T> *da, const BlkArgs<T> *dk, cudaStream_t st);
// The products: first sym_items mirror-symmetric work items (sym_blocks CTAs), then items
// (blocks CTAs); spec, x and acc are the bases of the offsets (batches: NULL, the offsets
// whole addresses / sizeof(complex)).
struct MacLaunch {
    int sym_items = 0, sym_blocks = 0, items = 0, blocks = 0;
};
template <typename T>
cudaError_t launch_blk_mac(const MacLaunch &l, const MacItem *items, const MacTerm *terms, const size_t *xo,
                           const size_t *ao, const void *spec, const void *x, void *acc, int ncomp, cudaStream_t st);
// Kernel attributes of the block passes (plan creation).
template <typename T>
cudaError_t blk_prepare();
// CTAs a pass of a stage takes (BLK_IROWS: of one target of it).
int blk_blocks(int pass, const BlkStage &s, int ncomp);

}  // namespace sgf
