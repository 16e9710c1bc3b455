"""Index algebra of the block convolutions (sgf_block.cuh): a pair of patches m
apart, Cases 2 and 3 of Sec. 2.2 with a lattice offset A between the corners,
evaluated block by block with transforms of 2B points equals the direct double
sum over cells, whatever kernel the cell offsets carry."""
import numpy as np
import pytest


def _kernel(x, y):
    return np.sin(0.37 * x + 0.2) * np.cos(0.23 * y - 0.4) + 0.01 * x - 0.02 * y


def _direct(case, m, N, ax, ay, s):
    """Force-like sum at every target cell; x = source position minus target position, finer cells."""
    if case == 2:  # finer source s, coarser target
        src, tgt = np.arange(N) + 0.5, m * (np.arange(N) + 0.5)
        dx, dy = (src + ax)[None, :] - tgt[:, None], (src + ay)[None, :] - tgt[:, None]
    else:          # coarser source, finer target
        src, tgt = m * (np.arange(N) + 0.5), np.arange(N) + 0.5
        dx, dy = src[None, :] - (tgt + ax)[:, None], src[None, :] - (tgt + ay)[:, None]
    out = np.zeros((N, N))
    for j in range(N):
        for i in range(N):
            out[j, i] = (_kernel(dx[i][None, :], dy[j][:, None]) * s).sum()
    return out


def _blocks(case, m, N, ax, ay, s):
    B, P = N // m, 2 * (N // m)
    d = np.arange(P)
    d = np.where(d < B, d, d - P)
    valid = np.arange(P) != B
    out = np.zeros((N, N))
    X = {}
    for uy in range(m):
        for ux in range(m):
            unit = s[uy::m, ux::m] if case == 2 else s[uy * B:(uy + 1) * B, ux * B:(ux + 1) * B]
            X[uy, ux] = np.fft.rfft2(unit, (P, P))
    for qy in range(m):
        for qx in range(m):
            acc = 0.0
            for py in range(m):
                for px in range(m):
                    def pos(a, ph, blk):  # source minus target position at index D of the phase's convolution
                        D = blk * B + d if case == 2 else d - blk * B
                        if case == 2:
                            return -m * D + ph + 0.5 - 0.5 * m + a
                        return -m * D - ph - a - 0.5 + 0.5 * m
                    x = pos(ax, px, qx) if case == 2 else pos(ax, qx, px)
                    y = pos(ay, py, qy) if case == 2 else pos(ay, qy, py)
                    K = np.where(valid[None, :] & valid[:, None], _kernel(x[None, :], y[:, None]), 0.0)
                    acc = acc + np.fft.rfft2(K) * X[py, px]
            res = np.fft.irfft2(acc, (P, P))[:B, :B]
            if case == 2:
                out[qy * B:(qy + 1) * B, qx * B:(qx + 1) * B] = res
            else:
                out[qy::m, qx::m] = res
    return out


@pytest.mark.parametrize("case", [2, 3])
@pytest.mark.parametrize("m,N,ax,ay", [(2, 8, 3, -2), (2, 12, 0, 5), (4, 16, 7, 16), (8, 16, -3, 9)])
def test_blocks_equal_the_direct_sum(case, m, N, ax, ay):
    s = np.random.Generator(np.random.PCG64(m * N)).standard_normal((N, N))
    ref = _direct(case, m, N, ax, ay, s)
    # N^2 terms of order one, transforms of at most 2N points a side
    assert np.abs(_blocks(case, m, N, ax, ay, s) - ref).max() <= 64 * np.finfo(float).eps * N * N


@pytest.mark.parametrize("case", [2, 3])
@pytest.mark.parametrize("m,N", [(2, 8), (4, 16)])
@pytest.mark.parametrize("mx,my", [(True, False), (False, True), (True, True)])
def test_centred_pairs_are_mirror_images(case, m, N, mx, my):
    """A finer patch centred in the coarser one (A = N (m - 1)/2): the block of mirrored units
    is the block at the mirrored offsets, which per frequency is the value at -ky (y mirrored),
    its conjugate there (x mirrored) or its own conjugate (both), for a table even in both axes."""
    B, P, A = N // m, 2 * (N // m), N * (m - 1) // 2
    d = np.arange(P)
    d = np.where(d < B, d, d - P)
    live = np.arange(P) != B

    def edge(ph, blk):  # lower edge of the source cell, target centre at 0
        D = blk * B + d if case == 2 else d - blk * B
        return -m * D + ph - 0.5 * m + A if case == 2 else -m * D - ph - A - 0.5

    w = 1.0 if case == 2 else float(m)

    def block(p, q):  # p, q = (x, y): phase and block of Case 2, block and phase of Case 3
        ph, bl = (p, q) if case == 2 else (q, p)
        u, v = edge(ph[0], bl[0])[None, :] + 0.5 * w, edge(ph[1], bl[1])[:, None] + 0.5 * w
        return np.fft.fft2(np.where(live[None, :] & live[:, None], np.cos(0.3 * u) * np.exp(-0.01 * v * v), 0.0))

    back = -np.arange(P)
    for p in [(x, y) for x in range(m) for y in range(m)]:
        for q in [(x, y) for x in range(m) for y in range(m)]:
            mir = lambda a: (m - 1 - a[0] if mx else a[0], m - 1 - a[1] if my else a[1])
            K = block(p, q)
            want = K[back] if my and not mx else np.conj(K[back]) if mx and not my else np.conj(K)
            assert np.abs(block(mir(p), mir(q)) - want).max() <= 1e-12 * max(1.0, np.abs(K).max())
