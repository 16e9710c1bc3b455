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
