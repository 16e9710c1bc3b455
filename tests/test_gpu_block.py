"""Cross-level pairs as block convolutions (nests and forests of N >= 256): the
coarser patch cut into m x m blocks of B = N/m cells, every phase and block pair a
convolution zero-padded to 2B (Sec. 2.2, Eqs. eqnbmnn and eqnbnmn).  Against the
direct-sum oracle on sampled cells, within the bounds of tests/_gpu.py, at the
edges of the block sizes (B = 16 ... 2048), on odd offsets, embedded sizes,
forests (several sources per target) and potentials; the no-allocation solve and
batches (kernel spectra shared by up to four right-hand sides) bit for bit."""
import numpy as np
import pytest

import oracle
from paper_1603_03142_gb300 import workloads as W
from tests._gpu import run_gpu, sgf, tol, torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lib():
    return sgf()


def _sigma(geom, seed):
    rng = np.random.Generator(np.random.PCG64(seed))
    return [rng.uniform(0.2, 1.5, (geom.n, geom.n)) for _ in range(geom.levels)]


def _sample(geom, per_patch, seed):
    """Seeded uncovered cells of every patch, with the patch's corners and edges' midpoints."""
    rng = np.random.Generator(np.random.PCG64(seed))
    n, lv, ii, jj = geom.n, [], [], []
    edge = {(0, 0), (0, n - 1), (n - 1, 0), (n - 1, n - 1), (n // 2, 0), (0, n // 2), (n // 2, n - 1), (n - 1, n // 2)}
    for p in range(geom.levels):
        cov = geom.covered_mask(p)
        free = np.argwhere(~cov)
        pick = [tuple(x) for x in free[rng.choice(len(free), size=per_patch, replace=False)]]
        pick += [c for c in edge if not cov[c]][:max(0, per_patch // 2)]
        for j, i in pick:
            lv.append(p), jj.append(j), ii.append(i)
    return np.array(lv), np.array(ii), np.array(jj)


def _worst(geom, got, ref, samp):
    lv, ii, jj = samp
    worst = 0.0
    for p in range(geom.levels):
        m = lv == p
        scale = max(np.abs(r[m]).max() for r in ref)
        worst = max(worst, max(np.abs(g[p][jj[m], ii[m]] - r[m]).max() for g, r in zip(got, ref)) / scale)
    return worst


NESTS = {
    "512x2_corner": (W.Nest(n=512, levels=2, off=[(0, 0), (0, 256)]), ("fp32", "bf16x")),
    "256x3_odd": (W.Nest(n=256, levels=3, off=[(0, 0), (37, 90), (101, 3)]), ("fp32", "bf16x")),
    "256x5": (W.Nest(n=256, levels=5, off=[(0, 0), (64, 65), (63, 7), (128, 64), (31, 33)]), ("fp32",)),
    "256x3_centred": (W.centred_nest(256, 3), ("fp32",)),       # mirror-symmetric pairs in both axes
    "256x4_mirror_y": (W.centred_nest(256, 4, centre=(0.3, 0.0)), ("fp32",)),
    "512x3_mirror_x": (W.centred_nest(512, 3, centre=(0.0, -0.2)), ("fp32", "bf16x")),
    "300x3_embedded": (W.Nest(n=300, levels=3, off=[(0, 0), (75, 11), (150, 80)]), ("fp32",)),
    "1024x4": (W.Nest(n=1024, levels=4, off=[(0, 0), (255, 256), (301, 4), (256, 511)]), ("fp32",)),
    "2048x2": (W.Nest(n=2048, levels=2, off=[(0, 0), (513, 700)]), ("fp32",)),
    "4096x2": (W.Nest(n=4096, levels=2, off=[(0, 0), (1025, 1000)]), ("fp32",)),
    "two_patches512": (W.two_patch_forest(512), ("fp32",)),
    "example4_256": (W.example4_forest(256), ("fp32",)),
}


@pytest.mark.parametrize("name,prec", [(k, p) for k, (_, ps) in NESTS.items() for p in ps])
def test_block_pairs_against_oracle(lib, name, prec):
    geom = NESTS[name][0]
    sigma = _sigma(geom, 3)
    plan = lib.Plan(geom, prec)
    gx, gy = run_gpu(plan, sigma)
    plan.check()
    samp = _sample(geom, 4 if geom.n >= 2048 else 16, 5)
    ox, oy = oracle.force_at(geom, sigma, *samp)
    assert _worst(geom, (gx, gy), (ox, oy), samp) <= tol(prec, geom.n)


@pytest.mark.parametrize("name", ["512x2_corner", "256x3_odd", "256x5", "300x3_embedded", "256x3_centred",
                                  "256x4_mirror_y", "512x3_mirror_x"])
@pytest.mark.parametrize("prec", ["fp32", "fp64"])
def test_block_pairs_equal_whole_grid_pairs(lib, name, prec):
    """A plan over its spectra budget runs the whole-grid passes on the same FP64 tables: the
    same sums in another order (256 ulps, the bound of the budget tests).  In FP64 this says
    more than the oracle: away from m = 1 both paths share the tables' own error."""
    geom = NESTS[name][0]
    sigma = _sigma(geom, 11)
    plan = lib.Plan(geom, prec)
    whole = lib.Plan(geom, prec, spectra_budget=plan.stats()["spectra_bytes"] // 2)
    assert whole.stats()["spectra_sets_streamed"] > 0
    a, b = run_gpu(plan, sigma), run_gpu(whole, sigma)
    eps = np.finfo(np.float64 if prec == "fp64" else np.float32).eps
    for l in range(geom.levels):
        scale = max(np.abs(b[0][l]).max(), np.abs(b[1][l]).max())
        d = max(np.abs(a[c][l] - b[c][l]).max() for c in range(2))
        assert d <= 256 * eps * scale, (l, d / scale)


@pytest.mark.parametrize("name,prec", [("256x3_odd", "fp32"), ("256x3_centred", "fp32"), ("256x4_mirror_y", "fp32"),
                                       ("512x3_mirror_x", "fp32")])
def test_block_potential_against_oracle(lib, name, prec):
    geom = NESTS[name][0]
    sigma = _sigma(geom, 4)
    plan = lib.Plan(geom, prec, potential=True)
    dt = torch.float64 if prec == "fp64" else torch.float32
    phi = plan.solve_potential([torch.from_numpy(s).to(device="cuda", dtype=dt) for s in sigma])
    torch.cuda.synchronize()
    samp = _sample(geom, 16, 6)
    ref = oracle.potential_at(geom, sigma, *samp)
    assert _worst(geom, ([p.double().cpu().numpy() for p in phi],), (ref,), samp) <= tol(prec, geom.n)


def test_block_noalloc_is_bitwise_the_solve(lib):
    for geom in (W.Nest(n=256, levels=3, off=[(0, 0), (64, 20), (33, 64)]), W.two_patch_forest(256)):
        plan = lib.Plan(geom, "fp32")
        sig = [torch.from_numpy(s).float().cuda() for s in _sigma(geom, 8)]
        fx, fy = plan.solve(sig)
        gx, gy = [torch.empty_like(s) for s in sig], [torch.empty_like(s) for s in sig]
        plan.solve_noalloc_ptrs([s.data_ptr() for s in sig], [t.data_ptr() for t in gx], [t.data_ptr() for t in gy])
        torch.cuda.synchronize()
        for l in range(geom.levels):
            assert torch.equal(fx[l], gx[l]) and torch.equal(fy[l], gy[l])


@pytest.mark.parametrize("count", [1, 3, 6])
def test_block_batch_is_bitwise_the_single_solves(lib, count):
    """`count` centred nests on shared spectra (their level pairs share sets too), one nest of
    another shape, one deep nest on whole-grid passes (B would be 8), one uniform grid."""
    base = lib.Plan(W.centred_nest(256, 3), "fp32")
    plans = [base] + [base.share() for _ in range(count - 1)]
    plans += [lib.Plan(W.centred_nest(512, 2, centre=(0.3, 0.1)), "fp32"), lib.Plan(W.centred_nest(256, 6), "fp32"),
              lib.Plan(W.Nest(n=256), "fp32")]
    sig = [[torch.from_numpy(s).float().cuda() for s in _sigma(p.nest, 20 + k)] for k, p in enumerate(plans)]
    single = [p.solve(s) for p, s in zip(plans, sig)]
    torch.cuda.synchronize()
    batch = lib.Batch(plans)
    fx, fy = [[torch.empty_like(s) for s in lst] for lst in sig], [[torch.empty_like(s) for s in lst] for lst in sig]
    for _ in range(2):
        batch.solve(sig, fx, fy)
    torch.cuda.synchronize()
    for k, p in enumerate(plans):
        for l in range(p.levels):
            assert torch.equal(fx[k][l], single[k][0][l]) and torch.equal(fy[k][l], single[k][1][l]), (k, l)


def test_bf16x_depths_and_shared_spectra(lib):
    """SGF_BF16X of three levels keeps the whole-grid passes; a plan shared from FP32 takes the
    spectra as they are stored; both within the precision's bound of FP32."""
    for n, levels in ((512, 2), (256, 3)):
        nest = W.centred_nest(n, levels)
        sigma = _sigma(nest, 30)
        p32 = lib.Plan(nest, "fp32")
        ref = run_gpu(p32, sigma)
        for p in (lib.Plan(nest, "bf16x"), p32.share("bf16x"), lib.Plan(nest, "bf16x").share("fp32")):
            got = run_gpu(p, sigma)
            p.check()
            for l in range(levels):
                scale = max(np.abs(ref[0][l]).max(), np.abs(ref[1][l]).max())
                assert max(np.abs(got[c][l] - ref[c][l]).max() for c in range(2)) <= tol("bf16x", n) * scale


@pytest.mark.parametrize("n,levels,centre", [(256, 3, (0.0, 0.0)), (256, 4, (0.3, 0.0)), (256, 3, (0.3, -0.2)),
                                             (512, 2, (0.0, 0.0)), (128, 3, (0.0, 0.0)), (256, 1, (0.0, 0.0))])
def test_algorithmic_bytes_follow_the_reads(lib, n, levels, centre):
    """The plan's byte count is that of bench.py's split by pair of levels: the spectra as the
    products read them (halves and quarters of mirror-symmetric pairs, shared reads once)."""
    from bench import nest_pair_bytes
    nest = W.centred_nest(n, levels, centre=centre) if levels > 1 else W.Nest(n=n)
    plan = lib.Plan(nest, "fp32")
    assert plan.stats()["algorithmic_bytes"] == nest_pair_bytes([nest])["total"]


# The root's one finer patch and one of that patch's two lie alike, centred in x: the products of the
# root's pair sum mirror images over spectra that another target, of two sources, reads whole.
SHARED_MIRROR = W.Forest(n=256, level=[0, 1, 2, 2], org=[(0, 0), (128, 0), (384, 0), (384, 256)])


def test_mirror_images_over_spectra_read_whole_elsewhere(lib):
    sigma = _sigma(SHARED_MIRROR, 13)
    plan = lib.Plan(SHARED_MIRROR, "fp32")
    gx, gy = run_gpu(plan, sigma)
    samp = _sample(SHARED_MIRROR, 16, 7)
    ox, oy = oracle.force_at(SHARED_MIRROR, sigma, *samp)
    assert _worst(SHARED_MIRROR, (gx, gy), (ox, oy), samp) <= tol("fp32", 256)


def _tol64(geom):
    """FP64 bound of a nest: tol()'s 0.2 eps N^2 is that of lattice coordinates up to N; where levels m
    apart meet they are those of the finer lattice, m times as large, and so are the corner
    antiderivatives whose double differences leave the error (on both sides, oracle and tables)."""
    return 2 ** (geom.levels - 1) * tol("fp64", geom.n)


@pytest.mark.parametrize("name", ["256x3_odd", "300x3_embedded", "512x3_mirror_x", "2048x2"])
def test_block_pairs_fp64_against_oracle(lib, name):
    """B = 64 ... 256 and 1024, an instance of its own."""
    geom = NESTS[name][0]
    sigma = _sigma(geom, 3)
    gx, gy = run_gpu(lib.Plan(geom, "fp64"), sigma)
    samp = _sample(geom, 4 if geom.n >= 2048 else 16, 5)
    ox, oy = oracle.force_at(geom, sigma, *samp)
    assert _worst(geom, (gx, gy), (ox, oy), samp) <= _tol64(geom)


@pytest.mark.parametrize("name,prec", [("256x3_odd", "fp64"), ("512x2_corner", "fp64"), ("300x3_embedded", "fp64"),
                                       ("300x3_embedded", "fp32")])
def test_block_potential_fp64_and_embedded(lib, name, prec):
    geom = NESTS[name][0]
    sigma = _sigma(geom, 4)
    plan = lib.Plan(geom, prec, potential=True)
    dt = torch.float64 if prec == "fp64" else torch.float32
    phi = plan.solve_potential([torch.from_numpy(s).to(device="cuda", dtype=dt) for s in sigma])
    torch.cuda.synchronize()
    samp = _sample(geom, 16, 6)
    ref = oracle.potential_at(geom, sigma, *samp)
    worst = _worst(geom, ([p.double().cpu().numpy() for p in phi],), (ref,), samp)
    assert worst <= (_tol64(geom) if prec == "fp64" else tol(prec, geom.n))


@pytest.mark.parametrize("geom,prec,pot", [
    (W.centred_nest(512, 2), "fp32", False), (W.centred_nest(256, 4, centre=(0.3, 0.0)), "fp32", False),  # side stream
    (W.centred_nest(256, 2), "fp64", True), (W.two_patch_forest(256), "fp32", False),
    (W.centred_nest(512, 3), "fp32", False), (W.centred_nest(1024, 2), "fp32", True)],  # one after the other
    ids=["512x2", "256x4", "256x2_fp64_phi", "two_patches256", "512x3", "1024x2_phi"])
def test_captured_block_solves_replay_bitwise(lib, geom, prec, pot):
    """Captured into a graph before any eager solve, the side stream of small plans forked and joined
    inside the capture; replayed on another stream than the capture's."""
    dt = torch.float64 if prec == "fp64" else torch.float32
    plan = lib.Plan(geom, prec, potential=pot)
    ts = [torch.from_numpy(s).to(device="cuda", dtype=dt) for s in _sigma(geom, 17)]
    outs = [[torch.empty_like(t) for t in ts] for _ in range(1 if pot else 2)]
    ptrs = [[t.data_ptr() for t in lst] for lst in [ts] + outs]
    solve = plan.solve_potential_ptrs if pot else plan.solve_ptrs
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.graph(graph, stream=side):
        solve(*ptrs)
    torch.cuda.synchronize()
    eager = [[torch.empty_like(t) for t in ts] for _ in outs]
    for _ in range(2):
        for lst in outs:
            for t in lst:
                t.fill_(float("nan"))
        graph.replay()
        torch.cuda.synchronize()
        solve(ptrs[0], *[[t.data_ptr() for t in lst] for lst in eager])
        torch.cuda.synchronize()
        for a, b in zip(outs, eager):
            for x, y in zip(a, b):
                assert torch.equal(x, y)
