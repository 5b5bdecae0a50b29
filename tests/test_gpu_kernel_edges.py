"""GPU kernels at the edges of their tiles and of the rules that choose them.

Tolerances: against the FP64 oracle FMM / treecode on the same tree relative L2 <= 1e-5, the
parity tests' bound; against the FP64 direct sum 1e-6 for FP32 sums of at most a few thousand
terms (each sum's relative error is below n / 32 lanes of 2^-24 and its terms have one sign in phi).
"""
import numpy as np
import pytest

import oracle as O
from paper_1010_1482_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = 1e-5
TOL_DIRECT = 1e-6


@pytest.fixture(scope="module")
def G():
    from paper_1010_1482_gb300 import gbfmm

    gbfmm.lib()
    return gbfmm


@pytest.fixture(scope="module")
def ctx(G):
    c = G.gbfmm_create(0)
    yield c
    G.gbfmm_destroy(c)


def run(G, ctx, x, **kw):
    prm = G.gbfmm_default_params(**kw)
    _, ws = G.gbfmm_plan(prm, len(x))
    xd = torch.from_numpy(np.ascontiguousarray(x, dtype=np.float32)).cuda()
    out = torch.full_like(xd, float("nan"))
    G.gbfmm_evaluate(ctx, prm, xd, out, torch.empty(max(ws, 256), dtype=torch.uint8, device="cuda"))
    G.gbfmm_sync_status(ctx)
    return out.cpu().numpy().astype(np.float64)


def direct64(src, tgt, eps2):
    d = tgt[:, None, :3].astype(np.float64) - src[None, :, :3].astype(np.float64)
    r2 = (d * d).sum(-1)
    inv = np.where(r2 > 0, 1.0 / np.sqrt(np.where(r2 > 0, r2 + eps2, 1.0)), 0.0)
    w = inv * src[None, :, 3]
    return np.concatenate([w.sum(1)[:, None], -((w * inv * inv)[..., None] * d).sum(1)], axis=1)


# targets around the tile of 64, sources around the split of 8, groups of 4 and tiles of 512 a CTA
@pytest.mark.parametrize("ns,nt", [(1, 1), (3, 64), (8, 65), (31, 63), (33, 129), (100, 1), (4095, 200), (4097, 64),
                                   (8 * 513 + 1, 31)])
@pytest.mark.parametrize("eps2", [0.0, 1e-3])
def test_direct_tiles(G, ctx, ns, nt, eps2):
    src = inputs.uniform_cube(ns, 100 + ns)
    tgt = inputs.uniform_cube(nt, 200 + nt)
    k = min(ns, nt, 40)
    tgt[:k] = src[ns - k:]  # coincident pairs, the last of them in the remainder groups
    if ns > 8:
        src[1] = src[0]
    out = torch.full((nt, 4), float("nan"), device="cuda")
    G.gbfmm_direct(ctx, torch.from_numpy(src).cuda(), torch.from_numpy(tgt).cuda(), out, eps2)
    torch.cuda.synchronize()
    ref = direct64(src, tgt, eps2)
    got = out.cpu().numpy().astype(np.float64)
    assert np.all(np.isfinite(got))
    assert np.linalg.norm(got - ref) <= TOL_DIRECT * max(np.linalg.norm(ref), 1e-30) + (0 if ref.any() else 1e-30)


# both sides of the rules that choose the form: 32 and 128 sources, 1024 targets, 48 targets a source
# (up to 1024 sources), and the edges of each form's tiles beyond them
@pytest.mark.parametrize("ns,nt", [(32, 257), (33, 1024), (33, 1025), (128, 1025), (129, 48 * 129), (129, 48 * 129 + 1),
                                   (1023, 48 * 1023 + 1), (1024, 48 * 1024 + 1), (1025, 48 * 1025 + 1)])
@pytest.mark.parametrize("eps2", [0.0, 1e-3])
def test_direct_forms(G, ctx, ns, nt, eps2):
    src = inputs.uniform_cube(ns, 110 + ns)
    tgt = inputs.uniform_cube(nt, 210 + nt)
    tgt[:ns] = src[:nt]
    src[1] = src[0]
    out = torch.full((nt, 4), float("nan"), device="cuda")
    G.gbfmm_direct(ctx, torch.from_numpy(src).cuda(), torch.from_numpy(tgt).cuda(), out, eps2)
    torch.cuda.synchronize()
    got = out.cpu().numpy().astype(np.float64)
    pick = np.unique(np.r_[: min(nt, ns + 70), max(0, nt - 130): nt])  # coincident pairs, the last CTAs
    ref = direct64(src, tgt[pick], eps2)
    assert np.all(np.isfinite(got))
    assert np.linalg.norm(got[pick] - ref) <= TOL_DIRECT * np.linalg.norm(ref)


def test_direct_many_targets_few_sources_time(G, ctx):
    """A million targets of a few sources pay for their pairs, not for splitting the sources: at most
    three times a copy of the targets plus the pairs at half the rate of the all-pairs sum (8e11 a second)."""
    nt = 1 << 20
    tgt = torch.rand((nt, 4), device="cuda")
    out = torch.empty_like(tgt)

    def us(f):
        f()
        best = float("inf")
        for _ in range(5):
            a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            a.record()
            for _ in range(10):
                f()
            b.record()
            b.synchronize()
            best = min(best, 100 * a.elapsed_time(b))
        return best

    copy = us(lambda: out.copy_(tgt))
    for ns in (1, 16, 64, 256):
        src = torch.rand((ns, 4), device="cuda")
        assert us(lambda: G.gbfmm_direct(ctx, src, tgt, out)) <= 3 * copy + nt * ns / 8e5 + 20, ns


def test_direct_no_sources(G, ctx):
    tgt = torch.rand((70, 4), device="cuda")
    out = torch.full((70, 4), 7.0, device="cuda")
    G.gbfmm_direct(ctx, torch.empty((0, 4), device="cuda"), tgt, out, 0.0)
    torch.cuda.synchronize()
    assert not out.any()


# depths 0 to 3, where several CTAs take a leaf's targets: fewer targets than parts, uneven parts,
# parts of more than the 256 targets of one pass
@pytest.mark.parametrize("n,leaf", [(1, 64), (2, 1), (17, 64), (300, 300), (5000, 5000), (9000, 1200), (513, 64),
                                    (700, 2)])
def test_p2p_parts_of_small_trees(G, ctx, n, leaf):
    x = inputs.uniform_cube(n, 300 + n)
    if n >= 16:
        x[n // 2] = x[0]
    out = run(G, ctx, x, p=4, leaf_size=leaf, eps2=1e-5)
    ref = O.fmm(x, 4, leaf, eps2=1e-5)["out"]
    assert np.linalg.norm(out - ref) <= TOL * max(np.linalg.norm(ref), 1e-30)


# leaves of about 2 to 70 targets: remainder chunks of every pairs-of-cells grouping
@pytest.mark.parametrize("p", [4, 6, 8, 10])
@pytest.mark.parametrize("n,leaf", [(150, 2), (64 * 9, 16), (64 * 33, 40), (64 * 70, 90)])
def test_treecode_chunks(G, ctx, p, n, leaf):
    x = inputs.uniform_cube(n, 400 + n)
    out = run(G, ctx, x, p=p, leaf_size=leaf, method=G.METHOD_TREECODE)
    ref = O.fmm(x, p, leaf, method=O.TREECODE)["out"]
    assert O.rel_l2(out[:, 0], ref[:, 0]) <= TOL and O.rel_l2(out[:, 1:], ref[:, 1:]) <= TOL


# on the cells' z axes and in their x-y planes the real recurrences' lowered terms and their
# factors are zero or cancel
@pytest.mark.parametrize("p", [4, 10])
def test_expansions_on_cell_axes(G, ctx, p):
    n = 4096
    g = (np.arange(16) + 0.5) / 16
    x = np.zeros((n, 4), dtype=np.float32)
    x[:, :3] = np.stack(np.meshgrid(g, g, g, indexing="ij"), -1).reshape(n, 3)
    x[:, 3] = inputs.uniform01(5, n)
    x[::2, 2] += 0.01
    box = dict(has_box=1, box_origin=[0.0, 0.0, 0.0], box_side=1.0)
    for method, om in ((G.METHOD_FMM, O.FMM), (G.METHOD_TREECODE, O.TREECODE)):
        out = run(G, ctx, x, p=p, leaf_size=1, method=method, **box)
        alt = run(G, ctx, x, p=p, leaf_size=1, method=method, flags=G.FLAG_SERIAL, **box)
        assert np.array_equal(out, alt) and np.all(np.isfinite(out))
        # the same particles without the box have their extent as the root cube: compare the two
        # within the truncation error of the order
        free = run(G, ctx, x, p=p, leaf_size=1, method=method)
        assert O.rel_l2(out, free) <= {4: 2e-2, 10: 1e-4}[p]
        ref = O.fmm(x, p, 1, method=om)["out"]
        assert O.rel_l2(free, ref) <= TOL


# the same with the root cube [0, 1]^3 found from two particles in its corners, so that the oracle
# builds the same cells: every other particle on a z axis of all cells it meets, or in their middle
@pytest.mark.parametrize("p", [4, 6, 8, 10])
def test_expansions_on_cell_axes_against_oracle(G, ctx, p):
    n = 4096
    g = (np.arange(16) + 0.5) / 16
    x = np.zeros((n, 4), dtype=np.float32)
    x[:, :3] = np.stack(np.meshgrid(g, g, g, indexing="ij"), -1).reshape(n, 3)
    x[::2, 2] += 0.01
    x[1234, :3], x[2345, :3] = 0.0, 1.0
    x[:, 3] = inputs.uniform01(6, n)
    origin, side = O.root_box(x)[:2]
    assert not np.any(origin) and side == 1.0 and O.uniform_depth(n, 1) == 4
    for method, om in ((G.METHOD_FMM, O.FMM), (G.METHOD_TREECODE, O.TREECODE)):
        out = run(G, ctx, x, p=p, leaf_size=1, method=method)
        ref = O.fmm(x, p, 1, method=om)["out"]
        assert O.rel_l2(out[:, 0], ref[:, 0]) <= TOL and O.rel_l2(out[:, 1:], ref[:, 1:]) <= TOL


# both sides of the rules on the expected number of leaves (8 or 32 lanes a leaf in P2M, 16 or 32
# a cell in P2L): 8,192 leaves
@pytest.mark.parametrize("p", [4, 8])
@pytest.mark.parametrize("n,leaf", [(30000, 11), (30000, 10), (21845, 8), (21846, 8)])
def test_adaptive_lanes_by_leaves(G, ctx, p, n, leaf):
    x = inputs.plummer(n, 500 + leaf)
    out = run(G, ctx, x, p=p, leaf_size=leaf, tree=G.TREE_ADAPTIVE)
    ref = O.fmm_adaptive(x, p, leaf)["out"]
    assert O.rel_l2(out, ref) <= TOL


# depth 5 (32,768 leaves, most of them holding 0 to 3 particles): P2M's eight lanes a leaf
def test_uniform_sparse_leaves(G, ctx):
    x = inputs.uniform_cube(33000, 17)
    out = run(G, ctx, x, p=6, leaf_size=2)
    assert O.rel_l2(out, O.fmm(x, 6, 2)["out"]) <= TOL


# the same tree in a batch, whose levels beyond k_m2m_small's range take a looping form over the
# counts of the creation, and alone: bit for bit
@pytest.mark.parametrize("p", [4, 6, 8, 10])
def test_m2m_forms_agree_in_batches(G, ctx, p):
    sizes = [2000, 30000]
    xs = [inputs.plummer(n, 600 + n) for n in sizes]
    x = torch.from_numpy(np.concatenate(xs)).cuda()
    out = torch.empty_like(x)
    prm = [G.gbfmm_default_params(p=p, leaf_size=8, tree=G.TREE_ADAPTIVE) for _ in sizes]
    offs = [0, sizes[0], sum(sizes)]
    b = G.gbfmm_batch_create(ctx, offs, prm, x, out, lanes=2)
    out.fill_(0)
    G.gbfmm_batch_launch(ctx, b)
    G.gbfmm_sync_status(ctx)
    got = out.cpu().numpy()
    G.gbfmm_batch_destroy(b)
    for i, xi in enumerate(xs):
        alone = run(G, ctx, xi, p=p, leaf_size=8, tree=G.TREE_ADAPTIVE, flags=G.FLAG_SERIAL)
        assert np.array_equal(got[offs[i]:offs[i + 1]].astype(np.float64), alone)


# A translation's sums do not depend on the kernel that takes its level.  A batch chooses by the
# counts of the particles it was created with, an evaluation by those it has (parents of levels 2, 3, ...):
#   600 Plummer 16, 30, 56, .. refilled with uniform 64, 339, 165, ..: runs of levels in one cluster
#     launch against a launch a level
#   6000: 32, 83, 184, .. with 64, 512, 3161, ..: the eight positions at once against 16 or 32 cells a CTA
#   30000: 49, 180, 401, 950 with 64, 512, 4095, 19411: the looping form too, against up to 64 cells
#   60000 and 160000 uniform, one a leaf, 44005 and 118411 on level 6: the looping form against 64 and
#     128 cells a CTA
@pytest.mark.parametrize("p", [4, 6, 8, 10])
@pytest.mark.parametrize("n,leaf,first", [(600, 2, "plummer"), (6000, 2, "plummer"), (30000, 2, "plummer"),
                                          (60000, 1, "uniform"), (160000, 1, "uniform")])
def test_translation_forms_agree(G, ctx, p, n, leaf, first):
    x = torch.from_numpy(inputs.make_particles(n, first, 600 + n)).cuda()
    out = torch.empty_like(x)
    b = G.gbfmm_batch_create(ctx, [0, n], [G.gbfmm_default_params(p=p, leaf_size=leaf, tree=G.TREE_ADAPTIVE)], x, out,
                             lanes=1)
    then = inputs.make_particles(n, "uniform", 600 + n)
    x.copy_(torch.from_numpy(then))
    out.fill_(0)
    G.gbfmm_batch_launch(ctx, b)
    G.gbfmm_sync_status(ctx)
    got = out.cpu().numpy().astype(np.float64)
    G.gbfmm_batch_destroy(b)
    assert np.array_equal(got, run(G, ctx, then, p=p, leaf_size=leaf, tree=G.TREE_ADAPTIVE, flags=G.FLAG_SERIAL))


# the scan of the level histograms by one CTA (up to 16,384 values, 23 bins x 712 blocks of 256
# particles) and by three kernels, and trees on both sides
@pytest.mark.parametrize("n", [712 * 256, 712 * 256 + 1])
def test_adaptive_tree_around_scan_sizes(G, ctx, n):
    x = inputs.plummer(n, 700)
    run(G, ctx, x, p=4, leaf_size=64, tree=G.TREE_ADAPTIVE)
    t = O.build_adaptive_tree(x, 64)
    g = G.gbfmm_export_adaptive_tree(ctx, n)
    assert g["ncells"] == t["ncells"]
    for k in ("level", "key", "begin", "count", "parent"):
        assert np.array_equal(g[k], t[k]), k
    lists = O.build_adaptive_lists(t)
    for kind, name in ((G.LIST_U, "u"), (G.LIST_V, "v"), (G.LIST_W, "w"), (G.LIST_X, "x")):
        offs, ids = G.gbfmm_export_lists(ctx, kind, t["ncells"])
        ref, row = lists[name + "_ids"], np.repeat(np.arange(t["ncells"]), np.diff(lists[name + "_offs"]))
        assert np.array_equal(offs, lists[name + "_offs"]) and len(ids) == len(ref)
        assert np.array_equal(ids, ref[np.lexsort((ref, row))]), name


# more units than the classes of one launch hold (1 GB: 335,000 at p = 10): the tiles in turns
def test_block_m2l_in_turns(G, ctx):
    x = inputs.plummer(1_000_000, 800)
    kw = dict(p=10, leaf_size=1, tree=G.TREE_ADAPTIVE)
    out = run(G, ctx, x, **kw)
    t = G.gbfmm_export_adaptive_tree(ctx, len(x))
    inner = len(np.unique(t["parent"])) - 1  # cells with children
    assert inner > 335_544
    ref = run(G, ctx, x, flags=G.FLAG_M2L_GATHERED, **kw)
    assert O.rel_l2(out[:, 0], ref[:, 0]) <= TOL and O.rel_l2(out[:, 1:], ref[:, 1:]) <= TOL
