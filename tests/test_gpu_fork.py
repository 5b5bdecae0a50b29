"""Forked evaluations (P2P and M2P beside the M2L): their stage times, and no slower than serial ones."""
import numpy as np
import pytest

from paper_1010_1482_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


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


def timed(G, ctx, n, flags=0, reps=15, **kw):
    """Median evaluation time in us (adaptive tree, Plummer sphere) and, if asked for, of the stages."""
    x = torch.from_numpy(inputs.plummer(n, 900)).cuda()
    out = torch.empty_like(x)
    ws = torch.empty(256, dtype=torch.uint8, device="cuda")
    prm = G.gbfmm_default_params(tree=G.TREE_ADAPTIVE, flags=flags, **kw)
    ts, st = [], []
    for i in range(reps + 3):
        a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
        a.record()
        G.gbfmm_evaluate(ctx, prm, x, out, ws)
        b.record()
        G.gbfmm_sync_status(ctx)
        if i >= 3:
            ts.append(1e3 * a.elapsed_time(b))
            if flags & G.FLAG_STAGE_TIMING:
                st.append(G.gbfmm_stage_times(ctx))
    return float(np.median(ts)), {k: 1e3 * float(np.median([s[k] for s in st])) for k in (st[0] if st else ())}


def test_fork_of_heavy_leaves(G, ctx):
    """P2P of few heavy leaves bounds this evaluation: beside the far field it takes what it takes
    alone or a little more (crowded onto the SMs that P2M left free it took a third more)."""
    kw = dict(p=10, leaf_size=1024)
    assert timed(G, ctx, 100_000, **kw)[0] <= 1.05 * timed(G, ctx, 100_000, flags=G.FLAG_SERIAL, **kw)[0]


@pytest.mark.parametrize("n,p,leaf", [(100_000, 10, 64), (20_000, 10, 512)])
def test_stage_times_hold_m2p(G, ctx, n, p, leaf):
    """M2P over the W rows is part of the reported L2P stage, serial or forked, on either stream."""
    kw = dict(p=p, leaf_size=leaf)
    serial = timed(G, ctx, n, flags=G.FLAG_SERIAL | G.FLAG_STAGE_TIMING, **kw)[1]
    fork = timed(G, ctx, n, flags=G.FLAG_STAGE_TIMING, **kw)[1]
    assert fork["L2P"] >= 0.75 * serial["L2P"], (fork, serial)


@pytest.mark.parametrize("n,p,leaf,flags", [(20_000, 10, 512, 0), (100_000, 6, 64, 2)])
def test_m2p_stays_off_the_longer_side(G, ctx, n, p, leaf, flags):
    """Where P2P is the longer side (512 a leaf), or the M2L's CTAs crowd (CUDA cores, p = 6), M2P is
    not put before the end of either: the fork keeps hiding what it can."""
    kw = dict(p=p, leaf_size=leaf)
    a, b = (timed(G, ctx, n, flags=flags | f, **kw)[0] for f in (0, G.FLAG_SERIAL))
    assert a <= {512: 0.85, 64: 1.05}[leaf] * b, (a, b)
