"""A workspace planned for n particles serves fewer (gbfmm_plan's size never falls with n)."""
import pytest

from paper_1010_1482_gb300 import gbfmm as G


@pytest.mark.parametrize("p", [4, 6, 8, 10])
@pytest.mark.parametrize("leaf", [1, 32, 64, 1000])
def test_plan_is_monotone(p, leaf):
    edges = [leaf * 8**e for e in range(8)] + [1 << 17, 1 << 19, 1 << 20, 1 << 22]
    prm, last = G.gbfmm_default_params(p=p, leaf_size=leaf), 0
    for n in sorted({m + d for m in edges for d in (-1, 0, 1) if 0 < m + d <= 40_000_000}):
        try:
            _, ws = G.gbfmm_plan(prm, n)
        except G.GbfmmError as e:
            assert e.code == G.GBFMM_EUNSUPPORTED  # deeper than level 10
            break
        assert ws >= last, n
        last = ws
