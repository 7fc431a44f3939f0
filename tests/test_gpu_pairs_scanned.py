"""The first pass's count of scanned pairs covers every query (needs a GPU).

pd_stats.pairs_first counts the (query, candidate) pairs of the first neighbour pass,
on whichever kernel a query ends: a query that takes its S nearest has scanned S
others at least (S = 8 up to k = 6, else 17; for the k = 1 density cost 2 settle it).
"""
import numpy as np
import pytest

from paper_2311_17604_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _dense_spot():
    """3000 points in cells that no level splits, in a cloud of 33 km."""
    return np.concatenate([synth.random_cloud(1, 3000, 30), synth.random_cloud(2, 400, (1 << 25) - 1)])


CLOUDS = {
    "room": lambda: synth.room_scan(seed=1, n_az=200, n_el=50).xyz,
    "sparse": lambda: synth.random_cloud(3, 4000, 1 << 24),
    "coarse": lambda: synth.random_cloud(4, 3000, 20000),
    "dense_spot": _dense_spot,
}


@pytest.mark.parametrize("k,colour", [(1, False), (4, False), (16, False), (4, True), (16, True)])
@pytest.mark.parametrize("name", sorted(CLOUDS))
def test_every_query_counts(name, k, colour):
    from paper_2311_17604_gb300 import build
    build.build()
    import paper_2311_17604_gb300.pd as pd
    x = np.unique(CLOUDS[name](), axis=0)
    rgb = torch.zeros((len(x), 3), dtype=torch.uint8, device="cuda") if colour else None
    ctx = pd.Context()
    g = pd.Grid(ctx, torch.from_numpy(x).cuda(), rgb=rgb)
    pd.pd_decimate_count(g, len(x) - 1, k=k, term=pd.PD_TERM_COLOR if colour else pd.PD_TERM_NONE,
                         weight=0.3 if colour else 0.0)
    st = g.stats()
    g.free()
    ctx.close()
    assert st["q_first"] == len(x)
    least = 2 if k == 1 and not colour else (8 if k <= 6 else 17)
    assert st["pairs_first"] >= len(x) * least
