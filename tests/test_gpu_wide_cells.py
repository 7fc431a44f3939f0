"""Full neighbour passes over cells of any width (needs a GPU).

The leaf-group kernel orders a group's candidates by 32-bit keys.  Where the largest
distance does not fit beside a candidate's number, the keys hold its leading bits
and the exact distances settle the rest, so clouds of any spacing, with equal and
nearly equal distances, must give the oracle's neighbours and costs: densities in
every bit, weighted costs within the roundings of k terms (16 a term and k in the
sum on either side: 2 (16 + k) 2^-53 relative) and their neighbours in the order of
(distance, input index).
"""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

U64 = 2.0 ** -53


@pytest.fixture(scope="module")
def pd():
    from paper_2311_17604_gb300 import build
    build.build()
    import paper_2311_17604_gb300.pd as pdm
    return pdm


@pytest.fixture(scope="module")
def ctx(pd):
    c = pd.Context()
    yield c
    c.close()


def _terrain(spacing, n=3000):
    r = np.random.default_rng(spacing)
    x = r.uniform(0, spacing * n ** 0.5, (n, 3))
    x[:, 2] *= 0.02
    return x.astype(np.int32)


def _raster(spacing, side=55):
    """A gridded height model: equal distances on level ground, a slope beside it."""
    i = np.arange(side)
    a, b = (v.reshape(-1) for v in np.meshgrid(i, i, indexing="ij"))
    x = np.stack([a * spacing, b * spacing, np.maximum(a - 20, 0) * (spacing // 7)], axis=1)
    return np.ascontiguousarray(x[np.random.default_rng(1).permutation(len(x))], dtype=np.int32)


def _near_ties(spacing, n=3000):
    """A lattice moved by a millimetre or none: distances that differ in the last bits."""
    r = np.random.default_rng(2)
    i = np.arange(15) * spacing
    x = np.stack(np.meshgrid(i, i, i, indexing="ij"), axis=-1).reshape(-1, 3)[:n]
    return np.ascontiguousarray(x + r.integers(0, 2, x.shape), dtype=np.int32)


CLOUDS = [
    ("terrain_40", lambda: _terrain(40)),
    ("terrain_300", lambda: _terrain(300)),
    ("terrain_1000", lambda: _terrain(1000)),
    ("terrain_5000", lambda: _terrain(5000)),
    ("terrain_600000", lambda: _terrain(600000)),
    ("raster_1000", lambda: _raster(1000)),
    ("raster_5600", lambda: _raster(5600)),
    ("ties_900", lambda: _near_ties(900)),
    ("ties_7000", lambda: _near_ties(7000)),
    ("ties_2000000", lambda: _near_ties(2000000)),
]


@pytest.mark.parametrize("k", [1, 6, 7, 16])
@pytest.mark.parametrize("name,cloud", CLOUDS, ids=[c[0] for c in CLOUDS])
def test_density(pd, ctx, name, cloud, k):
    x = cloud()
    d2, _, ref = oracle.knn_cost(x, k)
    for leaf in (4, 32):
        g = pd.Grid(ctx, torch.from_numpy(x).cuda(), leaf_max=leaf)
        cost, knn = (t.cpu().numpy() for t in pd.pd_knn_cost(g, k=k))
        g.free()
        y = x.astype(np.int64)
        d = y[np.maximum(knn, 0)] - y[:, None, :]
        assert np.array_equal((d * d).sum(axis=2), d2)
        assert all(len(set(r)) == k for r in knn.tolist())
        assert np.array_equal(cost, ref)


@pytest.mark.parametrize("k", [1, 6, 7, 16])
@pytest.mark.parametrize("name,cloud", CLOUDS, ids=[c[0] for c in CLOUDS])
def test_weighted(pd, ctx, name, cloud, k):
    x = cloud()
    rgb = np.random.default_rng(6).integers(0, 256, (len(x), 3)).astype(np.uint8)
    _, idx, ref = oracle.knn_cost(x, k, term=oracle.TERM_COLOR, a=0.3, rgb=rgb)
    for leaf in (4, 32):
        g = pd.Grid(ctx, torch.from_numpy(x).cuda(), rgb=torch.from_numpy(rgb).cuda(), leaf_max=leaf)
        cost, knn = pd.pd_knn_cost(g, k=k, term=pd.PD_TERM_COLOR, weight=0.3)
        g.free()
        assert np.array_equal(knn.cpu().numpy(), idx)
        assert np.all(np.abs(cost.cpu().numpy() - ref) <= 2 * (16 + k) * U64 * np.abs(ref))


@pytest.mark.parametrize("k", [1, 4])
@pytest.mark.parametrize("name,cloud", CLOUDS[1:], ids=[c[0] for c in CLOUDS[1:]])
def test_decimation(pd, ctx, name, cloud, k):
    """The stored lists behind the costs: a decimation lives on them."""
    x = cloud()
    m = len(x) // 4
    g = pd.Grid(ctx, torch.from_numpy(x).cuda())
    keep = pd.pd_decimate_count(g, m, k=k).cpu().numpy()
    g.free()
    assert np.array_equal(keep, oracle.decimate(x, k, m))
