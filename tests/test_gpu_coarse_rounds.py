"""Removal rounds on coarse clouds, whose searches climb several levels (needs a GPU).

A round's search without an order among equal distances takes its cells by two
lists: one of 27-bit distances on cells of up to 2^11 mm, one of 64-bit distances
beyond.  A search that needs both hands the farthest distance found over as a bound,
and every point at that distance has to stay wanted.  The clouds here have spacings
of 0.2 to 5 m and extents of 2^11 to 2^15 mm, so that queries end on either list or
pass from one to the other, with the whole cloud inside the last cube or not;
coordinates on a lattice make equal distances the rule.  Retained sets equal the
oracle's (section "Sub-sampling algorithm").
"""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


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


def _lattice(extent, step, frac, seed):
    """A random part of the lattice of this step, in random order."""
    r = np.random.default_rng(seed)
    i = np.arange(extent // step + 1) * step
    x = np.stack(np.meshgrid(i, i, i, indexing="ij"), axis=-1).reshape(-1, 3)
    x = x[r.random(len(x)) < frac]
    return np.ascontiguousarray(x[r.permutation(len(x))], dtype=np.int32)


def _clump(extent, seed):
    """A dense lattice in one corner, single points metres away from it, and a pair
    of opposite corners that fix the extent."""
    r = np.random.default_rng(seed)
    i = np.arange(6) * 160
    x = np.stack(np.meshgrid(i, i, i, indexing="ij"), axis=-1).reshape(-1, 3)
    far = r.integers(2, extent // 1024, (30, 3)) * 1024
    return np.unique(np.concatenate([x, far, [[0, 0, 0], [extent] * 3]]), axis=0).astype(np.int32)


CLOUDS = [
    ("2m", lambda: _lattice(2047, 190, 0.5, 1)),
    ("4m", lambda: _lattice(4095, 500, 0.9, 2)),
    ("8m_500", lambda: _lattice(8190, 500, 0.5, 0)),
    ("8m_1000", lambda: _lattice(8190, 1000, 0.5, 1)),
    ("8m_2340", lambda: _lattice(8190, 2340, 0.9, 0)),
    ("8m_2700", lambda: _lattice(8190, 2700, 0.9, 0)),
    ("16m_1900", lambda: _lattice(16383, 1900, 0.5, 3)),
    ("33m_4700", lambda: _lattice(32767, 4700, 0.9, 4)),
    ("clump_8m", lambda: _clump(8190, 5)),
    ("clump_30m", lambda: _clump(30000, 6)),
]


@pytest.mark.parametrize("k", [1, 2, 4, 5, 6, 16])
@pytest.mark.parametrize("name,cloud", CLOUDS, ids=[c[0] for c in CLOUDS])
def test_rounds(pd, ctx, name, cloud, k):
    x = cloud()
    n = len(x)
    for m in sorted({20, 40, n // 3, 2 * n // 3}):
        if m <= k or m >= n:
            continue
        ref = oracle.decimate(x, k, m)
        for leaf in (4, 8, 32):
            g = pd.Grid(ctx, torch.from_numpy(x).cuda(), leaf_max=leaf)
            keep = pd.pd_decimate_count(g, m, k=k).cpu().numpy()
            g.free()
            assert np.array_equal(keep, ref), (m, leaf)


@pytest.mark.parametrize("k", [1, 4])
def test_packed(pd, ctx, k):
    """The same clouds as the scans of one packed batch."""
    scans = [c() for _, c in CLOUDS]
    clouds = [{"xyz": torch.from_numpy(x).cuda(), "ratio": 0.3} for x in scans]
    keeps, _ = pd.pd_decimate_batch(ctx, clouds, k=k, concurrency=pd.PD_BATCH_PACKED)
    for x, keep in zip(scans, keeps):
        assert np.array_equal(keep.cpu().numpy(), oracle.decimate(x, k, oracle.target_count(len(x), 0.3)))
