"""Threshold selection over long lists of keys that agree in 24 bits (needs a GPU).

A lattice of 70^3 points has 343,000 equal costs at k = 1: the list of the first
round goes to one cluster of blocks, that of the second, once the first was long,
to the whole grid; in a packed batch it belongs to one scan among others.  Retained
sets equal the oracle's (section "Sub-sampling algorithm").
"""
import numpy as np
import pytest

import oracle
from paper_2311_17604_gb300 import synth

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


@pytest.fixture(scope="module")
def lattice():
    i = np.arange(70, dtype=np.int32) * 10
    x = np.stack(np.meshgrid(i, i, i, indexing="ij"), axis=-1).reshape(-1, 3)
    return np.ascontiguousarray(x[np.random.default_rng(1).permutation(len(x))])


@pytest.mark.parametrize("k,m", [(1, 171500), (1, 60000), (4, 300000)])
def test_one_cloud(pd, ctx, lattice, k, m):
    g = pd.Grid(ctx, torch.from_numpy(lattice).cuda())
    keep = pd.pd_decimate_count(g, m, k=k).cpu().numpy()
    g.free()
    assert np.array_equal(keep, oracle.decimate(lattice, k, m))


@pytest.mark.parametrize("k", [1, 6])
def test_wup(pd, ctx, lattice, k):
    m = 150000
    g = pd.Grid(ctx, torch.from_numpy(lattice).cuda())
    keep = pd.pd_decimate_wup(g, m, k=k).cpu().numpy()
    g.free()
    assert np.array_equal(keep, oracle.decimate_wup(lattice, k, m)[0])


@pytest.mark.parametrize("others", [2, 70, 300])
def test_one_scan_of_a_batch(pd, ctx, lattice, others):
    scans = [synth.random_cloud(i, 400 + 37 * i, 3000) for i in range(others)]
    scans.insert(others // 2, lattice)
    clouds = [{"xyz": torch.from_numpy(x).cuda(), "ratio": 0.3} for x in scans]
    keeps, _ = pd.pd_decimate_batch(ctx, clouds, k=1, concurrency=pd.PD_BATCH_PACKED)
    for x, keep in zip(scans, keeps):
        assert np.array_equal(keep.cpu().numpy(), oracle.decimate(x, 1, oracle.target_count(len(x), 0.3)))
