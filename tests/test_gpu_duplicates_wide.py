"""Coincident points in clouds beyond 2^21 mm (needs a GPU).

Such a cloud's Morton cells are 2 mm and more wide, so coincident points need not be
neighbours in the Morton order: others of their cell lie between them.  They are the
first to go all the same, the largest input index first (section "Computing per-sample
costs": their cost is infinite), and a packed batch with more of them than a scan
must lose runs its scans apart.  Retained sets equal the oracle's.
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


def _cloud(seed, span, cells=60, each=40, width=3):
    """Points on few positions of far-apart cells, in random order."""
    r = np.random.default_rng(seed)
    at = r.integers(0, span - width, (cells, 3)) & ~15
    at[:2] = [[0, 0, 0], [span - 16] * 3]
    x = np.repeat(at, each, axis=0) + r.integers(0, width, (cells * each, 3))
    return np.ascontiguousarray(x[r.permutation(len(x))], dtype=np.int32)


@pytest.mark.parametrize("k", [1, 4])
@pytest.mark.parametrize("span", [1 << 20, 1 << 22, 1 << 24, 1 << 25])
def test_one_cloud(pd, ctx, span, k):
    x = _cloud(span, span)
    n, distinct = len(x), len(np.unique(x, axis=0))
    for m in (n - 7, n - 300, distinct, distinct - 50, distinct // 3):
        g = pd.Grid(ctx, torch.from_numpy(x).cuda())
        keep = pd.pd_decimate_count(g, m, k=k).cpu().numpy()
        g.free()
        assert np.array_equal(keep, oracle.decimate(x, k, m)), m


@pytest.mark.parametrize("k", [1, 4])
@pytest.mark.parametrize("ratio", [0.97, 0.8, 0.3, 0.1])
def test_packed(pd, ctx, k, ratio):
    scans = [_cloud(i, 1 << 20, cells=20) for i in range(4)] + [_cloud(9, 1 << 22)]
    clouds = [{"xyz": torch.from_numpy(x).cuda(), "ratio": ratio} for x in scans]
    keeps, _ = pd.pd_decimate_batch(ctx, clouds, k=k, concurrency=pd.PD_BATCH_PACKED)
    for x, keep in zip(scans, keeps):
        assert np.array_equal(keep.cpu().numpy(), oracle.decimate(x, k, oracle.target_count(len(x), ratio)))
