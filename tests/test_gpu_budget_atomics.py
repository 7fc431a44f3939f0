"""Blocks that the rounds update with atomics stay in device memory (needs a GPU).

Under a device-memory budget large blocks are placed in pinned host memory.  The
bitmap of a round's candidates (a bit a point), a packed batch's histograms (16 KB a
scan) and the quality report's (64 KB a radius) take atomics on every round or query,
so they stay with the allocator whatever the budget and however large they are.
"""
import pytest

from paper_2311_17604_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SPILL_FLOOR = 1 << 20  # no smaller block ever leaves device memory


@pytest.fixture(scope="module")
def pd():
    from paper_2311_17604_gb300 import build
    build.build()
    import paper_2311_17604_gb300.pd as pdm
    return pdm


@pytest.fixture
def device_sizes(monkeypatch):
    """Bytes of every block that a context asks the allocator for."""
    sizes = []
    alloc = torch.cuda.caching_allocator_alloc

    def record(nbytes, **kw):
        sizes.append(nbytes)
        return alloc(nbytes, **kw)

    monkeypatch.setattr(torch.cuda, "caching_allocator_alloc", record)
    return sizes


def _rounded(nbytes):
    assert nbytes >= SPILL_FLOOR
    return (nbytes + 255) // 256 * 256


def test_candidate_bitmap(pd, device_sizes):
    n = 8500000
    x = torch.randint(0, 40000, (n, 3), dtype=torch.int32, device="cuda",
                      generator=torch.Generator(device="cuda").manual_seed(1))
    keeps = []
    for budget in (0, 1):
        del device_sizes[:]
        ctx = pd.Context()
        ctx.set_device_budget(budget)
        g = pd.Grid(ctx, x)
        keeps.append(pd.pd_decimate_count(g, n - 3000, k=2))
        g.free()
        ctx.close()
    assert _rounded((n + 31) // 32 * 4) in device_sizes
    assert torch.equal(keeps[0], keeps[1])


def test_batch_histograms(pd, device_sizes):
    scans = [synth.random_cloud(i, 600 + i, 4000) for i in range(70)]
    keeps = []
    for budget in (0, 1):
        del device_sizes[:]
        ctx = pd.Context()
        ctx.set_device_budget(budget)
        clouds = [{"xyz": torch.from_numpy(x).cuda(), "ratio": 0.4} for x in scans]
        keeps.append(pd.pd_decimate_batch(ctx, clouds, k=1, concurrency=pd.PD_BATCH_PACKED)[0])
        ctx.close()
    assert _rounded(len(scans) * 4096 * 4) in device_sizes
    assert all(torch.equal(a, b) for a, b in zip(*keeps))


def test_quality_histograms(pd, device_sizes):
    x = torch.from_numpy(synth.random_cloud(5, 4000, 2000)).cuda()
    radii = list(range(10, 200, 10))
    got = []
    for budget in (0, 1):
        del device_sizes[:]
        ctx = pd.Context()
        ctx.set_device_budget(budget)
        got.append(pd.pd_quality_report(ctx, x, None, radii)["fractile"])
        ctx.close()
    assert _rounded(len(radii) * pd.PD_QUALITY_HIST * 4) in device_sizes
    assert got[0] == got[1]
