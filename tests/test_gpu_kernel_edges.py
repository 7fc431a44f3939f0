"""Edges of the kernels' tiles and of their dispatch rules (needs a GPU).

  * the full neighbour pass: clouds at which its 32-bit keys do not suffice and
    a query moves to the warp-per-query search (cells too wide for a key, more
    candidates than a group holds, equal distances at the end of a list), and
    clouds of fewer points than a list stores;
  * threshold selection, buffer update and candidate test: clouds one point
    around the sizes their blocks take, and many equal keys;
  * quality report: 64-bit distances, more nodes than a block lists, more than
    8 radii;
  * network: rows around the tiles of inference (32) and training (64), and
    arrays that start off a 16-byte boundary.

Density costs, retained sets and counts equal the oracle's exactly.  A weighted
cost of k positive terms takes at most 16 roundings a term on either side and k
in the sum: 2 (16 + k) 2^-53 relative.  The network's bound is that of the
bfloat16 operands (2^-8), see the gradient test.
"""
import numpy as np
import pytest

import oracle
from oracle import normals as N
from oracle import quality
from paper_2311_17604_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

U_BF16 = 2.0 ** -8
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


def _lattice(side, step):
    i = np.arange(side, dtype=np.int32) * step
    return np.stack(np.meshgrid(i, i, i, indexing="ij"), axis=-1).reshape(-1, 3).copy()


def _clump():
    # 4000 points on 27 positions inside a sparse cloud
    return np.concatenate([synth.random_cloud(11, 4000, 3), synth.random_cloud(12, 600, 4000)])


CLOUDS = {
    "n2": lambda: synth.random_cloud(1, 2, 50),
    "n7": lambda: synth.random_cloud(2, 7, 50),
    "n17": lambda: synth.random_cloud(3, 17, 50),
    "n33": lambda: synth.random_cloud(4, 33, 50),
    "widest": lambda: synth.random_cloud(5, 2500, (1 << 25) - 1),
    "lattice": lambda: _lattice(13, 10),
    "clump": _clump,
}


def _d2(xyz, idx):
    x = xyz.astype(np.int64)
    d = x[np.maximum(idx, 0)] - x[:, None, :]
    return np.where(idx >= 0, (d * d).sum(axis=2), oracle.D2_NONE)


@pytest.mark.parametrize("k", [1, 6, 16])
@pytest.mark.parametrize("name", sorted(CLOUDS))
def test_full_pass(pd, ctx, name, k):
    x = CLOUDS[name]()
    g = pd.Grid(ctx, torch.from_numpy(x).cuda())
    cost, knn = (t.cpu().numpy() for t in pd.pd_knn_cost(g, k=k))
    g.free()
    d2, _, ref = oracle.knn_cost(x, k)
    assert np.array_equal(_d2(x, knn), d2)
    assert np.array_equal(cost, ref)


@pytest.mark.parametrize("k", [1, 6, 16])
@pytest.mark.parametrize("name", ["lattice", "n7", "widest"])
def test_full_pass_weighted(pd, ctx, name, k):
    """Equal distances enter in the order of the input index."""
    x = CLOUDS[name]()
    rgb = np.random.default_rng(6).integers(0, 256, (len(x), 3)).astype(np.uint8)
    g = pd.Grid(ctx, torch.from_numpy(x).cuda(), rgb=torch.from_numpy(rgb).cuda())
    cost, knn = pd.pd_knn_cost(g, k=k, term=pd.PD_TERM_COLOR, weight=0.3)
    g.free()
    _, idx, ref = oracle.knn_cost(x, k, term=oracle.TERM_COLOR, a=0.3, rgb=rgb)
    assert np.array_equal(knn.cpu().numpy(), idx)
    assert np.all(np.abs(cost.cpu().numpy() - ref) <= 2 * (16 + k) * U64 * np.abs(ref))


@pytest.mark.parametrize("k", [1, 2, 4])
@pytest.mark.parametrize("n", [3, 31, 33, 511, 513, 1023, 1025, 2047, 2049, 8193])
def test_rounds_at_block_edges(pd, ctx, n, k):
    x = synth.random_cloud(n, n, 400)
    for m in (1, n // 3, n - 1):
        g = pd.Grid(ctx, torch.from_numpy(x).cuda())
        keep = pd.pd_decimate_count(g, m, k=k).cpu().numpy()
        g.free()
        assert np.array_equal(keep, oracle.decimate(x, k, m)), (n, k, m)


@pytest.mark.parametrize("k", [1, 4])
def test_rounds_equal_keys(pd, ctx, k):
    """A threshold among thousands of equal costs is settled by the input index."""
    x = _lattice(17, 10)
    x = x[np.random.default_rng(7).permutation(len(x))].copy()
    for m in (500, 4000):
        g = pd.Grid(ctx, torch.from_numpy(x).cuda())
        keep = pd.pd_decimate_count(g, m, k=k).cpu().numpy()
        g.free()
        assert np.array_equal(keep, oracle.decimate(x, k, m)), m


@pytest.mark.parametrize("name,radii", [
    ("widest", [3000000, 6000000]),
    ("widest", [9000, 2000000]),
    ("clump", [1, 2, 3, 400]),
    ("clump", [1, 2, 4, 8, 16, 32, 64, 128, 256]),
    ("n33", [1, 20, 100]),
    ("lattice", [9, 10, 14, 15, 17, 18, 8192]),
])
def test_quality(pd, ctx, name, radii):
    x = CLOUDS[name]()
    got = pd.pd_quality_report(ctx, torch.from_numpy(x).cuda(), None, radii)
    ref = quality.report(x, None, radii)
    assert got["points"] == ref["points"]
    assert got["fractile"] == ref["fractile"]
    assert np.allclose(got["mean"], ref["mean"], rtol=1e-12, atol=0)
    assert got["min_spacing2_mm2"] == ref["min_spacing2_mm2"]
    assert got["mean_spacing_mm"] == pytest.approx(ref["mean_spacing_mm"], rel=1e-9)


def _off_boundary(t):
    """A copy whose data starts 4 bytes past a 16-byte boundary."""
    step = 4 // t.element_size()
    buf = torch.empty(t.numel() + 16, dtype=t.dtype, device=t.device)
    out = buf[step:step + t.numel()].view(t.shape)
    out.copy_(t)
    assert out.data_ptr() % 16 == 4
    return out


def _rows(n, seed):
    """Feature rows as bfloat16 bits and a perturbed network."""
    rng = np.random.default_rng(seed)
    x = N.round_bf16(rng.uniform(-1, 1, (n, N.NF)))
    feat = torch.from_numpy(N.bf16_bits(x).view(np.int16).copy()).cuda()
    p = N.init_params(seed).astype(np.float32)
    p += (0.05 * rng.standard_normal(N.N_PARAMS)).astype(np.float32)
    return x, feat, p, torch.from_numpy(p).cuda()


@pytest.mark.parametrize("n", [1, 31, 32, 33, 255, 257])
def test_forward_rows(pd, n):
    x, feat, p, pc = _rows(n, n)
    u, nr = pd.pd_mlp_forward(pc, feat)
    _, _, o, ref = N.forward(p, x)
    assert N.angle(u.cpu().numpy(), ref).max() < 4 * U_BF16
    ref_nr = np.linalg.norm(o, axis=1)
    assert (np.abs(nr.cpu().numpy() - ref_nr) / ref_nr).max() < 4 * U_BF16
    u2, nr2 = pd.pd_mlp_forward(_off_boundary(pc), _off_boundary(feat))
    assert torch.equal(u, u2) and torch.equal(nr, nr2)


@pytest.mark.parametrize("n", [1, 16, 17, 63, 64, 65, 129, 1000])
def test_gradient_rows(pd, ctx, n):
    """Labels at 45 degrees to the outputs, so that no gradient cancels: what is
    left is the operands' rounding, 2 units of bfloat16 per block at most."""
    x, feat, p, pc = _rows(n, 100 + n)
    _, _, o, u = N.forward(p, x)
    v = np.cross(u, np.roll(u, 1, axis=1) + [0.3, 0.0, 0.0])
    y = u + v / np.linalg.norm(v, axis=1, keepdims=True)
    y = (y / np.linalg.norm(y, axis=1, keepdims=True)).astype(np.float32)
    loss, g = pd.pd_mlp_grad(ctx, pc, feat, torch.from_numpy(y).cuda())
    ref_loss, ref = N.grad(p, x, y)
    assert abs(loss - ref_loss) <= 2 * U_BF16 * ref_loss
    gh = g.cpu().numpy().astype(np.float64)
    ends = (N.O_W1, N.O_B1, N.O_W2, N.O_B2, N.O_W3, N.O_B3, N.N_PARAMS)
    for lo, hi in zip(ends, ends[1:]):
        err = np.linalg.norm(gh[lo:hi] - ref[lo:hi])
        assert err <= 2 * U_BF16 * np.linalg.norm(ref[lo:hi]), lo
    _, g2 = pd.pd_mlp_grad(ctx, _off_boundary(pc), _off_boundary(feat), torch.from_numpy(y).cuda())
    assert torch.equal(g, g2)


@pytest.mark.parametrize("batch", [1, 65, 300])
def test_training_steps_are_gradient_and_adam(pd, ctx, batch):
    """The overlapped launches of a training call give the steps that the
    gradient entry and Adam's formula give one at a time, with the weights of
    the step before: Adam moves a weight by lr g / (|g| + eps), so a weight
    whose gradient is near zero may move otherwise; the losses may not."""
    x, feat, p, pc = _rows(400, 9)
    _, _, _, u = N.forward(p, x)
    y = np.roll(u, 1, axis=0).astype(np.float32)
    tr = pd.MlpTrainer(params=pc.clone())
    losses = tr.train(ctx, feat, torch.from_numpy(y).cuda(), steps=5, batch=batch, lr=1e-3, seed=3)
    _, ref = N.train(p, x, y, np.ones(400, bool), 5, batch, 1e-3, seed=3)
    # |d loss| <= 2 |d u|, and the outputs agree to 4 units
    assert np.abs(losses.cpu().numpy() - ref).max() <= 8 * U_BF16


@pytest.mark.parametrize("n", [1, 2048, 2049, 4097, 2490367, 2700001])
def test_sort_is_stable(pd, ctx, n):
    """The sort keeps the input order of equal codes (full and half tiles, ragged
    ends): with as many points kept as there are positions, the first point of
    every position stays."""
    x = np.random.default_rng(n).integers(0, 40, (n, 3)).astype(np.int32) * [1, 3, 700]
    x = np.ascontiguousarray(x, dtype=np.int32)
    _, first = np.unique(x @ np.array([1, 10 ** 3, 10 ** 5], np.int64), return_index=True)
    g = pd.Grid(ctx, torch.from_numpy(x).cuda())
    keep = pd.pd_decimate_count(g, len(first), k=1).cpu().numpy()
    g.free()
    ref = np.zeros(n, np.uint8)
    ref[first] = 1
    assert np.array_equal(keep, ref)
