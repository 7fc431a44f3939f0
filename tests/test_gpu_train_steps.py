"""The overlapped launches of a training call, bit for bit (needs a GPU).

Within a call a step's gradient launch may start before the step ahead of it has
finished; the first step of a call may not.  N steps in one call and N calls of one
step must give the same weights, Adam state and losses in every bit: a step that read
the weights or the partial sums of any other step would differ.
"""
import numpy as np
import pytest

from oracle import normals as N

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("batch", [1, 65, 4096, 40000])
def test_one_call_equals_calls_of_one_step(batch):
    from paper_2311_17604_gb300 import build
    build.build()
    import paper_2311_17604_gb300.pd as pd
    rng = np.random.default_rng(batch)
    x = N.round_bf16(rng.uniform(-1, 1, (3000, N.NF)))
    feat = torch.from_numpy(N.bf16_bits(x).view(np.int16).copy()).cuda()
    y = rng.standard_normal((3000, 3))
    y = torch.from_numpy((y / np.linalg.norm(y, axis=1, keepdims=True)).astype(np.float32)).cuda()
    valid = torch.from_numpy((rng.random(3000) < 0.7).astype(np.uint8)).cuda()
    start = torch.from_numpy(N.init_params(4).astype(np.float32)).cuda()
    ctx = pd.Context()
    kw = dict(valid=valid, batch=batch, lr=1e-2, seed=6)
    one = pd.MlpTrainer(params=start.clone())
    losses = one.train(ctx, feat, y, steps=12, **kw)
    each = pd.MlpTrainer(params=start.clone())
    parts = [each.train(ctx, feat, y, steps=1, **kw) for _ in range(12)]
    ctx.close()
    assert torch.equal(losses, torch.cat(parts))
    assert torch.equal(one.params, each.params)
    assert torch.equal(one.adam, each.adam)
    assert not torch.equal(one.params, start)
