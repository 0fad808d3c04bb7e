"""The launches of a training loop overlap (a launch starts while the one before
it runs); a call of one step has nothing to overlap with its neighbours.  Both
give the same bits, whatever the launches' sizes: one block, a ragged few, and
more blocks than the chip holds at once."""
import numpy as np
import pytest

from paper_2508_15522_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sizes, B, K, steps", [((24, 16, 19), 1, 1, 60), ((70, 48, 256, 19), 33, 5, 40),
                                                ((80, 256, 256, 256, 19), 256, 8, 40),
                                                ((80, 256, 64, 19), 2100, 4, 12)])
def test_one_call_equals_single_steps(sizes, B, K, steps):
    import __graft_entry__ as ge
    ge.build()
    from paper_2508_15522_gb300 import gridff as G
    g = synth.rng(B)
    T = g.uniform(-1, 1, (500, 19))
    T[:, 3:7] /= np.linalg.norm(T[:, 3:7], axis=1, keepdims=True)
    mask = (g.random((500, 12)) < 0.5).astype(np.float32)
    desc = g.random(min(64, sizes[0] - 8)).astype(np.float32)
    out = []
    ctx = G.Context(0)
    Ws, bs = synth.mlp_weights(sizes, 3)
    for calls in ([steps], [1] * steps):
        net = G.MLP(ctx, sizes)
        net.set_params(Ws, bs)
        net.set_targets(T.astype(np.float32), mask)
        loss = np.concatenate([net.train(n, B, K, desc, 9, G.train_params(lr=1e-3, tile=(9.0, 9.0))) for n in calls])
        out.append((loss, net.get_params()))
        net.close()
    ctx.close()
    assert np.isfinite(out[0][0]).all() and np.array_equal(out[0][0], out[1][0])
    for a, b in zip(out[0][1], out[1][1]):
        for u, v in zip(a, b):
            assert np.array_equal(u, v)
