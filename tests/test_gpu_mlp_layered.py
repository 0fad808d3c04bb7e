"""The layer-by-layer form of the proposal network, which serves layers wider
than 256, more than 8 layers and more than 248 proposals per target: against
the oracle, and in turns with the four-launch form on one network."""
import numpy as np
import pytest

from oracle import mlp as omlp
from paper_2508_15522_gb300 import synth

pytestmark = pytest.mark.gpu
TILE = (11.28, 11.28)
# Of a tensor's scale: the products are those of bfloat16 operands on both sides; the FP32 order may
# turn the bfloat16 rounding of a single activation, 2^-8 of one term of a gradient.
REL = 2.0**-8


@pytest.fixture(scope="module")
def env():
    import __graft_entry__ as ge
    ge.build()
    from paper_2508_15522_gb300 import gridff
    ctx = gridff.Context(0)
    yield gridff, ctx
    ctx.close()


def data(sizes, B, K, seed):
    g = synth.rng(seed)
    X = g.standard_normal((B * K, sizes[0])).astype(np.float32)
    T = np.zeros((B, 19))
    T[:, :3] = g.random((B, 3)) * 5
    q = g.standard_normal((B, 4))
    T[:, 3:7] = q / np.linalg.norm(q, axis=1, keepdims=True)
    T[:, 7:] = g.uniform(-np.pi, np.pi, (B, 12))
    return X, T.astype(np.float32), (g.random((B, 12)) < 0.5).astype(np.float32)


def close(a, b):
    a, b = np.asarray(a, np.float64), np.asarray(b, np.float64)
    return np.abs(a - b).max() <= REL * max(np.abs(b).max(), 1e-30)


def weights(sizes, seed):
    Ws, bs = synth.mlp_weights(sizes, seed)
    return [W.astype(np.float32).astype(np.float64) for W in Ws], bs


WIDE, DEEP, FUSED = (40, 320, 64, 19), (24,) + (32,) * 8 + (19,), (40, 64, 48, 19)


@pytest.mark.parametrize("sizes, B, K", [(WIDE, 37, 3), (DEEP, 21, 2), (FUSED, 3, 249)])
def test_forward_and_gradients_match_the_oracle(env, sizes, B, K):
    G, ctx = env
    Ws, bs = weights(sizes, 3)
    net = G.MLP(ctx, sizes)
    net.set_params(Ws, bs)
    X, T, mask = data(sizes, B, K, 5)
    out, cache = omlp.forward(Ws, bs, X.astype(np.float64), mirror=True)
    assert close(net.forward(X), out)
    loss = net.train_step(X, T, K, G.train_params(lr=1e-3, tile=TILE), tors_mask=mask, update=False)
    # the winners by the library's own outputs: near ties are many among 249 proposals
    y = net.forward(X).astype(np.float64)
    L, dout, _ = omlp.wta_loss(y, T.astype(np.float64), mask.astype(np.float64), K, TILE)
    dWs, dbs = omlp.backward(Ws, cache, dout, mirror=True)
    assert loss == pytest.approx(L, rel=1e-3)
    gW, gb = net.unflatten(net.get_params()[1])
    for l in range(len(Ws)):
        assert close(gW[l], dWs[l]) and close(gb[l], dbs[l]), l
    net.close()


def test_forms_in_turn_share_the_weights(env):
    """Steps of 4 (four launches) and 249 proposals (layer by layer) by turns, then a
    forward pass of the trained parameters: neither form works on old operands."""
    G, ctx = env
    Ws, bs = weights(FUSED, 7)
    net = G.MLP(ctx, FUSED)
    net.set_params(Ws, bs)
    tp = G.train_params(lr=1e-2, tile=TILE)
    for turn in range(3):
        for B, K in ((30, 4), (2, 249)):
            X, T, mask = data(FUSED, B, K, 100 * turn + K)
            Wn, bn = net.unflatten(net.get_params()[0])
            Wn, bn = [W.astype(np.float64) for W in Wn], [b.astype(np.float64) for b in bn]
            out, _ = omlp.forward(Wn, bn, X.astype(np.float64), mirror=True)
            L, _, _ = omlp.wta_loss(out, T.astype(np.float64), mask.astype(np.float64), K, TILE)
            assert net.train_step(X, T, K, tp, tors_mask=mask) == pytest.approx(L, rel=5e-3)
            Wn, bn = net.unflatten(net.get_params()[0])
            out, _ = omlp.forward([W.astype(np.float64) for W in Wn], [b.astype(np.float64) for b in bn],
                                  X.astype(np.float64), mirror=True)
            assert close(net.forward(X), out)
    net.close()


def test_captured_loop_equals_its_split(env):
    """The captured loop in two calls gives the bits of one, also after steps of the other
    form have moved the weights."""
    G, ctx = env
    _, T, mask = data(FUSED, 50, 1, 9)
    desc = synth.rng(1).random(24).astype(np.float32)
    out = []
    for calls in ((6,), (2, 4)):
        net = G.MLP(ctx, FUSED)
        net.set_params(*weights(FUSED, 8))
        net.set_targets(T, mask)
        tp = G.train_params(lr=1e-3, tile=TILE)
        net.train(3, 16, 4, desc, 5, tp)
        loss = np.concatenate([net.train(k, 4, 249, desc, 5, tp) for k in calls])
        out.append((loss, net.get_params()[0]))
        net.close()
    assert np.isfinite(out[0][0]).all()
    assert np.array_equal(out[0][0], out[1][0]) and np.array_equal(out[0][1], out[1][1])


def test_both_forms_give_the_same_bits(env):
    """A network that the four launches serve, and the same one with 200 idle units in
    its second layer (no weights, no biases), which goes layer by layer: outputs,
    gradients and two Adam steps of 111 rows (one part each in the sums over rows)."""
    G, ctx = env
    Ws, bs = weights(FUSED, 11)
    big = (FUSED[0], FUSED[1] + 200) + FUSED[2:]
    Wb = [np.zeros((j, i)) for i, j in zip(big[:-1], big[1:])]
    bb = [np.zeros(j) for j in big[1:]]
    for l, (W, b) in enumerate(zip(Ws, bs)):
        Wb[l][:W.shape[0], :W.shape[1]] = W
        bb[l][:len(b)] = b
    X, T, mask = data(FUSED, 37, 3, 12)
    tp = G.train_params(lr=1e-3, tile=TILE)
    out = []
    for sizes, W, b in ((FUSED, Ws, bs), (big, Wb, bb)):
        net = G.MLP(ctx, sizes)
        net.set_params(W, b)
        res = [net.forward(X), np.float32(net.train_step(X, T, 3, tp, tors_mask=mask))]
        res.append(np.float32(net.train_step(X, T, 3, tp, tors_mask=mask)))
        for flat in net.get_params():
            Wn, bn = net.unflatten(flat)
            for l, (w0, b0) in enumerate(zip(Ws, bs)):
                res += [Wn[l][:w0.shape[0], :w0.shape[1]], bn[l][:len(b0)]]
        out.append(res)
        net.close()
    for a, b in zip(*out):
        assert np.array_equal(a, b)
