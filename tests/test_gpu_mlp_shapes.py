"""The emulator's fused kernels over widths, depths and row counts where a block
of rows, a chunk of weights or a gradient tile is partly filled, against the
float64 oracle with the bounds of a bf16 network (outputs 2e-2 of their spread,
gradients cosine >= 0.999 and relative L2 <= 2e-2), predictions bit for bit the
same at every row count, and one Adam step against the update formed from the
library's own float32 gradients."""

import numpy as np
import pytest

from oracle import mlp as OM

pytestmark = pytest.mark.gpu


def _bf16(a):
    u = np.asarray(a, np.float32).view(np.uint32).astype(np.uint64)
    return ((((u + 0x7FFF + ((u >> 16) & 1)) >> 16) << 16).astype(np.uint32)).view(np.float32).astype(np.float64)


def _emulator(n_in, width, depth):
    import paper_2501_12928_gb300 as P
    em = P.Emulator(n_in, width, depth, seed=3)
    norm = (np.full(n_in, 0.1, np.float32), np.full(n_in, 0.5, np.float32), 40.0, 20.0)
    em.set_norm(*norm)
    rng = np.random.default_rng(width + depth)
    for layer in range(depth + 1):   # biases that matter
        W, b = em.get_params(layer)
        em.set_params(layer, W, rng.uniform(-0.3, 0.3, b.shape).astype(np.float32))
    params = [(_bf16(W), b.astype(np.float64)) for W, b in (em.get_params(l) for l in range(depth + 1))]
    return em, norm, params


def _data(n, n_in):
    rng = np.random.default_rng(n)
    x = rng.uniform(-2, 2, (n, n_in)).astype(np.float32)
    return x, (50.0 - 3.0 * np.sum((x - 0.3) ** 2, axis=1)).astype(np.float32)


SHAPES = [(1, 16, 1), (9, 48, 2), (16, 240, 4), (9, 256, 8), (5, 64, 5)]


@pytest.mark.parametrize("n_in,width,depth", SHAPES)
def test_forward(n_in, width, depth):
    em, norm, params = _emulator(n_in, width, depth)
    x, _ = _data(5003, n_in)
    y = em.infer(x)
    ref = OM.forward(params, x.astype(np.float64), norm[0], norm[1])[0] * norm[3] + norm[2]
    assert np.linalg.norm(y - ref) <= 2e-2 * np.linalg.norm(ref - ref.mean()) + 1e-3 * np.linalg.norm(ref)
    for n in (1, 15, 17, 64, 4864, 4865):   # a row's operations do not depend on how many there are
        np.testing.assert_array_equal(em.infer(x[:n]), y[:n])


@pytest.mark.parametrize("n_in,width,depth", SHAPES)
def test_gradients_and_adam_step(n_in, width, depth):
    em, norm, params = _emulator(n_in, width, depth)
    lr, b1, b2, eps = 1e-3, 0.9, 0.999, 1e-8
    for n in (63, 300, 1025):
        x, t = _data(n, n_in)
        params = [(_bf16(W), b.astype(np.float64)) for W, b in (em.get_params(l) for l in range(depth + 1))]
        loss, ref = OM.loss_and_grads(params, x.astype(np.float64), t.astype(np.float64), norm[0].astype(np.float64),
                                      norm[1].astype(np.float64), norm[2], norm[3])
        for layer in range(depth + 1):
            dW, db, got = em.grad(x, t, layer)
            gr = ref[layer][0]
            assert np.sum(dW * gr) >= 0.999 * np.linalg.norm(dW) * np.linalg.norm(gr)
            assert np.linalg.norm(dW - gr) <= 2e-2 * np.linalg.norm(gr)
            assert np.linalg.norm(db - ref[layer][1]) <= 2e-2 * np.linalg.norm(ref[layer][1])
            assert abs(got - loss) <= 2e-2 * loss
    # first step of Adam: m / c1 = g, v / c2 = g^2, each to a few float32 roundings
    grads = [em.grad(x, t, layer)[:2] for layer in range(depth + 1)]
    before = [em.get_params(layer) for layer in range(depth + 1)]
    em.train_step(x, t, lr, b1, b2, eps)
    for layer in range(depth + 1):
        for p, g, q in zip(before[layer], grads[layer], em.get_params(layer)):
            g = g.astype(np.float64)
            want = p - lr * g / (np.abs(g) + eps)
            # 12 roundings of the step, and 1 - b2 in float32 (2^-24 / 0.001 of v, half of it in the step)
            tol = lr * (12 * 2.0 ** -24 + 2.0 ** -24 / 0.001) + 2.0 ** -24 * np.abs(p).max()
            assert np.abs(q - want).max() <= tol


@pytest.mark.parametrize("n_in,width,depth", [(9, 48, 2), (9, 256, 4)])
def test_forward_of_many_rows(n_in, width, depth):
    """Whole waves of rows and a rest (on 152 SMs 19,456 rows and up to 2,432)."""
    em, _, _ = _emulator(n_in, width, depth)
    x, _ = _data(41500, n_in)
    y = np.concatenate([em.infer(x[i:i + 4000]) for i in range(0, len(x), 4000)])
    for n in (19455, 19456, 19457, 21888, 21889, 38912, 38913, 41500):
        np.testing.assert_array_equal(em.infer(x[:n]), y[:n])
