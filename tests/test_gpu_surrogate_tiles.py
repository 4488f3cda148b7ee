"""The surrogate's fused kernels at the edges of their tiles.

Inference works on pairs of 128-row tiles, one CTA each, and a row's answer
depends on that row alone: any prefix of a prediction equals the prediction
of the prefix bit for bit, whatever tile, CTA or turn of the loop it falls in,
and rows with infinities or NaN leave their neighbours as they are.

Training works on 128-row tiles of a minibatch, four CTAs to a tile: losses
and gradients at row counts around the edges of 16, 128 and 512 rows against
the FP64 oracle on the BF16-rounded weights and inputs, within the 2e-2 that
BF16 activations and gradients are held to elsewhere (2^-9 per rounding, a
dozen of them on the longest path).
"""

import numpy as np
import pytest

import oracle as O
from paper_2005_02498_gb300 import ptadd
from test_gpu_mlp import DIMS, MAT, bf16, relfro, split, target_fn, weights_bf16

pytestmark = pytest.mark.gpu


def features(rng, n):
    return np.hstack([rng.uniform(-220e6, 220e6, size=(n, 6)), 10 ** rng.uniform(10.8, 13.2, size=(n, 24))])


@pytest.fixture(scope="module")
def fitted():
    rng = np.random.default_rng(41)
    fit = np.hstack([rng.uniform(-200e6, 200e6, size=(2048, 6)), 10 ** rng.uniform(11, 13, size=(2048, 24))])
    with ptadd.Context(MAT, ptadd.PTADD_FP64, 0) as c:
        c.surrogate_fit(fit, np.tanh(fit[:, :6] / 1e8) * 20.0, epochs=4, batch=256, lr=2e-3, seed=5)
        test = features(rng, 3 * 152 * 128 + 1)
        yield c, test, c.surrogate_predict(test)


@pytest.mark.parametrize("n", [1, 2, 127, 128, 129, 255, 256, 257, 152 * 128 - 1, 152 * 128, 152 * 128 + 1,
                               2 * 152 * 128 + 129])
def test_prefix_of_a_prediction(fitted, n):
    c, test, (lp, inside) = fitted
    lp_n, inside_n = c.surrogate_predict(test[:n])
    assert np.all(np.isfinite(lp_n))
    assert np.array_equal(lp_n, lp[:n]) and np.array_equal(inside_n, inside[:n])


@pytest.mark.parametrize("value", [np.nan, np.inf, -np.inf, 1e300, 0.0, 5e-324, 1e-40])
def test_one_bad_row_leaves_the_others(fitted, value):
    c, test, (lp, inside) = fitted
    bad = np.array([0, 77, 127, 128, 255, 700])
    x = test[:1000].copy()
    x[bad] = value
    lp_b, inside_b = c.surrogate_predict(x)
    rest = np.setdiff1d(np.arange(1000), bad)
    assert np.array_equal(lp_b[rest], lp[rest]) and np.array_equal(inside_b[rest], inside[rest])
    assert not inside_b[bad].any()  # densities of zero lie outside the box as well
    if abs(value) < 1.0:  # a finite input has a finite answer, the same in every row and with every tiny value
        one, _ = c.surrogate_predict(np.zeros((1, 30)))
        assert np.all(np.isfinite(one)) and np.array_equal(lp_b[bad], np.repeat(one, len(bad), axis=0))


def test_prediction_follows_new_parameters_and_maps(fitted):
    c, test, (lp, inside) = fitted
    state = c.surrogate_get_state()
    with ptadd.Context(MAT, ptadd.PTADD_FP64, 0) as d:
        d.surrogate_set_state(state)
        lp_d, inside_d = d.surrogate_predict(test[:300])
        assert np.array_equal(lp_d, lp[:300]) and np.array_equal(inside_d, inside[:300])
        p = d.mlp_get_params()
        d.mlp_set_params(0.0 * p)  # zero weights and biases: the mean answer in every row
        lp_0, _ = d.surrogate_predict(test[:300])
        assert np.array_equal(lp_0, np.repeat(lp_0[:1], 300, axis=0)) and not np.array_equal(lp_0, lp_d)
        d.mlp_set_params(p)
        lp_p, _ = d.surrogate_predict(test[:300])
        assert np.array_equal(lp_p, lp_d)
        x = np.random.default_rng(2).normal(size=(64, 30)).astype(np.float32)
        d.mlp_train(x, target_fn(x.astype(np.float64)).astype(np.float32), epochs=2, batch=32)
        trained = d.surrogate_get_state()
        lp_t, _ = d.surrogate_predict(test[:300])
        assert not np.array_equal(lp_t, lp_d)
    with ptadd.Context(MAT, ptadd.PTADD_FP64, 0) as d:
        d.surrogate_set_state(trained)
        assert np.array_equal(d.surrogate_predict(test[:300])[0], lp_t)


@pytest.mark.parametrize("n", [1, 15, 16, 17, 127, 128, 129, 511, 513, 1000])
def test_loss_and_gradient_at_tile_edges(n):
    rng = np.random.default_rng(1000 + n)
    x = rng.normal(size=(n, 30)).astype(np.float32)
    y = target_fn(x.astype(np.float64)).astype(np.float32)
    with ptadd.Context(MAT, ptadd.PTADD_FP64, 0) as c:
        c.mlp_init(seed=7)
        p = c.mlp_get_params().astype(np.float64)
        loss, g = c.mlp_loss_grad(x, y)
    lo, go = O.mlp_loss_grad(DIMS, weights_bf16(p), bf16(x), y.astype(np.float64))
    assert abs(loss / lo - 1) <= 2e-2
    for (Wg, bg), (Wo, bo) in zip(split(g), split(go)):
        assert relfro(Wg, Wo) <= 2e-2
        assert relfro(bg, bo) <= 2e-2


@pytest.mark.parametrize("n,batch", [(16, 16), (130, 64), (304, 304), (1040, 1040), (700, 16)])
def test_training_steps(n, batch):
    """The loss of the first epochs against oracle Adam on the same minibatches; shuffling is
    taken out by one minibatch per epoch where the sizes allow it, else the losses only have to fall."""
    rng = np.random.default_rng(7 * n + batch)
    x = rng.normal(size=(n, 30)).astype(np.float32)
    y = target_fn(x.astype(np.float64)).astype(np.float32)
    with ptadd.Context(MAT, ptadd.PTADD_FP64, 0) as c:
        c.mlp_init(seed=9)
        p = weights_bf16(c.mlp_get_params().astype(np.float64))
        losses = c.mlp_train(x, y, epochs=12, batch=batch, lr=1e-3, seed=1)
    assert np.all(np.isfinite(losses)) and losses[-1] < losses[0]
    if batch >= n:
        m, v, ora = np.zeros_like(p), np.zeros_like(p), []
        for t in range(1, 13):
            lo, go = O.mlp_loss_grad(DIMS, p, bf16(x), y.astype(np.float64))
            ora.append(lo)
            O.adam_step(p, go, m, v, t, lr=1e-3)
        assert np.max(np.abs(losses - np.array(ora)) / np.array(ora)) <= 3e-2
