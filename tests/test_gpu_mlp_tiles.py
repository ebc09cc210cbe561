"""Ranker kernels at the edges of their tiles (128 rows, at most 64 partial gradients, so from 8193
rows on a CTA takes several tiles): predictions row by row must not depend on how many rows a call
has, and the gradient and loss of n rows must be the mean of those of its parts.

Tolerances: a row's forward pass is the same arithmetic wherever it sits (bitwise).  Gradients are
FP32 sums of n bf16 products, rounded per operand the same way in every split except dz, which is
scaled by 1/n before it is rounded to bf16: with n and the parts' sizes powers of two times the same
odd number that scaling is exact, and what differs is the order of FP32 sums, bounded by
n * 2^-24 relative to the sum of magnitudes; 1e-4 covers n = 16384 with cancellation."""
import numpy as np
import pytest

from oracle import mlp_oracle as M

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def kg():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__ as g
    g.build_library()
    from paper_1501_04552_gb300 import kg as K
    p = M.init_params(11)
    rng = np.random.default_rng(12)
    for k in ("b1", "b2", "b3"):
        p[k] = rng.normal(0.0, 0.05, size=M.SHAPES[k])
    K.kg_mlp_set_params(M.flatten(p).astype(np.float32))
    yield K
    K.kg_mlp_finalize()


def data(n):
    rng = np.random.default_rng(n)
    return (rng.standard_normal((n, M.D_IN)).astype(np.float32), (rng.uniform(size=n) < 0.4).astype(np.float32),
            rng.uniform(-0.5, 2.0, size=n).astype(np.float32))


@pytest.mark.parametrize("n", [1, 127, 128, 129, 8193, 19456, 19585, 40000])
def test_predictions_do_not_depend_on_the_call(kg, n):
    X, _, _ = data(n)
    p, t = kg.kg_mlp_predict(X)
    cut = max(1, n // 3)
    q = [kg.kg_mlp_predict(X[:cut])] + ([kg.kg_mlp_predict(X[cut:])] if cut < n else [])
    assert np.array_equal(p, np.concatenate([a for a, _ in q]))
    assert np.array_equal(t, np.concatenate([b for _, b in q]))


@pytest.mark.parametrize("n", [2, 256, 8192, 16384, 16380])
def test_gradient_of_a_batch_is_the_mean_of_its_halves(kg, n):
    X, y, l = data(n)
    loss, g = kg.kg_mlp_grad(X, y, l)
    h = n // 2
    la, ga = kg.kg_mlp_grad(X[:h], y[:h], l[:h])
    lb, gb = kg.kg_mlp_grad(X[h:], y[h:], l[h:])
    assert abs(loss - 0.5 * (la + lb)) <= 1e-5 * abs(loss)
    ref = 0.5 * (ga.astype(np.float64) + gb)
    assert np.linalg.norm(g - ref) <= 1e-4 * np.linalg.norm(ref)


@pytest.mark.parametrize("batch", [1, 128, 100, 5000])
def test_training_repeats_itself(kg, batch):
    """partial gradients are summed in order: two runs from the same parameters are the same run"""
    X, y, l = data(5000)
    start = kg.kg_mlp_get_params()
    out = []
    for _ in range(2):
        kg.kg_mlp_set_params(start)
        loss = kg.kg_mlp_train(X[:500] if batch == 1 else X, y[:500] if batch == 1 else y, l[:500] if batch == 1 else l,
                               epochs=3, batch=batch, lr=1e-3, T=10.0, seed=5)
        out.append((loss, kg.kg_mlp_get_params()))
    kg.kg_mlp_set_params(start)
    assert out[0][0] == out[1][0] and np.array_equal(out[0][1], out[1][1])
