"""Gradients of batches with more tiles than partial gradients (128, of 128 rows each), several a CTA, against
the FP64 network with the same rounding points, ragged and whole.

Tolerance: the tensor cores' FP32 accumulation drops up to 2^-23 of the sum at each of a tile's eight
products (1e-6); between the tiles of a part and the 128 parts sums are rounded, 15 + 127 times at most, like
the square root: 0.7e-6.  2e-6 of the gradient's norm holds both, and the few units of 1e-7 that the
batch's rounding to bfloat16 on opposite sides of a tie adds."""
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
    yield K
    K.kg_mlp_finalize()


@pytest.mark.parametrize("rows", [8192, 8193, 16384 + 100, 65536, 262144 - 1])
def test_gradient_of_many_tiles(kg, rows):
    rng = np.random.default_rng(1)
    params = (rng.standard_normal(kg.kg_mlp_param_count()) * 0.1).astype(np.float32)
    X = rng.standard_normal((rows, 6)).astype(np.float32)
    y = (rng.random(rows) < 0.4).astype(np.float32)
    ell = rng.standard_normal(rows).astype(np.float32)
    kg.kg_mlp_set_params(params)
    loss, grad = kg.kg_mlp_grad(X, y, ell, 10.0)
    rloss, rgrad = M.loss_and_grads(M.unflatten(params.astype(np.float64)), X.astype(np.float64), y, ell, 10.0, True)
    rgrad = M.flatten(rgrad)
    err = np.linalg.norm(grad - rgrad) / np.linalg.norm(rgrad)
    print("rows %d: gradient %.2e, loss %.2e" % (rows, err, abs(loss - rloss) / rloss))
    assert err <= 2e-6
    assert abs(loss - rloss) <= 2e-6 * rloss
