"""The FP64 transforms with twiddles and rotations fused into FMAs, against numpy's FFT: every
stage plan the grids have (transform lengths 8 to 512: radix-8 stages with a last radix 2, 4 or
none), forward (kg_fetch_spectral) and inverse (kg_fetch), on noise.  log2(N^3) <= 27 levels of sums
with a few roundings of 2^-53 each, growing like the square root in L2: 1e-15 * 27 bounds it.
Power-of-two scalings by the exponent field must treat zeros and subnormals as products do."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

L = 32.0
TOL = 27e-15


@pytest.fixture(scope="module")
def kg():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__ as g
    g.build_library()
    from paper_1501_04552_gb300 import kg as K
    yield K
    K.kg_finalize()
    K.kg_set_options()


def rel(a, b):
    return float(np.linalg.norm((a - b).ravel()) / np.linalg.norm(b.ravel()))


@pytest.mark.parametrize("N", [16, 32, 64, 128, 256])
@pytest.mark.parametrize("cplx", [False, True])
def test_transforms(kg, N, cplx):
    rng = np.random.default_rng(N)
    u = rng.standard_normal((N, N, N))
    if cplx:
        u = u + 1j * rng.standard_normal((N, N, N))
    kg.kg_set_options(precision="fp64", nonlinearity=0.0)
    (kg.kg_init_complex if cplx else kg.kg_init)(N, L, 1e-3, u)
    a, _ = kg.kg_fetch_spectral(N)
    assert rel(a, np.fft.fftn(u) if cplx else np.fft.rfftn(u)) <= TOL
    assert rel(kg.kg_fetch_complex(N) if cplx else kg.kg_fetch(N), u) <= 2 * TOL


@pytest.mark.parametrize("size", [0.0, 1e-320, 1e-310, 1e-300])
def test_scales(kg, size):
    """a constant field of any size: the linear step keeps it constant, max |u| is its size"""
    N = 32
    u = np.full((N, N, N), size)
    kg.kg_set_options(precision="fp64", nonlinearity=0.0)
    kg.kg_init(N, L, 1e-3, u)
    kg.kg_step(1)
    m = kg.kg_status()["maxabs"]
    assert abs(m - size) <= 1e-14 * size + 5e-324 * N ** 3   # sums of subnormals round to their spacing
    assert np.isfinite(kg.kg_fetch(N)).all()
    kg.kg_set_options()
