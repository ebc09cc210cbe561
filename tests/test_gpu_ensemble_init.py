"""The ensemble's set-up from products of 1D transforms: the field of level 0 read back against the
Gaussian itself, and the first level against the single-instance solver, whose set-up transforms the
field in 3D -- for widths from one grid cell to far beyond the box (where the field does not decay
at the boundary), amplitudes of either sign and zero, both grids, every precision, with and without
the nonlinearity.

Tolerances: level 0 is an FP64 read-out of FP64 products of compensated sums, 1e-13 in L2 (21
roundings of a transform at 2^-53 and a few of the products, times a safety of 20); level 1 adds the
single solver's double-float set-up, itself good to 5e-14: 1e-13; FP32 transforms 1e-9 as in the
ensemble's other tests."""
import numpy as np
import pytest

from paper_1501_04552_gb300 import inputs as I

pytestmark = pytest.mark.gpu

L, DT = 32.0, 0.005
CASES = [(64, 1.0, 0.5), (64, -0.8, 2.0), (128, 0.9, 0.25), (128, 0.7, 1.3), (64, 0.0, 1.0), (128, -0.4, 40.0), (64, 0.3, 9.0)]


@pytest.fixture(scope="module")
def kg():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__ as g
    g.build_library()
    from paper_1501_04552_gb300 import kg as K
    yield K
    K.kg_ens_finalize()
    K.kg_finalize()
    K.kg_set_options()


def close(a, b, tol):
    return np.linalg.norm(a - b) <= tol * max(np.linalg.norm(b), 1e-300)


@pytest.mark.parametrize("prec", ["df64", "mixed", "fp64"])
@pytest.mark.parametrize("lam", [1.0, 0.0, -2.5])
def test_levels_zero_and_one(kg, prec, lam):
    Ns, A, s = (np.array(c) for c in zip(*CASES))
    kg.kg_set_options(precision=prec, nonlinearity=lam)
    kg.kg_ens_init(Ns.astype(np.int32), L, DT, A, s)
    for i, (N, a, w) in enumerate(CASES):
        assert close(kg.kg_ens_fetch(i), I.gaussian(N, L, a, w), 1e-13), i
    kg.kg_ens_run(1)
    first = [kg.kg_ens_fetch(i) for i in range(len(CASES))]
    kg.kg_ens_finalize()
    for i, (N, a, w) in enumerate(CASES):
        kg.kg_init(N, L, DT, I.gaussian(N, L, a, w), None)
        kg.kg_step(1)
        assert close(first[i], kg.kg_fetch(N), 1e-9 if prec == "mixed" else 1e-13), i
    kg.kg_set_options()
