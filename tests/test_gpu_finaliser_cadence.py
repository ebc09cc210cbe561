"""Energies recorded at a cadence: most steps' finalisers only advance the level, and the one after
may have to reduce, so the branch changes from step to step.  At a level that both record, the
energy is that of the run that records every level, bit for bit (the same sums of the same fields),
and so is the state; every CTA size that the finalisers run in, real and complex fields."""
import numpy as np
import pytest

from paper_1501_04552_gb300 import inputs as I

pytestmark = pytest.mark.gpu

L = 32.0


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


@pytest.mark.parametrize("cplx", [False, True])
@pytest.mark.parametrize("prec", ["df64", "mixed", "fp64"])
@pytest.mark.parametrize("N", [16, 32, 64, 128, 256])
def test_cadences_agree(kg, N, prec, cplx):
    u = I.gaussian(N, L, 0.3, 2.0)
    got = {}
    for every in (1, 2, 3):
        kg.kg_set_options(precision=prec, energy_every=every)
        if cplx:
            kg.kg_init_complex(N, L, 0.01, u * np.exp(0.5j))
        else:
            kg.kg_init(N, L, 0.01, u)
        out = []
        for _ in range(4):
            kg.kg_step(6)
            out.append(kg.kg_energy())
        got[every] = (out, kg.kg_status(), kg.kg_fetch_spectral(N))
    for every in (2, 3):
        assert got[every][:2] == got[1][:2]
        for a, b in zip(got[every][2], got[1][2]):
            assert np.array_equal(a, b)
    kg.kg_set_options()
