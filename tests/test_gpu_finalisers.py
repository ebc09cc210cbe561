"""The finalisers that ride in the y passes (one more CTA of 16 to 1024 threads, by grid): on
every grid size the level, the blow-up level, max |u| and the recorded energies must be the
oracle's, with the energy recorded at every level, and a frozen state must stay as it is when the
energy is asked for and more steps are taken.

Tolerances: max |u| is kept as a float by the double-float and FP32 passes (2^-23 relative, half
an ulp either way, and FP32 transforms 1e-5 as elsewhere in these tests); the energies are sums of
N^3 non-negative terms, compensated, of fields good to 1e-13 (double-float, FP64)."""
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


@pytest.mark.parametrize("N", [16, 32, 64, 128])
@pytest.mark.parametrize("prec", ["df64", "mixed", "fp64"])
def test_energy_and_max_at_every_level(kg, N, prec):
    from oracle import oracle as O
    dt = 0.02
    u0 = I.gaussian(N, L, 0.8, 3.0)
    kg.kg_set_options(precision=prec, energy_every=1)
    kg.kg_init(N, L, dt, u0, None)
    ref = O.Solver(N, L, dt, u0, None)
    etol, mtol = (1e-12, 2.0 ** -23) if prec != "mixed" else (1e-6, 1e-5)
    for n in range(1, 6):
        kg.kg_step(1)
        ref.step(1)
        e = ref.energy()
        assert abs(kg.kg_energy() - e) <= etol * abs(e), n
        st = kg.kg_status()
        assert st["level"] == n and not st["frozen"]
        assert abs(st["maxabs"] - ref.last_maxabs) <= mtol * ref.last_maxabs, n
    ref.close()
    kg.kg_set_options()


@pytest.mark.parametrize("N", [16, 64])
@pytest.mark.parametrize("prec", ["df64", "mixed", "fp64"])
def test_frozen_state_is_left_alone(kg, N, prec):
    from oracle import oracle as O
    dt, thr = 0.02, 50.0
    u0 = I.gaussian(N, L, 4.0, 4.0)
    kg.kg_set_options(precision=prec, energy_every=1, blowup_threshold=thr)
    kg.kg_init(N, L, dt, u0, None)
    ref = O.Solver(N, L, dt, u0, None)
    blown, level = ref.step(60, threshold=thr)
    ref.close()
    kg.kg_step(60)
    st = kg.kg_status()
    assert blown and st["frozen"] and st["blowup_level"] == level == st["level"]
    a, b = kg.kg_fetch_spectral(N)
    e = kg.kg_energy()
    kg.kg_step(3)
    assert kg.kg_energy() == e
    kg.kg_step(2)
    assert kg.kg_status() == st
    a1, b1 = kg.kg_fetch_spectral(N)
    assert np.array_equal(a, a1) and np.array_equal(b, b1)
    kg.kg_set_options()
