"""Small real grids in double-float step with the y, x and y passes of a z-plane in one kernel.
Against IEEE FP64, which takes the separate passes, on every grid that has the form (one CTA a
plane with and without idle row blocks, two CTAs a plane), both schemes, with calls between the steps that use the
work arrays or change the order of the passes (read-out, energy, timed steps, a checkpoint); these
must leave the steps as they are, bit for bit.  Then the blow-up check, which the z pass makes.

Tolerance: the double-float transforms and state carry 2^-46 or better per operation, and a short
run amplifies that by less than 1e3: 1e-11 of max |u|, the bound used for double-float elsewhere."""
import numpy as np
import pytest

from paper_1501_04552_gb300 import inputs as I

pytestmark = pytest.mark.gpu

L, DT = 32.0, 0.02


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
    K.kg_set_scheme()
    K.kg_set_options()


def start(kg, prec, scheme, N, **opt):
    rng = np.random.default_rng(N)
    x = rng.standard_normal((N, N, N))
    kg.kg_set_options(precision=prec, **opt)
    kg.kg_set_scheme(scheme)
    kg.kg_init(N, L, DT, I.gaussian(N, L, 0.8, 3.0) + 0.01 * x, 0.05 * np.roll(x, 3, 1))


@pytest.mark.parametrize("scheme", ["eq2", "composed4"])
@pytest.mark.parametrize("N", [16, 32, 64])
def test_steps_and_what_comes_between(kg, N, scheme):
    start(kg, "df64", scheme, N)
    kg.kg_step(12)
    u = kg.kg_fetch(N)
    start(kg, "fp64", scheme, N)
    kg.kg_step(12)
    ref = kg.kg_fetch(N)
    e_ref = kg.kg_energy()
    assert np.abs(u - ref).max() <= 1e-11 * np.abs(ref).max()

    start(kg, "df64", scheme, N)
    kg.kg_energy()
    kg.kg_step(2)
    kg.kg_fetch(N)
    kg.kg_step(1)
    kg.kg_energy()
    kg.kg_fetch(N)
    kg.kg_step_timed(2)
    blob = kg.kg_save_state()
    kg.kg_step(3)
    kg.kg_load_state(blob)
    kg.kg_step_timed(1)
    kg.kg_step(6)
    assert np.array_equal(kg.kg_fetch(N), u)
    assert abs(kg.kg_energy() - e_ref) <= 1e-11 * abs(e_ref)


@pytest.mark.parametrize("ahead", [False, True])
@pytest.mark.parametrize("N", [16, 32, 64])
def test_blow_up_stops_the_update(kg, N, ahead):
    got = {}
    for prec in ("df64", "fp64"):
        kg.kg_set_options(precision=prec, blowup_threshold=50.0)
        kg.kg_set_scheme()
        kg.kg_init(N, L, DT, I.gaussian(N, L, 4.0, 4.0), None)
        for _ in range(40):
            kg.kg_step(5)
            if ahead:
                kg.kg_energy()
        st = kg.kg_status()
        got[prec] = (st["frozen"], st["blowup_level"], st["level"], kg.kg_fetch(N))
    a, b = got["df64"], got["fp64"]
    assert a[:3] == b[:3] and a[0]
    assert np.abs(a[3] - b[3]).max() <= 1e-9 * np.abs(b[3]).max()   # a field about to blow up
