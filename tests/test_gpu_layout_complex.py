"""Complex 512^3 double-float contexts tile their z-columns by four, in full tiles: the energy from the
FP64 state (k_energy_q and the FP64 inverse transforms, told of that layout) must be the recorded one
(sums of 1.3e8 terms of a field good to 1e-13: 1e-12), and a checkpoint must survive a load."""
import numpy as np
import pytest

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


def test_512_complex_double_float_tiles(kg):
    N, dt = 512, 0.005
    x = -L / 2 + (L / N) * np.arange(N)
    g = np.exp(-(x / 1.5) ** 2)
    u = 0.4 * g[:, None, None] * np.exp(-((x - 1.0) / 2.0) ** 2)[None, :, None] * (g * np.exp(3j * x))[None, None, :]
    e = {}
    for every in (0, 4):
        kg.kg_set_options(precision="df64", energy_every=every)
        kg.kg_init_complex(N, L, dt, u)
        kg.kg_step(4)
        e[every] = kg.kg_energy()
    assert abs(e[0] - e[4]) <= 1e-12 * abs(e[4])
    buf = kg.kg_save_state()
    kg.kg_step(1)
    a = kg.kg_fetch_complex(N)
    kg.kg_load_state(buf)
    assert np.array_equal(kg.kg_save_state(), buf)
    kg.kg_step(1)
    assert np.array_equal(kg.kg_fetch_complex(N), a)
    kg.kg_finalize()
    kg.kg_set_options()
