"""kg_step returns once its steps are enqueued: the driver's queue holds about a thousand launches,
so long calls go out as graphs of 32 steps after the first few hundred launches.  A long call must be
bit for bit the same steps as single calls (energies recorded, a blow-up between, every form of a
step), come back long before the GPU is done, and be only launches on a stream that is being captured."""
import time

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
    K.kg_set_stream(None)
    K.kg_set_scheme()
    K.kg_set_options()


def result(kg, N, cplx):
    return kg.kg_status(), kg.kg_energy(), (kg.kg_fetch_complex if cplx else kg.kg_fetch)(N)


# two, four and six launches a step, three passes a step (composed); calls that end inside a graph's worth
@pytest.mark.parametrize("N,prec,scheme,cplx,steps", [(16, "df64", "eq2", False, 450), (32, "mixed", "eq2", False, 233),
                                                      (16, "fp64", "eq2", False, 200), (16, "df64", "composed4", False, 140),
                                                      (32, "fp64", "composed4", False, 60), (16, "df64", "eq2", True, 230),
                                                      (64, "df64", "eq2", False, 450)])
@pytest.mark.parametrize("amplitude", [0.3, 4.0])
def test_long_calls_are_the_single_steps(kg, N, prec, scheme, cplx, steps, amplitude):
    u = I.gaussian(N, L, amplitude, 4.0)
    got = []
    for calls in ([steps], [1] * steps):
        kg.kg_set_options(precision=prec, energy_every=0 if scheme == "composed4" else 7,
                          blowup_threshold=50.0)
        kg.kg_set_scheme(scheme)
        if cplx:
            kg.kg_init_complex(N, L, 0.01, u * np.exp(0.5j))
        else:
            kg.kg_init(N, L, 0.01, u)
        for n in calls:
            kg.kg_step(n)
            if n == 1:
                kg.kg_status()        # waits for the GPU: no single step is ever in a graph
        got.append(result(kg, N, cplx))
    a, b = got
    assert a[0] == b[0] and a[1] == b[1] and np.array_equal(a[2], b[2])
    assert a[0]["frozen"] == (amplitude > 1.0)
    kg.kg_set_scheme()
    kg.kg_set_options()


def test_a_long_call_comes_back_early(kg):
    import torch
    kg.kg_set_options(precision="df64")
    kg.kg_init(128, L, 0.002, I.gaussian(128, L, 0.1, 1.5))
    kg.kg_step(300)                   # kernels loaded
    kg.kg_status()
    t0 = time.perf_counter()
    kg.kg_step(1000)
    t1 = time.perf_counter()
    torch.cuda.synchronize()
    t2 = time.perf_counter()
    # by launches alone three quarters of the steps have run when the call returns
    assert t1 - t0 < 0.25 * (t2 - t0), (t1 - t0, t2 - t0)


def test_a_captured_stream_takes_launches(kg):
    import torch
    N = 32
    u = I.gaussian(N, L, 0.3, 2.0)
    s = torch.cuda.Stream()
    kg.kg_set_options(precision="mixed")
    kg.kg_set_stream(s.cuda_stream)
    kg.kg_init(N, L, 0.01, u)
    kg.kg_step(400)                   # the queue counts as full from here on
    s.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        kg.kg_step(20)
    with torch.cuda.stream(s):
        g.replay()
        g.replay()
    a = result(kg, N, False)
    kg.kg_init(N, L, 0.01, u)
    kg.kg_step(440)
    b = result(kg, N, False)
    del g
    kg.kg_set_stream(None)
    assert a[0] == b[0] and a[1] == b[1] and np.array_equal(a[2], b[2])
    kg.kg_set_options()
