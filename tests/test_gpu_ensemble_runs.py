"""The ensemble's unit list at its edges: one instance, one grid size only, lists shorter and much
longer than the resident CTAs (runs of one and of several units, the last of a pass cut short), one
step, and more steps than one launch takes.  Every instance must follow the single-instance path,
whose arithmetic is the same (double-float: 1e-13, the bound of the ensemble's other tests)."""
import numpy as np
import pytest

from paper_1501_04552_gb300 import inputs as I

pytestmark = pytest.mark.gpu

L, DT = 32.0, 0.005


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


@pytest.mark.parametrize("n64,n128,steps", [(1, 0, 1), (0, 1, 3), (5, 1, 53), (1, 5, 7), (97, 0, 4), (67, 9, 101)])
@pytest.mark.parametrize("bps", [1, 4])
def test_instances_follow_the_single_path(kg, n64, n128, steps, bps):
    rng = np.random.default_rng(n64 + 10 * n128)
    Ns = np.array([64] * n64 + [128] * n128, dtype=np.int32)
    rng.shuffle(Ns)
    A, s = rng.uniform(0.5, 1.5, Ns.size), rng.uniform(0.7, 2.0, Ns.size)
    kg.kg_set_options(precision="df64")
    kg.kg_ens_init(Ns, L, DT, A, s)
    kg.kg_ens_set_schedule(0, bps, bps % 2)
    done, _ = kg.kg_ens_run(steps, 1e3)
    r = kg.kg_ens_results()
    assert done == steps and (r["level"] == steps).all() and not r["frozen"].any()
    for i in sorted({0, Ns.size // 2, Ns.size - 1}):
        N = int(Ns[i])
        u = kg.kg_ens_fetch(i)
        kg.kg_init(N, L, DT, I.gaussian(N, L, A[i], s[i]), None)
        kg.kg_step(steps)
        v = kg.kg_fetch(N)
        assert np.linalg.norm(u - v) <= 1e-13 * np.linalg.norm(v), i
        assert abs(r["maxabs"][i] - kg.kg_status()["maxabs"]) <= 2.0 ** -23 * r["maxabs"][i]
    kg.kg_ens_finalize()


def test_flags_within_one_launch(kg):
    """instances that blow up at different levels of the same launch, among others that do not"""
    n = 40
    A, s = np.linspace(3.0, 4.0, n), np.full(n, 1.5)
    Ns = np.full(n, 64, dtype=np.int32)
    kg.kg_set_options(precision="df64", blowup_threshold=20.0)
    kg.kg_ens_init(Ns, L, DT, A, s)
    kg.kg_ens_run(150, 20.0)
    r = kg.kg_ens_results()
    kg.kg_ens_finalize()
    assert 0 < r["frozen"].sum() and len(set(r["blowup_level"][r["frozen"]])) > 3
    for i in (0, n // 3, n - 1):
        kg.kg_init(64, L, DT, I.gaussian(64, L, A[i], s[i]), None)
        kg.kg_step(150)
        st = kg.kg_status()
        assert st["frozen"] == bool(r["frozen"][i]) and st["level"] == r["level"][i]
        assert st["blowup_level"] == r["blowup_level"][i]
    kg.kg_set_options()
