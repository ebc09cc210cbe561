"""The ranker network's calls keep device memory between them up to 2^20 rows; a call that fails
half-way through growing it must leave no more than that behind: the memory of a batch of 2^21
rows goes back when any of its allocations fails, and the next call works."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

ROWS = 1 << 21


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


@pytest.mark.parametrize("call,allocation", [("predict", 1), ("predict", 2), ("predict", 3), ("grad", 3),
                                             ("train", 4), ("train", 5), ("train", 6), ("train", 7)])
def test_a_failed_call_gives_its_memory_back(kg, monkeypatch, call, allocation):
    import torch
    rng = np.random.default_rng(0)
    X = rng.standard_normal((ROWS, 6)).astype(np.float32)
    y, l = np.zeros(ROWS, np.float32), np.zeros(ROWS, np.float32)
    calls = {"predict": lambda n: kg.kg_mlp_predict(X[:n]), "grad": lambda n: kg.kg_mlp_grad(X[:n], y[:n], l[:n]),
             "train": lambda n: kg.kg_mlp_train(X[:n], y[:n], l[:n], epochs=1, batch=n)}
    kg.kg_mlp_finalize()
    kg.kg_mlp_set_params(np.linspace(-0.2, 0.2, kg.kg_mlp_param_count()))
    calls["train"](256)                       # kernels loaded, small staging kept
    calls[call](ROWS)                         # beyond what is kept: released when it is done
    before = torch.cuda.mem_get_info()[0]
    monkeypatch.setenv("KG_TEST_FAIL_STAGING", str(allocation))
    with pytest.raises(kg.KgError):
        calls[call](ROWS)
    monkeypatch.delenv("KG_TEST_FAIL_STAGING")
    # the smallest allocation of such a call is 8 MiB; the small staging that it replaced is 2 MiB at most
    assert before - torch.cuda.mem_get_info()[0] < 4 << 20
    calls[call](300)
