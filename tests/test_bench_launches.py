"""The launch count of a bench line, for every form of a step."""
import importlib.util
import os

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_launches_of_the_timed_region():
    spec = importlib.util.spec_from_file_location("bench_under_test", os.path.join(ROOT, "bench.py"))
    bench = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(bench)
    plain = [(5, True), (10, True), (5, False)]                # 20 steps, two energies
    assert bench.timed_launches("df64", 512, plain) == 82
    assert bench.timed_launches("mixed", 64, [(20, False)]) == 80
    assert bench.timed_launches("fp64", 512, plain) == 122     # six kernels a step
    assert bench.timed_launches("fp64", 32, plain) == 122
    assert bench.timed_launches("df64", 64, plain) == 40       # two; the finaliser rides in them
    assert bench.timed_launches("df64", 128, plain) == 82
    assert bench.timed_launches("mixed", 512, plain, xy_fusion=True) == 87   # an inverse y pass per call
    assert bench.timed_launches("df64", 512, plain, xy_fusion=True) == 82    # built for FP32 only
