"""Options that change between kg_energy, which runs the next step's x pass ahead, and the step that
follows: on small double-float grids (k_plane, finalisers in the z pass) the levels, flags and energies
must be those of the IEEE FP64 path, whose passes are separate.

Tolerance: 1e-11 of the energy and of max |u|, as between these paths elsewhere; the steps are few."""
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
    K.kg_set_options()


def run(kg, prec, N, amplitude, script):
    """script: options (a dict), steps (a number) or "e" (kg_energy) in order"""
    kg.kg_set_options(precision=prec)
    kg.kg_init(N, L, DT, I.gaussian(N, L, amplitude, 4.0))
    flags, energies = [], []
    for s in script:
        if s == "e":
            energies.append(kg.kg_energy())
        elif isinstance(s, dict):
            kg.kg_set_options(precision=prec, **s)
        else:
            kg.kg_step(s)
            st = kg.kg_status()
            flags.append((st["level"], st["frozen"], st["blowup_level"], st["maxabs"]))
    return flags, energies, kg.kg_fetch(N)


on, off = dict(blowup_threshold=2.0), dict()
SCRIPTS = {
    # the cadence changes while the x pass of the next step has run
    "cadence": (0.8, [3, "e", dict(energy_every=1), 1, "e", 2, "e", dict(energy_every=3), 3, "e", off, 1, "e", 2, "e"]),
    # a threshold that the field exceeds comes while the x pass has run without it: the next level freezes
    "threshold on": (4.0, [2, "e", on, 1, "e", 2, "e"]),
    "threshold on, no energy": (4.0, [2, on, 1, "e", 2, "e"]),
    # ... and goes again before it was ever looked at
    "threshold off": (4.0, [2, "e", on, off, 1, "e", 2, "e"]),
    # the x pass run ahead has frozen the state: taking the threshold away does not thaw it
    "frozen ahead": (4.0, [2, on, "e", off, 1, "e", 2, "e"]),
}


@pytest.mark.parametrize("N", [16, 32, 64])
@pytest.mark.parametrize("case", sorted(SCRIPTS))
def test_options_between_energy_and_step(kg, N, case):
    amplitude, script = SCRIPTS[case]
    flags, energies, u = run(kg, "df64", N, amplitude, script)
    rflags, renergies, ref = run(kg, "fp64", N, amplitude, script)
    assert [f[:3] for f in flags] == [f[:3] for f in rflags]
    for f, r in zip(flags, rflags):
        assert abs(f[3] - r[3]) <= 2.0 ** -23 * r[3]      # the double-float passes keep max |u| as a float
    for e, r in zip(energies, renergies):
        assert abs(e - r) <= 1e-11 * abs(r)
    assert np.abs(u - ref).max() <= 1e-11 * np.abs(ref).max()
    assert any(f[1] for f in flags) == (case in ("threshold on", "threshold on, no energy", "frozen ahead"))
