"""The spectral arrays' internal layouts (x-lines with padded rows, tiled z-columns) seen from
outside: the spectrum handed out by kg_fetch_spectral is numpy's transform in the packed order
[kz][ky][kx], a checkpoint's payload is that same data, and a checkpoint loaded and saved again
is byte for byte the first one -- on grids whose last column tile holds one mode and seven slots
of padding, and on a full tile per row (complex fields).

Tolerance: set-up transforms run in double-float (48-bit significand) or FP64; a transform of
N^3 points accumulates about log2(N^3) roundings of 2^-48 relative to the norm, under 21 * 3.6e-15
= 8e-14 at N = 128."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

L = 32.0
TOL = 8e-14


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


def rel(a, b):
    return float(np.linalg.norm((a - b).ravel()) / np.linalg.norm(b.ravel()))


@pytest.mark.parametrize("N", [16, 32, 64, 128])
@pytest.mark.parametrize("prec", ["df64", "mixed", "fp64"])
@pytest.mark.parametrize("cplx", [False, True])
def test_packed_spectrum_and_checkpoint(kg, N, prec, cplx):
    rng = np.random.default_rng(N)
    u = rng.standard_normal((N, N, N))
    if cplx:
        u = u + 1j * rng.standard_normal((N, N, N))
    kg.kg_set_options(precision=prec)
    (kg.kg_init_complex if cplx else kg.kg_init)(N, L, 0.001, u)
    a, b = kg.kg_fetch_spectral(N)
    assert rel(a, np.fft.fftn(u) if cplx else np.fft.rfftn(u)) <= TOL
    buf = kg.kg_save_state()
    payload = buf[kg.STATE_HEADER_BYTES:].view(np.complex128).reshape((2,) + a.shape)
    assert np.array_equal(payload[0], a) and np.array_equal(payload[1], b)
    kg.kg_step(3)
    kg.kg_load_state(buf)
    assert np.array_equal(kg.kg_save_state(), buf)
    back = kg.kg_fetch_complex(N) if cplx else kg.kg_fetch(N)
    assert rel(back, u) <= TOL


def test_512_double_float_tiles(kg):
    """512^3 double-float contexts tile their z-columns by four: the energy from the FP64 state
    (k_energy_q and the FP64 inverse transforms, told of that layout) must be the recorded one
    (sums of 6.7e7 terms of a field good to 1e-13: 1e-12), and a checkpoint must survive a load"""
    import torch
    N, dt = 512, 0.005
    x = -L / 2 + (L / N) * torch.arange(N, dtype=torch.float64, device="cuda")
    g = torch.exp(-(x / 1.5) ** 2)
    u = 0.4 * g[:, None, None] * torch.exp(-((x - 1.0) / 2.0) ** 2)[None, :, None] * (g * torch.cos(3 * x))[None, None, :]
    u = u.contiguous()
    torch.cuda.synchronize()
    e = {}
    for every in (0, 4):
        kg.kg_set_options(precision="df64", energy_every=every)
        kg.kg_init_device(N, L, dt, u)
        kg.kg_step(4)
        e[every] = kg.kg_energy()
    assert abs(e[0] - e[4]) <= 1e-12 * abs(e[4])
    buf = kg.kg_save_state()
    kg.kg_step(1)
    a = kg.kg_fetch(N)
    kg.kg_load_state(buf)
    assert np.array_equal(kg.kg_save_state(), buf)
    kg.kg_step(1)
    assert np.array_equal(kg.kg_fetch(N), a)
    kg.kg_finalize()
    kg.kg_set_options()
