"""The device passes of the spectral diagnostics against the FP64 oracle and against the
tensor operations that other tensors take (the same function on the CPU)."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lbm():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2608_13437_gb300 import build, lbm as L
    build.build()
    L.lib()
    return L


# odd, even and unit sides; more modes than one wave of blocks; rows of one mode
@pytest.mark.parametrize("shape", [(1, 1, 1), (2, 2, 2), (3, 5, 7), (4, 6, 9), (9, 4, 2), (16, 16, 16),
                                   (33, 20, 31), (5, 1, 64), (72, 70, 66)])
@pytest.mark.parametrize("sutherland", [0, 1])
def test_device_passes_match_oracle_and_tensor_path(lbm, shape, sutherland):
    """Tolerance: 1e-12 of the largest value (FP64 transforms and sums, a few hundred ulp)."""
    import torch
    from oracle import spectral as ospec
    from paper_2608_13437_gb300 import spectral
    rng = np.random.default_rng(sum(shape))
    prim = np.abs(rng.standard_normal((6,) + shape)) + 0.2
    prim[1:4] = rng.standard_normal((3,) + shape)
    L_box, mu, T_ref, rho = 2 * math.pi * 1.3, 2e-3, 0.7, 1.1
    dev = torch.from_numpy(prim).cuda()
    es, ed = spectral.dissipation(dev, mu, T_ref, sutherland, rho, L_box)
    for ref in (spectral.dissipation(torch.from_numpy(prim), mu, T_ref, sutherland, rho, L_box),
                ospec.dissipation(prim[1:4], prim[4], mu, T_ref, sutherland, rho, L_box)):
        scale = max(abs(ref[0]), abs(ref[1]), 1e-300)
        assert abs(es - ref[0]) <= 1e-12 * scale and abs(ed - ref[1]) <= 1e-12 * scale
    k, e = spectral.energy_spectrum(dev[1:4], L_box)
    kc, ec = spectral.energy_spectrum(torch.from_numpy(prim)[1:4], L_box)
    assert torch.equal(k.cpu(), kc) and e.dtype == ec.dtype and e.device == dev.device
    assert float((e.cpu() - ec).abs().max()) <= 1e-12 * float(ec.max())
    # a strided view takes the same passes
    strided = torch.empty((12,) + shape, dtype=torch.float64, device="cuda")[::2]
    strided.copy_(dev)
    assert spectral.dissipation(strided, mu, T_ref, sutherland, rho, L_box) == pytest.approx((es, ed), rel=1e-12)


def test_tensors_under_autograd_take_tensor_operations(lbm):
    """E(k) of a velocity that requires a gradient stays differentiable."""
    import torch
    from paper_2608_13437_gb300 import spectral
    u = torch.randn(3, 6, 6, 6, dtype=torch.float64, device="cuda", requires_grad=True)
    _, e = spectral.energy_spectrum(u)
    e.sum().backward()
    assert torch.allclose(u.grad, u.detach() / 216, rtol=1e-9, atol=1e-12)


@pytest.mark.parametrize("sutherland", [0, 1])
def test_a_view_that_negates_takes_its_values(lbm, sutherland):
    """PyTorch may hand over a tensor whose stored values are the negative ones (a view with the
    negative bit): the result is that of the tensor itself (1e-12, as above)."""
    import torch
    from paper_2608_13437_gb300 import spectral
    g = torch.Generator(device="cuda").manual_seed(3)
    prim = torch.rand(6, 9, 10, 12, dtype=torch.float64, device="cuda", generator=g) + 0.5
    view = torch._neg_view(-prim)
    assert view.is_neg() and torch.equal(view, prim)
    want = spectral.dissipation(prim, 2e-3, 0.7, sutherland, 1.1)
    assert spectral.dissipation(view, 2e-3, 0.7, sutherland, 1.1) == pytest.approx(want, rel=1e-12)
    assert torch.allclose(spectral.energy_spectrum(view[1:4])[1], spectral.energy_spectrum(prim[1:4])[1],
                          rtol=1e-12, atol=0)


def test_deterministic_mode_gives_the_same_bits(lbm, monkeypatch):
    """Under torch.use_deterministic_algorithms the shells are summed by PyTorch, whose sums then
    come out the same every time: not by this library's pass, whose order varies."""
    import torch
    from paper_2608_13437_gb300 import spectral
    u = torch.randn(3, 70, 66, 72, dtype=torch.float64, device="cuda")
    _, loose = spectral.energy_spectrum(u)
    L = lbm.lib()
    monkeypatch.setattr(L, "lbm_spectral_shells", None)
    torch.use_deterministic_algorithms(True)
    try:
        first, *others = [spectral.energy_spectrum(u)[1] for _ in range(4)]
    finally:
        torch.use_deterministic_algorithms(False)
    assert all(torch.equal(first, e) for e in others)
    assert torch.allclose(first, loose, rtol=1e-12, atol=0)


def _outcome(f, *args):
    """What a call gives, or the kind of error it raises."""
    try:
        r = f(*args)
    except Exception as e:
        return type(e)
    return tuple(np.asarray(v.cpu() if hasattr(v, "cpu") else v, dtype=np.float64) for v in r)


@pytest.mark.parametrize("name,value", [
    ("L_box", 0.0), ("L_box", 0), ("L_box", -2.0), ("L_box", math.nan), ("L_box", math.inf), ("rho_ref", 0.0),
    ("rho_ref", -1.1), ("rho_ref", math.nan), ("T_ref", 0.0), ("T_ref", -0.7), ("T_ref", 1e-310),
    ("T_ref", math.inf), ("mu", 0), ("mu", math.nan), ("mu", -1.0)])
def test_unusual_numbers_do_what_they_do_on_the_cpu(lbm, name, value):
    """Zero, negative and non-finite parameters give the tensor operations' values or errors."""
    import torch
    from paper_2608_13437_gb300 import spectral
    g = torch.Generator().manual_seed(5)
    cpu = torch.rand(6, 4, 6, 5, dtype=torch.float64, generator=g) + 0.5
    dev = cpu.cuda()
    for sutherland in (0, 1):
        a = dict(mu=2e-3, T_ref=0.7, sutherland=sutherland, rho_ref=1.1, L_box=6.0)
        a[name] = value
        got, want = (_outcome(spectral.dissipation, t, *a.values()) for t in (dev, cpu))
        if isinstance(want, type):
            assert got == want, sutherland
        else:
            np.testing.assert_allclose(got, want, rtol=1e-12)
    if name == "L_box":  # no shells of such a box: refused before anything is launched
        for t in (dev[1:4], dev[1:4].float()):
            assert _outcome(spectral.energy_spectrum, t, value) == (IndexError if value < 0 else RuntimeError)
