"""Transfers between host arrays and the state: populations and moments in staged pieces of whole
tiles (domains above the staging size) and in one, pageable, page-locked and device buffers,
and initial fields from separate host arrays."""
import ctypes

import numpy as np
import pytest

from paper_2608_13437_gb300 import inputs

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


def _domain(lbm, shape, store="f32", held=0, **kw):
    nx, ny, nz = shape
    p = inputs.sod_params(64) if held else inputs.tgv_params(16)
    p.update(nx=nx, ny=ny, nz=nz, dx=2 * np.pi / 40, **kw)
    if not held:
        p.update(sutherland=0, f_mu=0.3, J_min=1e-3, tau_R=0.05, tau_q=0.05)
    return lbm.Domain(p, store=store)


# two pieces of FP64 populations (342400 cells each at most), one piece, rows shorter than a
# tile, one cell
@pytest.mark.parametrize("shape", [(96, 75, 72), (40, 9, 5), (5, 7, 3), (1, 1, 1)])
@pytest.mark.parametrize("store,held,streaming", [("f32", 0, 0), ("f16", 0, 1), ("bf16", 1, 0)])
def test_populations_in_every_form(lbm, shape, store, held, streaming):
    """FP64 and FP32 values are f = w Q_ref + s g of the native bits, rounded once; native bits set
    into another handle come back, and FP64 values give what their rounding to the storage
    type gives (the encoding rule on the host), at both parities."""
    import torch
    nx, ny, nz = shape
    s = inputs.random_smooth_state(nx, ny, nz, seed=3, amp=0.1)
    fields = (s["rho"], s["ux"], s["uy"], s["uz"], s["p"])
    d = _domain(lbm, shape, store, held, streaming=streaming)
    e = _domain(lbm, shape, store, held, streaming=streaming)
    d.init_fields(*fields)
    e.init_fields(*fields)
    d.step(2)
    for n in (1, 1):
        d.step(n)
        e.step(1)  # the parity of d or the other one: the canonical order does not know it
        bits = d.populations("native")
        info = d.info()
        w = np.array([0.25] + [0.125] * 6)[None, :, None, None, None]
        ref = np.zeros((14, 1, 1, 1, 1))
        ref[0], ref[4] = info["rho_ref"], info["E_ref"]
        scale = np.float32(info["scale"]).astype(np.float64)[:, None, None, None, None]
        g = bits if store == "f32" else (bits.view(np.float16) if store == "f16" else
                                         (bits.astype(np.uint32) << 16).view(np.float32))
        f64 = d.populations(np.float64)
        if not held:  # a held end reads the ghost value, which 16-bit storage does not round
            assert np.array_equal(f64, w * ref + scale * g.astype(np.float64))
        assert np.array_equal(d.populations(np.float32), f64.astype(np.float32))
        dev = torch.empty(bits.size, dtype=torch.int32 if store == "f32" else torch.int16, device="cuda")
        pin = torch.empty_like(dev, device="cpu").pin_memory()
        for t, on in ((dev, 1), (pin, 0)):
            lbm.check(lbm.lib().lbm_populations_get(d.handle, ctypes.c_void_p(t.data_ptr()), on, lbm.DT_NATIVE))
            torch.cuda.synchronize()
            assert np.array_equal(t.cpu().numpy().view(bits.dtype).reshape(bits.shape), bits)
        e.set_populations(np.zeros_like(bits), native=True)
        e.set_populations(bits, native=True)
        assert np.array_equal(e.populations("native"), bits)
        e.set_populations(f64)
        dev32 = (f64 - w * ref).astype(np.float32) * (np.float32(1) / scale.astype(np.float32))
        if store == "f32":
            want = dev32
        elif store == "f16":
            want = dev32.astype(np.float16).view(np.uint16)
        else:  # round to nearest even on the upper 16 bits
            u = dev32.view(np.uint32)
            want = ((u + 0x7FFF + ((u >> 16) & 1)) >> 16).astype(np.uint16)
        got = e.populations("native")
        if held:  # the inward populations of the held cells stay the ghost's
            got[:, 1, :, :, 0], got[:, 2, :, :, -1] = want[:, 1, :, :, 0], want[:, 2, :, :, -1]
        assert np.array_equal(got, want)
        e.set_populations(np.zeros_like(bits), native=True)
        lbm.check(lbm.lib().lbm_populations_set(e.handle, ctypes.c_void_p(dev.data_ptr()), 1, lbm.DT_NATIVE))
        assert np.array_equal(e.populations("native"), bits)
    d.close()
    e.close()


def test_moments_and_sensor_to_the_host_in_pieces(lbm):
    """2.5 M cells: the FP64 moments take two pieces; host and device outputs are equal."""
    import torch
    d = _domain(lbm, (150, 137, 123), "f16")
    d.init_tgv(1.0, 0.9, 1.0)
    d.step(3)
    for which in (0, 1):
        assert np.array_equal(d.moments(which), d.moments_device(which, torch.float64).cpu().numpy())
    out = torch.empty((3,) + d.shape, dtype=torch.float64, device="cuda")
    lbm.check(lbm.lib().lbm_sensor(d.handle, ctypes.c_void_p(out.data_ptr()), 1, lbm.DT_F64))
    assert np.array_equal(np.stack(d.sensor()), out.cpu().numpy())
    d.close()


@pytest.mark.parametrize("dtype", [np.float64, np.float32])
def test_initial_fields_from_separate_arrays(lbm, dtype):
    """Scalars, read-only, strided and single-precision arrays give the state that one array of
    all five gives."""
    shape = (33, 20, 7)
    s = inputs.random_smooth_state(*shape, seed=9, amp=0.1)
    uy = np.asfortranarray(s["uy"])
    p = s["p"].astype(np.float32)
    p.flags.writeable = False
    a, b = _domain(lbm, shape), _domain(lbm, shape)
    a.init_fields(s["rho"], 0.25, uy, s["uz"][:, :, :1], p, dtype=dtype)
    full = np.stack([np.broadcast_to(v, a.shape) for v in (s["rho"], 0.25, uy, s["uz"][:, :, :1], p)])
    full = np.ascontiguousarray(full, dtype=dtype)
    lbm.check(lbm.lib().lbm_init_fields(b.handle, lbm._np_ptr(full), 0,
                                        lbm.DT_F64 if dtype == np.float64 else lbm.DT_F32))
    assert np.array_equal(a.populations("native"), b.populations("native"))
    ptrs = (ctypes.c_void_p * 5)(*[full[j].ctypes.data for j in range(4)], None)
    assert lbm.lib().lbm_init_fields_arrays(a.handle, ptrs, lbm.DT_F64) == lbm.LBM_E_INVAL
    with pytest.raises(lbm.LbmError):
        a.init_fields(np.nan, 0.0, 0.0, 0.0, 1.0, dtype=dtype)
    a.close()
    b.close()


# rows of whole tiles and ragged ones, held x ends and periodic, both parities
@pytest.mark.parametrize("shape", [(64, 5, 3), (37, 6, 5)])
@pytest.mark.parametrize("held", [0, 1])
@pytest.mark.parametrize("store", ["f32", "f16", "bf16"])
def test_primitives_follow_from_the_moments(lbm, shape, held, store):
    """Primitives and all 14 moments come from kernels of their own; density, velocity and
    pressure agree with what the moments say to FP32 rounding (a sum of eight terms and the
    closure: 4e-6 of the largest value)."""
    nx, ny, nz = shape
    s = inputs.random_smooth_state(nx, ny, nz, seed=9, amp=0.1)
    for streaming in (0, 1):
        d = _domain(lbm, shape, store, held, streaming=streaming)
        d.init_fields(s["rho"], s["ux"] + 0.1, s["uy"], s["uz"], s["p"])
        for _ in range(3):
            d.step(1)
            Q, P = d.moments(lbm.MOM_Q), d.primitives()
            gamma = d.params["gamma"]
            u = Q[1:4] / Q[0]
            want = [Q[0], *u, (gamma - 1) * (Q[4] - 0.5 * Q[0] * (u * u).sum(0))]
            for j, w in zip((0, 1, 2, 3, 5), want):
                assert np.abs(P[j] - w).max() <= 4e-6 * np.abs(w).max(), (j, streaming)
        d.close()


def test_transfers_with_little_device_memory_left(lbm):
    """With 160 MB left on the device, a domain whose transfers stage 256 MB at a time takes
    smaller pieces, and calls that need memory of their own get what the staging buffer holds."""
    import torch
    shape = (96, 96, 96)  # 347 MB of populations
    s = inputs.random_smooth_state(*shape, seed=13, amp=0.1)
    fields = (s["rho"], s["ux"], s["uy"], s["uz"], s["p"])

    def run(d):
        d.init_fields(*fields)
        d.step(3)
        f = d.populations("native")
        g = d.populations(np.float64)
        d.init_fields(*fields)
        d.set_populations(f, native=True)
        return f, g, d.moments(), d.sensor(), d.diag()["sum_E"]

    a = _domain(lbm, shape)
    want = run(a)
    a.close()
    torch.cuda.empty_cache()
    d = _domain(lbm, shape)
    hog = torch.empty(torch.cuda.mem_get_info()[0] - (160 << 20), dtype=torch.uint8, device="cuda")
    try:
        got = run(d)
        d.step(5)
        e = d.step_diag(2)
    finally:
        del hog
        torch.cuda.empty_cache()
    assert e["status"] == lbm.LBM_OK
    d.close()
    for x, y in zip(want, got):
        assert np.array_equal(np.asarray(x), np.asarray(y))
