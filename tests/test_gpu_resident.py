"""Small domains: lbm_step takes many steps in one launch with the populations held on the
chip. The result has to be the one-launch-per-step kernel's (use_graphs = 0), bit for bit."""
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


# shapes: the configurations in use, bricks that do not divide a side, one brick, two bricks
# along an axis (both neighbours are the same one), sides of one and two cells, long rows,
# the largest domain that fits 152 SMs and one just above it (the plain kernel's, as are
# the sizes at which the plain kernel is the faster one).
SHAPES = [(32, 32, 32), (20, 12, 9), (37, 6, 5), (1, 1, 1), (2, 1, 1), (1, 1, 700), (385, 1, 1),
          (5, 4, 3), (64, 8, 4), (33, 31, 35), (7, 61, 3), (1000, 3, 2), (48, 32, 38), (38, 38, 40)]
FORMS = [("f32", 0, 0), ("f32", 0, 1), ("f16", 0, 0), ("f16", 1, 1), ("bf16", 1, 0), ("bf16", 0, 1)]


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("held", [0, 1])
def test_resident_steps_equal_plain_steps(lbm, shape, held):
    nx, ny, nz = shape
    for j, (store, sr, streaming) in enumerate(FORMS):
        p = inputs.sod_params(64) if held else inputs.tgv_params(16)
        p.update(nx=nx, ny=ny, nz=nz, dx=2 * np.pi / 40, streaming=streaming, stochastic_round=sr)
        if not held:
            p.update(sutherland=j & 1, f_mu=0.3, J_min=1e-3, tau_R=0.05, tau_q=0.05)
        s = inputs.random_smooth_state(nx, ny, nz, seed=11 + j, amp=0.15)
        a, b = lbm.Domain(p, store=store), lbm.Domain(p, store=store, use_graphs=False)
        for d in (a, b):
            d.init_fields(s["rho"], s["ux"], s["uy"] + 0.1, s["uz"], s["p"])
        for n in (8, 9, 1, 8, 11, 3):  # both parities at either end of a launch, plain steps between
            a.step(n)
            b.step(n)
        a.synchronize()
        assert a.step_count == b.step_count == 40
        assert np.array_equal(a.populations("native"), b.populations("native")), (store, sr, streaming)
        whole = nx * ny * nz % 32 == 0  # otherwise the last tile has lanes that nothing writes
        if whole:
            assert lbm_equal(a.buffer, b.buffer), (store, sr, streaming)
        a.close()
        b.close()


def lbm_equal(a, b):
    return bool((a == b).all())


def test_resident_flags_nonfinite_and_recovers(lbm):
    """A NaN put into one cell is reported at the next synchronising call, steps are refused,
    and a re-init gives a fresh handle's result."""
    p = inputs.tgv_params(32)
    d, e = lbm.Domain(p), lbm.Domain(p, use_graphs=False)
    d.init_tgv(1.0, 1.25, 1.0)
    f = d.populations(np.float64)
    f[0, 0, 3, 4, 5] = np.nan
    d.set_populations(f)
    d.step(10)
    with pytest.raises(lbm.LbmError) as ei:
        d.synchronize()
    assert ei.value.status == lbm.LBM_E_NONFINITE
    with pytest.raises(lbm.LbmError):
        d.step(8)
    for h in (d, e):
        h.init_tgv(1.0, 1.25, 1.0)
        h.step(9)
    assert np.array_equal(d.populations("native"), e.populations("native"))
    d.close()
    e.close()


def test_resident_handles_on_two_streams(lbm):
    """Two small domains stepped from two streams at once: each equals its own plain run."""
    import torch
    p = inputs.tgv_params(32)
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    doms, refs = [], []
    for j, st in enumerate(streams):
        with torch.cuda.stream(st):
            doms.append(lbm.Domain(p))
            doms[-1].init_tgv(1.0, 1.0 + 0.1 * j, 1.0)
    for _ in range(5):
        for d in doms:
            d.step(40)
    for j, d in enumerate(doms):
        d.synchronize()
        r = lbm.Domain(p, use_graphs=False)
        r.init_tgv(1.0, 1.0 + 0.1 * j, 1.0)
        r.step(200)
        assert np.array_equal(d.populations("native"), r.populations("native"))
        r.close()
        d.close()


@pytest.mark.parametrize("store,steps", [("f32", 40), ("f16", 5000)])
def test_resident_wait_runs_out_and_is_reported(lbm, store, steps):
    """Failure detection without a fault: one block does nothing, so its neighbours' bounded
    waits run out. The next synchronising call reports LBM_E_TIMEOUT and steps are refused;
    after a re-init the handle steps exactly like a fresh one, whether the host has seen the
    failure in between or not. Launches queued behind the failed one end at once."""
    import time
    p = inputs.tgv_params(32)
    d = lbm.Domain(p, store=store)
    L = lbm.lib()
    assert L.lbm_test_stall_resident(None, 0, 100) == lbm.LBM_E_INVAL
    for block, polls in ((-1, 100), (100000, 100), (0, 0)):
        assert L.lbm_test_stall_resident(d.handle, block, polls) == lbm.LBM_E_INVAL
    ref = lbm.Domain(p, store=store, use_graphs=False)
    assert L.lbm_test_stall_resident(ref.handle, 0, 100) == lbm.LBM_E_INVAL  # plain steps
    ref.init_tgv(1.0, 1.25, 1.0)
    ref.step(33)
    want = ref.populations("native")
    ref.close()
    for synchronise in (True, False, True):
        d.init_tgv(1.0, 1.25, 1.0)
        d.step(9)
        assert L.lbm_test_stall_resident(d.handle, 5, 4000) == lbm.LBM_OK
        t0 = time.time()
        d.step(steps)
        if synchronise:
            with pytest.raises(lbm.LbmError) as ei:
                d.synchronize()
            assert ei.value.status == lbm.LBM_E_TIMEOUT and "neighbouring block" in str(ei.value)
            with pytest.raises(lbm.LbmError) as ei:
                d.step(8)
            assert ei.value.status == lbm.LBM_E_TIMEOUT
        d.init_tgv(1.0, 1.25, 1.0)
        assert time.time() - t0 < 1.0  # 4000 tries are a few ms
        d.step(9)
        d.step(24)
        d.synchronize()
        assert np.array_equal(d.populations("native"), want), synchronise
    d.close()


def test_load_after_a_wait_that_ran_out(lbm, tmp_path):
    """A checkpoint loaded into a handle whose last launch gave up, before the host has seen
    it, steps like the handle that was saved."""
    p = inputs.tgv_params(32)
    a, b = lbm.Domain(p), lbm.Domain(p)
    for d in (a, b):
        d.init_tgv(1.0, 1.25, 1.0)
        d.step(9)
    path = str(tmp_path / "ck.bin")
    a.save(path)
    assert lbm.lib().lbm_test_stall_resident(b.handle, 3, 4000) == lbm.LBM_OK
    b.step(10)
    b.load(path)
    for d in (a, b):
        d.step(11)
        d.synchronize()
    assert np.array_equal(a.populations("native"), b.populations("native"))
    a.close()
    b.close()


def test_creating_a_small_domain_does_not_wait_for_other_work(lbm):
    """lbm_create returns while a kernel on the default stream is still running, and the
    handle's steps on another stream give the plain steps' result."""
    import torch
    p = inputs.tgv_params(32)
    side = torch.cuda.Stream()
    for busy in (False, True):  # the first round fills PyTorch's memory pool
        with torch.cuda.stream(side):
            torch.cuda.synchronize()
            done = torch.cuda.Event()
            if busy:
                with torch.cuda.stream(torch.cuda.default_stream()):
                    torch.cuda._sleep(1 << 29)  # about a quarter of a second
                    done.record()
            d = lbm.Domain(p)
            if busy:
                assert not done.query()
            d.init_tgv(1.0, 1.25, 1.0)
            d.step(20)
            d.synchronize()
            got = d.populations("native")
            d.close()
    r = lbm.Domain(p, use_graphs=False)
    r.init_tgv(1.0, 1.25, 1.0)
    r.step(20)
    assert np.array_equal(got, r.populations("native"))
    r.close()


def resident_steps(lbm, d):
    import ctypes
    n = ctypes.c_longlong()
    lbm.check(lbm.lib().lbm_resident_steps(d.handle, ctypes.byref(n)))
    return n.value


def _cut(shape):
    """The cubes and tubes of this file as parameters and an initial state of their own."""
    nx, ny, nz = shape
    p = inputs.tgv_params(16)
    p.update(nx=nx, ny=ny, nz=nz, dx=2 * np.pi / 40, sutherland=0, f_mu=0.3, J_min=1e-3, tau_R=0.05,
             tau_q=0.05)
    return p


# shape, store, streams, whether domains on that many streams still step on the chip: launches
# that fit beside each other, ones that take turns but are the faster form all the same, and
# ones that would take turns at a loss
@pytest.mark.parametrize("shape,store,streams,on_chip", [
    ((32, 32, 32), "f32", 1, True), ((32, 32, 32), "f32", 2, False), ((32, 32, 32), "f16", 2, False),
    ((1024, 4, 4), "f32", 2, True), ((1024, 4, 4), "f32", 4, True), ((1024, 4, 4), "f16", 8, False),
    ((64, 4, 4), "f16", 12, True), ((38, 38, 38), "bf16", 2, False), ((24, 24, 24), "f32", 2, True)])
def test_small_domains_on_several_streams(lbm, shape, store, streams, on_chip):
    import torch
    doms, refs = [], []
    for j in range(streams):
        s = inputs.random_smooth_state(*shape, seed=5 + j, amp=0.1)
        fields = (s["rho"], s["ux"], s["uy"], s["uz"], s["p"])
        with torch.cuda.stream(torch.cuda.Stream()):
            doms.append(lbm.Domain(_cut(shape), store=store))
            doms[-1].init_fields(*fields)
        r = lbm.Domain(_cut(shape), store=store, use_graphs=False)
        r.init_fields(*fields)
        r.step(60)
        refs.append(r.populations("native"))
        r.close()
    for _ in range(3):
        for d in doms:
            d.step(20)
    for d, ref in zip(doms, refs):
        assert resident_steps(lbm, d) == (60 if on_chip else 0)
        assert np.array_equal(d.populations("native"), ref)
    for d in doms[1:]:
        d.close()
    doms[0].step(20)  # the others are gone
    assert resident_steps(lbm, doms[0]) == (80 if on_chip else 20)
    doms[0].close()


def test_small_domains_on_one_stream_do_not_count_twice(lbm):
    """Three handles on one stream, and a call of more steps than one launch takes."""
    import torch
    shape = (64, 8, 4)
    s = inputs.random_smooth_state(*shape, seed=2, amp=0.01)
    fields = (s["rho"], s["ux"], s["uy"], s["uz"], s["p"])
    side = torch.cuda.Stream()
    with torch.cuda.stream(side):
        doms = [lbm.Domain(_cut(shape)) for _ in range(3)]
        for d in doms:
            d.init_fields(*fields)
            d.step(4200)
            assert resident_steps(lbm, d) == 4200
    a = doms[0].populations("native")
    r = lbm.Domain(_cut(shape), use_graphs=False)
    r.init_fields(*fields)
    r.step(4200)
    assert np.isfinite(a).all() and a.std() > 0
    assert np.array_equal(a, r.populations("native"))
    for d in doms + [r]:
        d.close()


@pytest.mark.parametrize("shape,f32,bits16", [(s, True, True) for s in SHAPES] +
                         [((16, 16, 16), False, True), ((38, 38, 41), False, False), ((64, 64, 64), False, False)])
def test_which_domains_step_on_the_chip(lbm, shape, f32, bits16):
    """The shapes above take the form they are there for; calls of fewer than eight steps, a
    kernel form that was asked for and use_graphs = 0 do not (152 SMs)."""
    import torch
    if torch.cuda.get_device_properties(0).multi_processor_count != 152:
        pytest.skip("the choice is for 152 SMs")
    for store, on_chip in (("f32", f32), ("f16", bits16), ("bf16", bits16)):
        for direct, form in ((False, False), (True, False), (False, True)):
            d = lbm.Domain(_cut(shape), store=store, use_graphs=not direct)
            if form:
                d.set_kernel_config(64, 0)
            d.init_fields(1.0, 0.1, 0.0, 0.0, 1.0)
            d.step(7)
            assert resident_steps(lbm, d) == 0
            d.step(8)
            assert resident_steps(lbm, d) == (8 if on_chip and not direct and not form else 0), store
            d.close()


# above the size limit of the resident form, below it with a kernel form asked for, held x ends
@pytest.mark.parametrize("shape,held,form", [((64, 64, 64), 0, None), ((32, 32, 32), 0, (64, 0)),
                                             ((40, 9, 5), 0, (32, 1)), ((128, 6, 4), 1, (64, 0)),
                                             ((1024, 8, 8), 1, None)])
@pytest.mark.parametrize("store", ["f32", "f16", "bf16"])
def test_graph_replays_equal_direct_launches(lbm, shape, held, form, store):
    """The graphs of two and of 32 steps, with single steps before and after, against one launch
    per step: bit for bit, both streaming maps."""
    nx, ny, nz = shape
    for streaming in (0, 1):
        p = dict(inputs.sod_params(64), nx=nx, ny=ny, nz=nz) if held else _cut(shape)
        p["streaming"] = streaming
        s = inputs.random_smooth_state(nx, ny, nz, seed=21, amp=0.1)
        got = []
        for graphs in (True, False):
            d = lbm.Domain(p, store=store, use_graphs=graphs)
            if form:
                d.set_kernel_config(*form)
            d.init_fields(s["rho"], s["ux"], s["uy"], s["uz"], s["p"])
            d.step(1)
            d.step(70)  # odd parity: one step, two replays of 32, two of 2, one step
            assert resident_steps(lbm, d) == 0
            d.step(33)
            got.append(d.populations("native"))
            d.close()
        assert np.isfinite(got[0].view(np.float32 if store == "f32" else np.uint16).astype(np.float64)).all()
        assert np.array_equal(*got), streaming
