"""Tuning: the autotuner's candidates include what an untuned handle runs with, and the distance
that a handle reports is told apart from the one its steps use."""
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


# 822 MB of FP32 populations (beyond the L2: 256 tiles untuned), 411 MB of FP16 (1024), and 13
# and 6 MB (none; rows of one tile take blocks of 64 only)
@pytest.mark.parametrize("n,store,candidates", [(128, "f32", 20), (128, "f16", 16), (32, "f32", 8), (32, "f16", 8)])
def test_autotune_tries_the_distance_of_an_untuned_handle(lbm, n, store, candidates):
    d = lbm.Domain(inputs.tgv_params(n), store=store)
    d.init_tgv(1.0, 1.25, 1.0)
    t = d.autotune(pairs_per_trial=1)
    assert t["candidates"] == candidates
    assert t["prefetch_tiles"] in ((0, 256, 512, 1024, 2048) if candidates == 20 else (0, 512, 1024, 2048))
    assert d.info()["prefetch_tiles"] == t["prefetch_tiles"]
    d.close()


@pytest.mark.parametrize("sizes,store", [((16, 20), "f16"), ((16, 20), "f32"), ((96, 64), "bf16")])
def test_batch_autotune_keeps_the_result(lbm, sizes, store):
    """From a pool that the L2 holds and one that it does not: the tuned batch steps like an
    untuned one, bit for bit."""
    P = [inputs.tgv_params(n) for n in sizes]
    a, b = lbm.Batch(P, store=store), lbm.Batch(P, store=store)
    args = [1.0] * 2, [1.25, 1.1], [1.0] * 2
    a.init_tgv(*args)
    assert a.autotune(2)["prefetch_tiles"] in (0, 512, 1024, 2048)
    for B in (a, b):
        B.init_tgv(*args)
        B.step(7)
        B.synchronize()
    for d in range(2):
        assert np.array_equal(a.moments(d), b.moments(d))
    a.close()
    b.close()


def _in_effect(lbm, d):
    import ctypes
    n = ctypes.c_int(-1)
    lbm.check(lbm.lib().lbm_prefetch_in_effect(d.handle, ctypes.byref(n)))
    return n.value


# untuned: none while the L2 holds the state, else 256 tiles (FP32) or 1024 (16-bit), ragged
# rows too; the reported default is the storage type's
@pytest.mark.parametrize("shape,store,untuned,default", [
    ((32, 32, 32), "f32", 0, 0), ((128, 128, 128), "f32", 256, 0), ((150, 100, 60), "f32", 256, 0),
    ((64, 64, 64), "f16", 0, 1024), ((128, 128, 128), "bf16", 1024, 1024)])
def test_prefetch_distance_in_effect(lbm, shape, store, untuned, default):
    assert lbm.lib().lbm_prefetch_in_effect(None, None) == lbm.LBM_E_INVAL
    p = inputs.tgv_params(32)
    p.update(nx=shape[0], ny=shape[1], nz=shape[2])
    d = lbm.Domain(p, store=store)
    assert (_in_effect(lbm, d), d.info()["prefetch_tiles"]) == (untuned, default)
    d.set_prefetch(7)
    assert (_in_effect(lbm, d), d.info()["prefetch_tiles"]) == (7, 7)
    d.close()
