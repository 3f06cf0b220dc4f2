"""Domain.init_fields hands the library arrays of the type it names, whatever it is given."""
import ctypes

import numpy as np
import pytest

from paper_2608_13437_gb300 import lbm


class FakeLibrary:
    """Records the values that an initialisation would read."""

    def __init__(self, cells):
        self.cells, self.seen = cells, []

    def _read(self, at, n, dtype):
        t = ctypes.c_double if dtype == lbm.DT_F64 else ctypes.c_float
        return np.ctypeslib.as_array((t * n).from_address(at)).astype(np.float64)

    def lbm_init_fields_arrays(self, h, ptrs, dtype):
        self.seen.append(("arrays", dtype, [p for p in ptrs]))
        return lbm.LBM_OK

    def lbm_init_fields(self, h, fields, on_device, dtype):
        at = ctypes.cast(fields, ctypes.c_void_p).value
        self.seen.append(("stacked", dtype, self._read(at, 5 * self.cells, dtype)))
        return lbm.LBM_OK


@pytest.fixture
def domain(monkeypatch):
    d = lbm.Domain.__new__(lbm.Domain)
    d._h, d.shape = None, (2, 3, 4)
    fake = FakeLibrary(24)
    monkeypatch.setattr(lbm, "lib", lambda: fake)
    return d, fake


@pytest.mark.parametrize("types", [("f8", "f4", "f8", "f4", "f8"), ("f4",) * 5, ("f4", "f4", "f4", "f4", "f8")])
def test_no_type_given_takes_the_common_one(domain, types):
    """dtype=None: the arrays are of different sizes, so they are stacked to their common type."""
    d, fake = domain
    arrs = [np.full(d.shape, j + 0.5, dtype=t) for j, t in enumerate(types)]
    d.init_fields(*arrs, dtype=None)
    (how, dtype, values), = fake.seen
    assert how == "stacked"
    assert dtype == (lbm.DT_F64 if "f8" in types else lbm.DT_F32)
    assert np.array_equal(values.reshape(5, 24), np.repeat(np.arange(5) + 0.5, 24).reshape(5, 24))


@pytest.mark.parametrize("dtype", [np.float32, np.float64, "f4", float])
def test_a_type_given_goes_as_five_arrays(domain, dtype):
    d, fake = domain
    d.init_fields(1.0, np.zeros(d.shape, np.float32), 0, np.arange(4), np.ones(d.shape), dtype=dtype)
    (how, dt, _), = fake.seen
    assert how == "arrays" and dt == (lbm.DT_F64 if np.dtype(dtype) == np.float64 else lbm.DT_F32)
