"""The gradient pass of the diagnostics cuts its columns along z into pieces whose height
depends on how many columns the domain has, and its last block finishes the reductions."""
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


@pytest.mark.parametrize("shape", [(32, 16, 1), (32, 17, 2), (33, 5, 3), (64, 16, 7), (7, 3, 33),
                                   (40, 33, 12), (96, 64, 37)])
def test_diag_against_oracle_over_column_cuts(lbm, shape):
    """One plane, odd plane counts, a last piece of one plane, partial columns; both
    diagnostic paths, twice on the same scratch. Tolerances as in the parity tests: 2e-6
    on sums and extrema, 1e-4 on the dissipation integrals, FP32 against the FP64 oracle."""
    from oracle import oracle as O
    nx, ny, nz = shape
    p = inputs.tgv_params(16)
    p.update(nx=nx, ny=ny, nz=nz, dx=2 * np.pi / 40, sutherland=0, f_mu=0.3, J_min=1e-3,
             tau_R=0.05, tau_q=0.05)
    s = inputs.random_smooth_state(nx, ny, nz, seed=nx + nz, amp=0.1)
    fields = (s["rho"], s["ux"] + 0.1, s["uy"] + 0.1, s["uz"] + 0.1, s["p"])
    dom = lbm.Domain(p)
    dom.init_fields(*fields)
    q = dict(p)
    o = O.Oracle(q.pop("nx"), q.pop("ny"), q.pop("nz"), q.pop("dx"), **q)
    o.init_fields(*fields)
    for n in (3, 2):
        dom.step(n)
        o.step(n)
        r = o.diag()
        st = lbm.LbmDiag()
        lbm.check(lbm.lib().lbm_diag_static(dom.handle, ctypes.byref(st)))
        first = dom.diag()
        assert {k: getattr(st, k) for k in lbm.DIAG_FIELDS} == {k: first[k] for k in lbm.DIAG_FIELDS}
        for g in (first, dom.step_diag(1)):
            for k in ("sum_rho", "sum_E", "ek_mean", "min_rho", "min_T", "max_mach", "max_cfl"):
                assert g[k] == pytest.approx(r[k], rel=2e-6), k
            for k in ("sum_mx", "sum_my", "sum_mz"):
                assert g[k] == pytest.approx(r[k], abs=2e-6 * r["sum_rho"]), k
            for k in ("eps_s_raw", "eps_d_raw"):
                assert g[k] == pytest.approx(r[k], rel=1e-4), k
            assert g["nonfinite"] == 0
        o.step(1)
    dom.close()
