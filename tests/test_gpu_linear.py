"""Domains whose rows are not whole 32-cell tiles (and held x ends) take one warp per tile over
the linear cell index, with the L2 prefetch of tiles ahead."""
import numpy as np
import pytest

from conftest import make_oracle
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


# rows shorter than a tile that end several rows and planes inside it, rows that end once, a
# last tile of one cell, and (held) rows of whole tiles
@pytest.mark.parametrize("shape", [(1, 1, 40), (3, 2, 20), (5, 7, 11), (31, 3, 2), (33, 1, 5), (40, 5, 3), (64, 2, 3)])
@pytest.mark.parametrize("held", [0, 1])
def test_linear_steps_against_oracle_and_over_prefetch_distances(lbm, shape, held):
    """FP32 within a relative L2 of 1e-5 of the FP64 oracle (the parity bar) after 9 steps, both
    maps, both register budgets; populations equal bit for bit over prefetch distances that
    land inside the domain, wrap along z and lie beyond it; in-step diagnostics as lbm_diag's."""
    nx, ny, nz = shape
    p = inputs.sod_params(64) if held else inputs.tgv_params(16)
    p.update(nx=nx, ny=ny, nz=nz, dx=2 * np.pi / 40)
    if not held:
        p.update(sutherland=0, f_mu=0.3, J_min=1e-3, tau_R=0.05, tau_q=0.05)
    s = inputs.random_smooth_state(nx, ny, nz, seed=5, amp=0.1)
    fields = (s["rho"], s["ux"] + 0.1, s["uy"] + 0.1, s["uz"] + 0.1, s["p"])
    o = make_oracle(p)
    o.init_fields(*fields)
    o.step(9)
    ref = o.primitives()
    bits = None
    for streaming in (0, 1):
        for pf, variant in ((0, 0), (1, 0), (3, 1), (1024, 0)):
            d = lbm.Domain(dict(p, streaming=streaming))
            d.set_kernel_config(64, variant)
            d.set_prefetch(pf)
            d.init_fields(*fields)
            d.step(4)
            first = d.diag()
            got = d.step_diag(5)
            for k in ("max_mach", "max_cfl", "min_rho", "min_T", "eps_s_raw", "eps_d_raw"):
                assert got[k] == first[k], k
            assert got["sum_rho"] == pytest.approx(first["sum_rho"], rel=1e-11)
            f = d.populations("native")
            bits = f if bits is None else bits
            assert np.array_equal(f, bits), (streaming, pf, variant)
            prim = d.primitives()
            for j in (0, 1, 2, 3, 4):
                err = np.linalg.norm(prim[j] - ref[j]) / max(np.linalg.norm(ref[j]), 1e-300)
                assert err < 1e-5, (j, err)
            d.close()
