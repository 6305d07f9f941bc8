"""FP64 solves that meet their tolerance only in a second pass."""
import pytest

import cpm_inputs as ci
from gpu_common import need_gpu

pytestmark = pytest.mark.gpu


def test_a_pass_that_starts_just_above_tol_ends_below_it():
    """Adjoint solves at tol 1e-11 often end their first pass with a true residual a few per cent above it
    (the recursion's rounding): 2 of 20 such solves ended not converged when the next pass aimed at tol itself."""
    torch = need_gpu()
    from paper_2305_04711_gb300.cpm import Band
    curves = [ci.torus_meridian(a, 1.0, 0.4) for a in (0.3, 2.5)]
    band = Band(ci.torus(), 1 / 22.86).set_boundary(curves)
    gen = torch.Generator(device="cuda")
    for seed in range(20):
        gen.manual_seed(seed)
        g = torch.randn(band.N, generator=gen, dtype=torch.float64, device="cuda")
        _, st = band.solve(0.0, 1.0, g, tol=1e-11, adjoint=True)
        assert st.status == "CPM_OK" and st.relres <= max(1e-11, 4 * st.relres_floor)
