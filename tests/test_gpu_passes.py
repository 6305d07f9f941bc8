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


@pytest.mark.parametrize("adjoint", [False, True])
def test_fp64_finish_of_a_few_columns(adjoint):
    """A refined batch of 16 whose columns 3 and 11 are left after one FP32 step: an FP64 solve of these two
    alone ends them, the others keep their bits."""
    torch = need_gpu()
    from paper_2305_04711_gb300.cpm import Band
    w = ci.config2(1 / 16)
    band = Band(w.shape, w.h).set_boundary(w.curves)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(4)
    f = torch.randn((band.N, 16), generator=gen, dtype=torch.float64, device="cuda")
    done, st = band.solve(0.0, 1.0, f, tol=1e-11, mode="fp64", adjoint=adjoint)
    x0 = done.clone()
    x0[:, [3, 11]] = 0.0
    x, st = band.solve(0.0, 1.0, f, x0=x0, tol=1e-10, mode="fp32_ir", max_refine=1, adjoint=adjoint)
    assert st.status == "CPM_OK" and st.refinements == 1 and st.fp64_iterations > 0, st
    rest = [c for c in range(16) if c not in (3, 11)]
    assert torch.equal(x[:, rest], done[:, rest])
    rel = (f - band.apply(0.0, 1.0, x, transpose=adjoint)).norm(dim=0) / f.norm(dim=0)
    assert float(rel.max()) <= 1.01 * max(1e-10, 4 * st.relres_floor)
    assert abs(float(rel.max()) - st.relres) <= 0.01 * st.relres
    for c in (3, 11):
        one, _ = band.solve(0.0, 1.0, f[:, c].contiguous(), tol=1e-11, adjoint=adjoint)
        # both residuals are below 1e-10 of f; the smallest eigenvalue between the circles is about 1
        assert float((x[:, c] - one).norm()) <= 1e-6 * float(one.norm())
