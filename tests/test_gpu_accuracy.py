"""Solution accuracy against the oracle where the paper's workloads put it:
the torus diffusion-curve batch (8 meridians, 64 right-hand sides through
cpm_rhs's samples) at a grid the oracle factorises directly; the bumpy sphere
(App. A closest points) for the product, the solves and the heat pair (Sec.
7.2); the heat pipeline stage by stage; the FP32 + refinement adjoint; and the
two stopping norms.

Bars: FP64 solves within 1e-10 relative L-inf of the oracle's direct solve,
FP32 + FP64 refinement within 1e-9."""
import math

import numpy as np
import pytest

import cpm_inputs as ci
from gpu_common import need_gpu, pair, rel_inf

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch_mod():
    return need_gpu()


def torus_batch_workload(h, seed=0):
    """8 meridians at equal spacing turned by a seeded phase (the seeded angles of
    the full-size workload crowd two meridians to 0.24 rad, which only grids
    finer than h = 1/115 resolve), 64 U[0,1] value sets."""
    rng = np.random.default_rng(seed)
    phase = rng.uniform(0.0, 2 * math.pi / 8)
    ang = phase + 2 * math.pi * np.arange(8) / 8
    curves = [ci.torus_meridian(float(a), 1.0, 0.4, ci.BC_DIR1) for a in ang]
    g = np.random.default_rng(seed + 1).uniform(0.0, 1.0, size=(8, 64))
    return ci.Workload("torus_batch_small", ci.torus(1.0, 0.4), h, curves, 0.0, 1.0), ang, g


def test_torus_batch_of_64_against_oracle(oracle_mod, torch_mod):
    torch = torch_mod
    w, ang, g = torus_batch_workload(1 / 36)
    band, ref = pair(oracle_mod, w, n_samples=[1] * 8)
    F = band.rhs(samples=torch.tensor(g, device="cuda").contiguous(), nrhs=64)
    Fr = np.stack([ref.rhs(np.zeros(ref.NS), g[:, k][ref.bc_curve]) for k in range(64)], axis=1)
    # a one-sample curve's value is interpolated as (1 - t) g + t g: within an
    # ulp of g
    assert np.max(np.abs(F.cpu().numpy() - Fr)) <= 2.3e-16 * np.max(np.abs(Fr))
    import scipy.sparse.linalg as spla
    lu = spla.splu(ref.A(0.0, 1.0).tocsc())
    Xr = lu.solve(Fr)
    for mode, bar in (("fp32_ir", 1e-9), ("fp64", 1e-10)):
        x, st = band.solve(0.0, 1.0, F, tol=1e-12, mode=mode, raise_on_error=False)
        assert st.status == "CPM_OK" and st.relres <= max(1e-12, 4 * st.relres_floor), (mode, st)
        X = x.cpu().numpy()
        worst = max(rel_inf(X[:, k], Xr[:, k]) for k in range(64))
        assert worst < bar, (mode, worst, st)
    # the closed form: piecewise linear in the toroidal angle between meridians
    a = band.extend(x).cpu().numpy()
    phi = np.arctan2(ref.cp[:, 1], ref.cp[:, 0]) % (2 * math.pi)
    o = np.argsort(ang % (2 * math.pi))
    aa = np.concatenate([(ang % (2 * math.pi))[o], [(ang % (2 * math.pi))[o][0] + 2 * math.pi]])
    for k in (0, 63):
        gg = np.concatenate([g[o, k], [g[o, k][0]]])
        ex = np.interp(np.where(phi < aa[0], phi + 2 * math.pi, phi), aa, gg)
        assert np.max(np.abs(a[:, k] - ex)) < 0.05


@pytest.fixture(scope="module")
def bumpy(oracle_mod, torch_mod):
    """The bumpy sphere at h = 1/24 with a point source at +z (the heat pair's
    setting); skipped if the two bands differ (closest points near the band
    radius may differ in the last bits between the two exp())."""
    sh = ci.bumpy_sphere(16, seed=0)
    h = 1 / 24
    rho = float(ci.bumpy_radius(sh, np.array([0.0, 0.0, 1.0])))
    w = ci.Workload("bumpy_heat", sh, h, [ci.point_curve((0.0, 0.0, rho))], 1.0, -h)
    band, ref = pair(oracle_mod, w)
    ijk, cp = band.export_band()
    if band.NS != ref.NS or not np.array_equal(ijk.cpu().numpy(), ref.ijk):
        pytest.skip("bands differ at nodes on the band radius")
    assert np.max(np.abs(cp.cpu().numpy() - ref.cp)) < 1e-12
    return w, band, ref


@pytest.fixture(scope="module")
def bumpy_refs(bumpy):
    """The oracle's solutions on the bumpy band, each matrix factorised once:
    A(1, -h) for the random right-hand side and the heat step, A(0, 1) for the
    Poisson step from the oracle's own normalised gradient."""
    import scipy.sparse.linalg as spla
    w, band, ref = bumpy
    lu = spla.splu(ref.A(w.m, w.n).tocsc())
    rng = np.random.default_rng(3)
    s = rng.uniform(-1, 1, ref.NS)
    out = {"s": s, "xr": lu.solve(ref.rhs(s, np.ones(ref.NC))), "vr": lu.solve(ref.rhs(None, np.ones(ref.NC)))}
    out["Xr"] = ref.surface_gradient(out["vr"], normalize=True)
    out["br"] = ref.surface_divergence(out["Xr"])
    out["phir"] = spla.splu(ref.A(0.0, 1.0).tocsc()).solve(ref.rhs(out["br"], np.zeros(ref.NC)))
    return out


def test_bumpy_products_and_solves(bumpy, bumpy_refs, torch_mod):
    torch = torch_mod
    w, band, ref = bumpy
    U = ci.random_vector(ref.N, seed=41, nrhs=3)
    VR = ref.A(w.m, w.n) @ U
    V = band.apply(w.m, w.n, torch.tensor(U, device="cuda")).cpu().numpy()
    # the closest points agree to ~1e-15, so the weights do too
    assert max(rel_inf(V[:, r], VR[:, r]) for r in range(3)) < 1e-12
    V32 = band.apply(w.m, w.n, torch.tensor(U, device="cuda", dtype=torch.float32)).cpu().numpy()
    assert np.max(np.abs(V32 - VR)) <= 2e-6 * np.max(np.abs(VR))
    s, xr = bumpy_refs["s"], bumpy_refs["xr"]
    fg = band.rhs(s=torch.tensor(s, device="cuda"), g=torch.ones(band.NC, dtype=torch.float64, device="cuda"))
    for mode, bar in (("fp64", 1e-10), ("fp32_ir", 1e-9)):
        x, st = band.solve(w.m, w.n, fg, tol=1e-13, mode=mode, raise_on_error=False)
        assert rel_inf(x.cpu().numpy(), xr) < bar, (mode, st)


@pytest.mark.parametrize("mode", ["fp64", "fp32_ir"])
def test_bumpy_heat_pair_stage_by_stage(bumpy, bumpy_refs, torch_mod, mode):
    """Sec. 7.2 on the bumpy sphere, each stage from the oracle's input to it:
    the heat step v, X = -grad v / |grad v| from the oracle's v, and phi from the
    oracle's X; then the whole pipeline."""
    torch = torch_mod
    w, band, ref = bumpy
    h = w.h
    bar = 1e-10 if mode == "fp64" else 1e-9
    # (1) heat step (I - dt M) v = [0 ; 1], dt = h
    assert (w.m, w.n) == (1.0, -h)
    vr = bumpy_refs["vr"]
    v, st = band.solve(1.0, -h, band.rhs(g=torch.ones(band.NC, dtype=torch.float64, device="cuda")), tol=1e-13,
                       mode=mode, raise_on_error=False)
    assert rel_inf(v.cpu().numpy(), vr) < bar, st
    # (2) normalised gradient of the oracle's v
    Xr = bumpy_refs["Xr"]
    X = band.surface_gradient(torch.tensor(vr, device="cuda"), normalize=True).cpu().numpy()
    assert rel_inf(X, Xr) < 1e-12
    # (3) divergence and Poisson solve from the oracle's X
    br = bumpy_refs["br"]
    b = band.surface_divergence(torch.tensor(Xr, device="cuda")).cpu().numpy()
    assert rel_inf(b, br) < 1e-12
    phir = bumpy_refs["phir"]
    phi, st = band.solve(0.0, 1.0, band.rhs(s=torch.tensor(br, device="cuda"),
                                            g=torch.zeros(band.NC, dtype=torch.float64, device="cuda")),
                         tol=1e-13, mode=mode, raise_on_error=False)
    assert rel_inf(phi.cpu().numpy(), phir) < bar, st


def test_heat_pipeline_stage_by_stage_on_the_sphere(oracle_mod, torch_mod):
    """The unit-sphere heat method (point at an off-axis point, h = 1/16) stage
    by stage: the whole pipeline's deviation is the normalisation's conditioning
    acting on the heat step's solver residual, so each stage is compared from the
    oracle's own input to it, at the solver's bar."""
    torch = torch_mod
    p = np.array([0.3, 0.2, 0.93]); p /= np.linalg.norm(p)
    h = 1 / 16
    w = ci.Workload("sph_pt", ci.sphere(), h, [ci.point_curve(tuple(p))], 0.0, 1.0)
    band, ref = pair(oracle_mod, w)
    vr = ref.solve_direct(1.0, -h, ref.rhs(None, np.ones(ref.NC)))
    v, st = band.solve(1.0, -h, band.rhs(g=torch.ones(band.NC, dtype=torch.float64, device="cuda")), tol=1e-13,
                       raise_on_error=False)
    assert rel_inf(v.cpu().numpy(), vr) < 1e-10
    Xr = ref.surface_gradient(vr, normalize=True)
    assert rel_inf(band.surface_gradient(torch.tensor(vr, device="cuda"), normalize=True).cpu().numpy(), Xr) < 1e-12
    br = ref.surface_divergence(Xr)
    phir = ref.solve_direct(0.0, 1.0, ref.rhs(br, np.zeros(ref.NC)))
    phi, st = band.solve(0.0, 1.0, band.rhs(s=torch.tensor(br, device="cuda"),
                                            g=torch.zeros(band.NC, dtype=torch.float64, device="cuda")), tol=1e-13,
                         raise_on_error=False)
    assert rel_inf(phi.cpu().numpy(), phir) < 1e-10


def test_fp32_refinement_adjoint_gradients(oracle_mod, torch_mod):
    """The autograd wrapper with FP32 + refinement solves (forward and adjoint):
    dL/dsamples against the oracle's B^T (c lambda_C), dL/ds = lambda on the PDE
    rows, and central differences of the quadratic loss (exact for any step)."""
    torch = torch_mod
    from paper_2305_04711_gb300.autograd import cpm_solve
    h = 1 / 12
    w, samples, coef = ci.config4(h, nsamples=64, seed=0)
    band, ref = pair(oracle_mod, w, n_samples=[len(samples)])
    target = torch.tensor(ci.target_field(coef, ref.cp), device="cuda")
    s0 = ci.random_vector(ref.NS, seed=9)
    s_dev = torch.tensor(s0, device="cuda", requires_grad=True)
    g_dev = torch.tensor(samples, device="cuda", requires_grad=True)

    def loss_of(sv, gv):
        u = cpm_solve(band, 0.0, 1.0, sv, gv, tol=1e-12, mode="fp32_ir")
        return 0.5 * ((u[:band.NS] - target) ** 2).sum()

    L = loss_of(s_dev, g_dev)
    L.backward()
    gs, gg = s_dev.grad.cpu().numpy(), g_dev.grad.cpu().numpy()
    B = ref.sample_matrix([len(samples)])
    u0 = ref.solve_direct(0.0, 1.0, ref.rhs(s0, B @ samples))
    rhs = np.zeros(ref.N)
    rhs[:ref.NS] = u0[:ref.NS] - ci.target_field(coef, ref.cp)
    lam = ref.solve_adjoint_direct(0.0, 1.0, rhs)
    assert rel_inf(gg, B.T @ (ref.bc_scale() * lam[ref.NS:])) < 1e-8
    assert rel_inf(gs, lam[:ref.NS]) < 1e-8
    rng = np.random.default_rng(5)
    with torch.no_grad():
        for k in rng.choice(len(samples), size=4, replace=False):
            e = torch.zeros_like(g_dev)
            e[k] = 1.0
            fd = (float(loss_of(s_dev, g_dev + e)) - float(loss_of(s_dev, g_dev - e))) / 2.0
            assert abs(fd - gg[k]) / max(abs(gg[k]), 1e-3 * np.max(np.abs(gg))) < 1e-6
        for k in rng.choice(ref.NS, size=4, replace=False):
            e = torch.zeros_like(s_dev)
            e[k] = 1.0
            fd = (float(loss_of(s_dev + e, g_dev)) - float(loss_of(s_dev - e, g_dev))) / 2.0
            assert abs(fd - gs[k]) / max(abs(gs[k]), 1e-3 * np.max(np.abs(gs))) < 1e-6


@pytest.mark.parametrize("norm", ["plain", "scaled"])
@pytest.mark.parametrize("mode", ["fp64", "fp32_ir"])
def test_stopping_norms(oracle_mod, torch_mod, norm, mode):
    """The reported relative residual is the requested norm of f - A x, computed
    here from the oracle's assembled A: plain |r|_2 / |f|_2 (Sec. 5.4) or the
    Jacobi-scaled one."""
    torch = torch_mod
    w = ci.config2(1 / 16, ci.BC_DIR2)
    band, ref = pair(oracle_mod, w)
    rng = np.random.default_rng(8)
    s = rng.uniform(-1, 1, ref.NS)
    g = rng.uniform(0, 1, ref.NC)
    f = ref.rhs(s, g)
    fg = band.rhs(s=torch.tensor(s, device="cuda"), g=torch.tensor(g, device="cuda"))
    x, st = band.solve(0.0, 1.0, fg, tol=1e-9, mode=mode, norm=norm)
    r = f - ref.A(0.0, 1.0) @ x.cpu().numpy()
    wgt = np.ones(ref.N)
    if norm == "scaled":
        wgt[:ref.NS] = ref.precond(0.0, 1.0)[0]
    rel = np.linalg.norm(wgt * r) / np.linalg.norm(wgt * f)
    assert rel <= 1e-9 * 1.01
    assert rel == pytest.approx(st.relres, rel=1e-3, abs=1e-14)


@pytest.mark.parametrize("p", [3, 2])
def test_every_launch_shape_keeps_the_products(oracle_mod, torch_mod, p):
    """Every launch-shape candidate of the tuner (x passes of the cell gather,
    its grid, the combine's grid; per-row or per-cell single gather), set through
    cpm_set_tune, computes the same product: FP64 within 1e-14 of the oracle,
    FP32 within 2e-6 of max |A u|, at 64 (two columns per lane) and 24 columns."""
    torch = torch_mod
    w = ci.config2(1 / 20, ci.BC_DIR2)
    band, ref = pair(oracle_mod, w, p=p)
    U = ci.random_vector(ref.N, seed=77, nrhs=64)
    VR = ref.A(0.0, 1.0) @ U
    np1 = p + 1
    for dt in (torch.float32, torch.float64):
        xhs = [x for x in (1, 2, 3, 4) if np1 % x == 0 and not (dt == torch.float64 and np1 // x > 2)]
        for nrhs in (64, 24):
            Ug = torch.tensor(U[:, :nrhs], device="cuda", dtype=dt).contiguous()
            for xh in xhs:
                for g in (4, 32):
                    for wps in (16, 128):
                        band.set_tune(nrhs, dt, cells_xh=xh, cells_blocks_per_sm=g, combine_warps_per_sm=wps)
                        V = band.apply(0.0, 1.0, Ug).cpu().numpy()
                        if dt == torch.float64:
                            assert max(rel_inf(V[:, r], VR[:, r]) for r in range(nrhs)) < 1e-14, (nrhs, xh, g, wps)
                        else:
                            assert np.max(np.abs(V - VR[:, :nrhs])) <= 2e-6 * np.max(np.abs(VR)), (nrhs, xh, g, wps)
        u1 = torch.tensor(U[:, 0], device="cuda", dtype=dt).contiguous()
        for mode in (0, 1, 2):
            band.set_tune(1, dt, single_mode=mode)
            v = band.apply(0.0, 1.0, u1).cpu().numpy()
            if dt == torch.float64:
                assert rel_inf(v, VR[:, 0]) < 1e-14, mode
            else:
                assert np.max(np.abs(v - VR[:, 0])) <= 2e-6 * np.max(np.abs(VR[:, 0])), mode
    from paper_2305_04711_gb300._lib import CpmError
    with pytest.raises(CpmError, match="CPM_ERR_ARG"):
        band.set_tune(64, torch.float32, cells_xh=np1 + 1)


def test_autotune_choices_keep_the_products(oracle_mod, torch_mod):
    """cpm_autotune picks launch shapes by timing and reports the kept ones; the
    batched products still match the oracle afterwards and a solve converges."""
    torch = torch_mod
    w = ci.config2(1 / 20, ci.BC_DIR2)
    band, ref = pair(oracle_mod, w)
    for dt in (torch.float32, torch.float64):
        info = band.autotune(64, dt)
        assert info["product_ms"] > 0 and info["product_ms"] <= info["product_ms_default"] * 1.0001
        assert info["cells_xh"] in ((1, 2, 4) if dt == torch.float32 else (2, 4)), info
        assert info["cells_blocks_per_sm"] in (4, 8, 16, 32) and info["combine_warps_per_sm"] in (16, 32, 64, 128)
        assert info["vec_blocks_per_sm"] in (1, 2, 4)
    U = ci.random_vector(ref.N, seed=77, nrhs=64)
    VR = ref.A(0.0, 1.0) @ U
    V = band.apply(0.0, 1.0, torch.tensor(U, device="cuda")).cpu().numpy()
    V32 = band.apply(0.0, 1.0, torch.tensor(U, device="cuda", dtype=torch.float32)).cpu().numpy()
    assert max(rel_inf(V[:, r], VR[:, r]) for r in range(64)) < 1e-14
    assert np.max(np.abs(V32 - VR)) <= 2e-6 * np.max(np.abs(VR))
    x, st = band.solve(0.0, 1.0, band.rhs(g=torch.ones((band.NC, 64), dtype=torch.float64, device="cuda"), nrhs=64),
                       tol=1e-10, mode="fp32_ir")
    assert st.status == "CPM_OK"


@pytest.mark.parametrize("dtype, nrhs, products", [("float32", 64, 9), ("float32", 65, 9), ("float64", 64, 5)])
def test_autotune_times_what_has_an_effect(torch_mod, dtype, nrhs, products):
    """Four products each (one untimed) of the shapes in force and of every candidate: four grids of the FP32 cell
    gather and four of the combine.  The report names the defaults that the products take."""
    torch = torch_mod
    from paper_2305_04711_gb300.cpm import Band
    w = ci.config2(1 / 16)
    band = Band(w.shape, w.h).set_boundary(w.curves)
    band.reserve(nrhs, fp32_ir=True)
    band.profile(True)
    info = band.autotune(nrhs, getattr(torch, dtype))
    assert band.profile(False)["applies"] == 4 * products
    assert info["product_ms"] <= info["product_ms_default"]
    assert info["cells_blocks_per_sm"] in ((4,) if dtype == "float64" else (4, 8, 16, 32))
