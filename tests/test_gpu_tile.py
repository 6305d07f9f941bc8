"""E u of one or a few columns by warp tiles (integer sums in FP64): every
stencil shape, tiles that end ragged, odd column counts and strides, values at
the ends of the exponent range, infinities and NaN, against the oracle.

Tolerance: both sides round at most 64 products and 20 operations on weights of
sum <= 1.25^3 in FP64, so they differ by at most (64 + 20) 2^-53 1.95 max|u| =
1.9e-14 max|u|; FP32 (apply only, existing bar) 2e-6 of max|A u|."""
import numpy as np
import pytest

import cpm_inputs as ci
from gpu_common import SMALL, need_gpu, pair

pytestmark = pytest.mark.gpu
TOL = 84 * 2.0 ** -53 * 1.95


def _wl(name):
    if name.startswith("torus"):  # odd spacing: ragged cell counts
        return ci.Workload("t", ci.torus(), 1 / 17.3, [ci.torus_meridian(0.3, 1.0, 0.4, ci.BC_DIR2)], 0.0, 1.0)
    return SMALL[name]()


@pytest.mark.parametrize("name", ["circle_dir1", "circle_dir2", "sphere_lat_dir2", "torus", "sphere_closed"])
@pytest.mark.parametrize("p", [3, 2])
def test_few_columns_match_oracle(oracle_mod, name, p):
    torch = need_gpu()
    w = _wl(name)
    band, ref = pair(oracle_mod, w, p=p)
    for nrhs in (1, 2, 3, 15):
        U = ci.random_vector(ref.N, seed=nrhs, nrhs=nrhs).reshape(ref.N, -1)
        Ug = torch.tensor(U if nrhs > 1 else U[:, 0], device="cuda")
        a = band.extend(Ug).cpu().numpy().reshape(ref.NS, -1)
        v = band.apply(0.0, 1.0, Ug).cpu().numpy().reshape(ref.N, -1)
        v32 = band.apply(0.0, 1.0, Ug.float()).cpu().numpy().reshape(ref.N, -1)
        for r in range(nrhs):
            assert np.max(np.abs(a[:, r] - ref.extend(U[:, r])[:ref.NS])) <= TOL * np.max(np.abs(U[:, r]))
            vr = ref.apply(0.0, 1.0, U[:, r])
            assert np.max(np.abs(v[:, r] - vr)) <= 1e-14 * np.max(np.abs(vr))
            assert np.max(np.abs(v32[:, r] - vr)) <= 2e-6 * np.max(np.abs(vr))


@pytest.mark.parametrize("scale", [2.0 ** -1060, 2.0 ** -950, 2.0 ** -600, 2.0 ** 600, 2.0 ** 1018])
def test_ends_of_the_exponent_range(oracle_mod, scale):
    """Scaled inputs give scaled outputs (absolute 64 denormals where they underflow)."""
    torch = need_gpu()
    w = SMALL["circle_dir2"]()
    band, ref = pair(oracle_mod, w)
    u = ci.random_vector(ref.N, seed=3)
    u[::7] *= 1e-9   # neighbours of very different size
    a = band.extend(torch.tensor(u * scale, device="cuda")).cpu().numpy()
    er = ref.extend(u)[:ref.NS] * scale
    assert np.max(np.abs(a - er)) <= TOL * scale + 64 * 2.0 ** -1074
    assert not np.any(band.extend(torch.zeros(ref.N, dtype=torch.float64, device="cuda")).cpu().numpy())


def test_infinities_and_nan_reach_the_same_rows(oracle_mod):
    torch = need_gpu()
    w = SMALL["sphere_closed"]()
    band, ref = pair(oracle_mod, w)
    for bad in (np.inf, -np.inf, np.nan):
        u = ci.random_vector(ref.N, seed=4)
        u[ref.N // 3] = bad
        with np.errstate(all="ignore"):
            er = ref.extend(u)[:ref.NS]
        a = band.extend(torch.tensor(u, device="cuda")).cpu().numpy()
        assert np.array_equal(np.isfinite(a), np.isfinite(er))
        ok = np.isfinite(er)
        assert np.max(np.abs(a[ok] - er[ok])) <= TOL


@pytest.mark.parametrize("name", ["circle_dir2", "sphere_lat_dir2", "torus"])
@pytest.mark.parametrize("p", [3, 2])
def test_batches_of_every_width_match_oracle(oracle_mod, name, p):
    """Column groups that end ragged, odd widths and more than 64 columns; columns
    of very different size, one of zeros and one holding an infinity."""
    torch = need_gpu()
    w = _wl(name)
    band, ref = pair(oracle_mod, w, p=p)
    A = ref.A(0.0, 1.0)
    for nrhs in (16, 31, 33, 34, 65, 66, 130):
        U = ci.random_vector(ref.N, seed=nrhs, nrhs=nrhs)
        VR = A @ U
        U32 = torch.tensor(U, device="cuda").float()
        V32 = band.apply(0.0, 1.0, U32).cpu().numpy()
        assert np.max(np.abs(V32 - VR)) <= 2e-6 * np.max(np.abs(VR))
        scale = np.ones(nrhs)
        scale[0], scale[1], scale[2] = 2.0 ** -800, 2.0 ** 800, 0.0
        Ug = torch.tensor(U * scale, device="cuda")
        Ug[ref.N // 2, 3] = float("inf")
        V = band.apply(0.0, 1.0, Ug).cpu().numpy()
        E = band.extend(Ug).cpu().numpy()
        for r in range(nrhs):
            if r == 3:
                assert not np.all(np.isfinite(V[:, r])) and np.any(np.isfinite(V[:, r]))
                continue
            assert np.max(np.abs(V[:, r] - VR[:, r] * scale[r])) <= 1e-14 * np.max(np.abs(VR[:, r])) * scale[r]
            er = ref.extend(U[:, r])[:ref.NS] * scale[r]
            assert np.max(np.abs(E[:, r] - er)) <= TOL * np.max(np.abs(U[:, r])) * scale[r]


def test_fp32_gather_takes_no_products_of_weights():
    """E u - u_i summed axis by axis over differences to u_i.  On rough fields of a closed sphere the product's
    rounding is 0.948 of that of the per-row gather, whose differences are to a common node (emulated operation by
    operation on this band; 0.995 where w_y w_z is rounded before it weighs a line).  The bar lies between."""
    torch = need_gpu()
    from paper_2305_04711_gb300.cpm import Band
    band = Band(ci.sphere(), 1 / 24).set_boundary([])
    u = torch.tensor(ci.random_vector(band.N, seed=5), device="cuda").float()
    v = band.apply(0.0, 1.0, u.double())
    err = []
    for mode in (0, 1):
        band.set_tune(1, torch.float32, single_mode=mode)
        err.append(float((band.apply(0.0, 1.0, u).double() - v).norm() / v.norm()))
    assert err[0] <= 0.97 * err[1], err


def test_fp32_of_smooth_columns_rounds_alike_in_every_width():
    """A smooth field's rounding is relative to local differences in every width: to u_i for a column alone (0.106
    of the result's own size in a model of random cells with linear fields), to a value from the middle of the
    stencil in batches (0.126; 0.35 to the stencil's first node).  The bar is a quarter above equality."""
    torch = need_gpu()
    from paper_2305_04711_gb300.cpm import Band
    band = Band(ci.sphere(), 1 / 12).set_boundary([])
    _, cp = band.export_band()
    gen = np.random.default_rng(6)
    U = torch.sin(cp @ torch.tensor(gen.normal(size=(3, 130)), device="cuda")
                  + torch.tensor(gen.uniform(0, 6, 130), device="cuda")).float()
    V = band.apply(0.0, 1.0, U[:, :8].double().contiguous())
    alone = torch.stack([band.apply(0.0, 1.0, U[:, r].contiguous()) for r in range(8)], 1)
    e1 = float((alone.double() - V).norm())
    for nrhs in (8, 16, 33, 64, 65, 66, 130):
        en = float((band.apply(0.0, 1.0, U[:, :nrhs].contiguous())[:, :8].double() - V).norm())
        assert en <= 1.25 * e1, (nrhs, en, e1)


@pytest.mark.parametrize("p", [3, 2])
def test_small_2d_batches_agree_with_columns_alone(p):
    """Both sides of the rule that takes small FP32 batches of a 2D band row by row, near curves too.  Two FP32
    products of the same column, each within 2e-6 of the largest entry."""
    torch = need_gpu()
    from paper_2305_04711_gb300.cpm import Band
    w = ci.config1(0.001, ci.BC_DIR2)
    band = Band(w.shape, w.h, p=p).set_boundary(w.curves)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(9)
    U = torch.randn((band.N, 35), generator=gen, device="cuda")
    alone = torch.stack([band.apply(0.3, 1.0, U[:, r].contiguous()) for r in range(35)], 1)
    top = float(alone.abs().max())
    for nrhs in (2, 5, 6, 7, 8, 15, 16, 33, 35):
        V = band.apply(0.3, 1.0, U[:, :nrhs].contiguous())
        assert float((V - alone[:, :nrhs]).abs().max()) <= 4e-6 * top, nrhs
    small = Band(w.shape, 0.01, p=p).set_boundary(w.curves)
    for nrhs in (33, 65, 129):
        U = torch.randn((small.N, nrhs), generator=gen, device="cuda")
        V = small.apply(0.3, 1.0, U)
        one = torch.stack([small.apply(0.3, 1.0, U[:, r].contiguous()) for r in range(nrhs)], 1)
        assert float((V - one).abs().max()) <= 4e-6 * float(one.abs().max()), nrhs
