"""The one right-hand side transposed product by cell blocks and bricks (integer
sums in FP64): every stencil shape, values at the ends of the exponent range,
infinities, and a band wide enough that cells hold more than 64 rows.

Tolerances are the repository's for products: 1e-14 (FP64) and 2e-6 (FP32) of the
largest entry of A^T lambda."""
import numpy as np
import pytest
import scipy.sparse as sp

import cpm_inputs as ci
from gpu_common import SMALL, need_gpu

pytestmark = pytest.mark.gpu


def _pair(oracle_mod, name, p, r_band=-1.0):
    from paper_2305_04711_gb300.cpm import Band
    w = ci.Workload("t", ci.torus(), 1 / 17.3, [ci.torus_meridian(0.3, 1.0, 0.4, ci.BC_DIR2)], 0.0, 1.0) \
        if name == "torus" else SMALL[name]()
    band = Band(w.shape, w.h, p=p).set_boundary(w.curves)
    ref = oracle_mod.Oracle(w.shape, w.h, p=p).set_curves(w.curves)
    return band, ref


@pytest.mark.parametrize("name", ["circle_dir1", "circle_dir2", "sphere_lat_dir2", "torus", "sphere_closed"])
@pytest.mark.parametrize("p", [3, 2])
def test_transpose_matches_oracle(oracle_mod, name, p):
    torch = need_gpu()
    band, ref = _pair(oracle_mod, name, p)
    A = sp.csr_matrix(ref.A(0.0, 1.0))
    lam = ci.random_vector(ref.N, seed=7)
    y = band.apply(0.0, 1.0, torch.tensor(lam, device="cuda"), transpose=True).cpu().numpy()
    yr = A.T @ lam
    top = np.max(np.abs(yr))
    assert np.max(np.abs(y - yr)) <= 1e-14 * top
    y32 = band.apply(0.0, 1.0, torch.tensor(lam, device="cuda").float(), transpose=True).cpu().numpy()
    assert np.max(np.abs(y32 - yr)) <= 2e-6 * top
    for scale in (2.0 ** -900, 2.0 ** 900, 0.0):
        ys = band.apply(0.0, 1.0, torch.tensor(lam * scale, device="cuda"), transpose=True).cpu().numpy()
        assert np.max(np.abs(ys - yr * scale)) <= 1e-14 * top * scale


def test_columns_one_by_one_and_at_once_agree(oracle_mod):
    """Both sides of the rules on the number of columns, strided columns included."""
    torch = need_gpu()
    from paper_2305_04711_gb300.cpm import Band
    w = ci.config2(1 / 32, ci.BC_DIR2)
    band = Band(w.shape, w.h).set_boundary(w.curves)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(2)
    U = torch.randn((band.N, 9), generator=gen, dtype=torch.float64, device="cuda")
    one = torch.stack([band.apply(0.0, 1.0, U[:, r].contiguous(), transpose=True) for r in range(9)], 1)
    top = float(one.abs().max())
    for nrhs in (2, 4, 5, 8, 9):
        V = band.apply(0.0, 1.0, U[:, :nrhs].contiguous(), transpose=True)
        assert float((V - one[:, :nrhs]).abs().max()) <= 1e-14 * top
        V32 = band.apply(0.0, 1.0, U[:, :nrhs].float().contiguous(), transpose=True)
        assert float((V32.double() - one[:, :nrhs]).abs().max()) <= 2e-6 * top


def test_an_infinity_stays_in_its_columns(oracle_mod):
    torch = need_gpu()
    band, ref = _pair(oracle_mod, "sphere_closed", 3)
    A = sp.csr_matrix(ref.A(0.0, 1.0))
    lam = ci.random_vector(ref.N, seed=8)
    k = ref.N // 3
    lam[k] = 0.0
    yr = A.T @ lam
    lam[k] = np.inf
    y = band.apply(0.0, 1.0, torch.tensor(lam, device="cuda"), transpose=True).cpu().numpy()
    touched = np.zeros(ref.N, dtype=bool)
    touched[A[k].indices] = True
    # (cells share a block: columns of the same cells may become NaN, others may not)
    ok = np.isfinite(y)
    assert not np.any(ok[touched] & (np.abs(A[k].toarray()[0][touched]) > 1e-6))
    assert np.all(np.abs(y[ok] - yr[ok]) <= 1e-11 * np.max(np.abs(yr)))
    assert ok.sum() > 0.9 * ref.N


def test_cells_with_many_rows():
    """A tube of three radii around the unit circle: over 100 rows share each of its cells."""
    torch = need_gpu()
    from paper_2305_04711_gb300.cpm import Band
    band = Band(ci.circle2d(), 0.05, r_band=3.0).set_boundary([])
    gen = torch.Generator(device="cuda")
    gen.manual_seed(1)
    u = torch.randn(band.N, generator=gen, dtype=torch.float64, device="cuda")
    v = torch.randn(band.N, generator=gen, dtype=torch.float64, device="cuda")
    a = float(torch.dot(band.apply(0.0, 1.0, u), v))
    b = float(torch.dot(u, band.apply(0.0, 1.0, v, transpose=True)))
    # rounding of the two products, each entry of size <= 8/h^2 * 3 per unit of u
    assert abs(a - b) <= 1e-13 * band.N * 24 / 0.05 ** 2


@pytest.mark.parametrize("p", [3, 2])
@pytest.mark.parametrize("shape, h, r_band", [("circle", 0.0451, 0.7), ("circle", 0.05, 1.0), ("circle", 0.05, 3.0),
                                              ("sphere", 0.25, 3.0)])
def test_wide_bands_with_values_of_one_sign(oracle_mod, shape, h, r_band, p):
    """40 to 200 rows share a cell and all add up: the sums come as close to their integer limits as a
    field can bring them.  The reference adds the assembled entries up in extended precision."""
    torch = need_gpu()
    from paper_2305_04711_gb300.cpm import Band
    sh = ci.circle2d() if shape == "circle" else ci.sphere()
    band = Band(sh, h, r_band=r_band, p=p).set_boundary([])
    ref = oracle_mod.Oracle(sh, h, rband=r_band, p=p).set_curves([])
    A = sp.csc_matrix(ref.A(0.0, 1.0))
    gen = np.random.default_rng(3)
    for lam in (np.ones(ref.N), np.full(ref.N, -1.99), gen.uniform(1.0, 2.0, ref.N)):
        terms = A.data.astype(np.longdouble) * lam[A.indices]
        yr = np.array([terms[a:b].sum() for a, b in zip(A.indptr[:-1], A.indptr[1:])])
        y = band.apply(0.0, 1.0, torch.tensor(lam, device="cuda"), transpose=True).cpu().numpy()
        assert np.max(np.abs(y - yr)) <= 1e-14 * np.max(np.abs(yr))


@pytest.mark.parametrize("name", ["circle_dir1", "sphere_closed"])
@pytest.mark.parametrize("p", [3, 2])
def test_fp32_weights_keep_their_relative_accuracy(oracle_mod, name, p):
    """Single rows of A in FP32, entry by entry: a term rounds three weights, b twice, three products, at
    most six additions in its cell and six at its node, the diagonal and its scale: 24 roundings of 2^-24 of the
    terms' sizes (and 1e-14 of the largest for the FP64 weights themselves).  A weight near zero formed from a fraction rounded to FP32 is off by far more than its own 2^-24."""
    torch = need_gpu()
    band, ref = _pair(oracle_mod, name, p)
    A = sp.csr_matrix(ref.A(0.0, 1.0))
    size = abs(ref.Loff)[:, :ref.NS] @ abs(ref.E) + sp.eye(ref.NS, ref.N, format="csr") * abs(ref.diagL())
    far = np.flatnonzero(ref.near_c < 0)
    for i in far[:: len(far) // 24]:
        lam = np.zeros(ref.N)
        lam[i] = 1.0
        y = band.apply(0.0, 1.0, torch.tensor(lam, device="cuda").float(), transpose=True).cpu().numpy()
        err = np.abs(y - A[i].toarray()[0])
        assert np.all(err <= 24 * 2.0 ** -24 * size[i].toarray()[0] + 1e-14 * size[i].max())


@pytest.mark.parametrize("p, inv_h", [(3, 12), (3, 18), (2, 16), (2, 28), (2, 40)])
def test_few_columns_on_both_sides_of_their_rule(p, inv_h):
    """Bands around the row counts from which 2 to 9 columns go one by one (12k to 130k rows), near curves too."""
    torch = need_gpu()
    from paper_2305_04711_gb300.cpm import Band
    w = ci.config2(1 / inv_h, ci.BC_DIR2)
    band = Band(w.shape, w.h, p=p).set_boundary(w.curves)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(3)
    U = torch.randn((band.N, 9), generator=gen, dtype=torch.float64, device="cuda")
    one = torch.stack([band.apply(0.3, 1.0, U[:, r].contiguous(), transpose=True) for r in range(9)], 1)
    top = float(one.abs().max())
    for nrhs in range(2, 10):
        V = band.apply(0.3, 1.0, U[:, :nrhs].contiguous(), transpose=True)
        assert float((V - one[:, :nrhs]).abs().max()) <= 1e-14 * top, nrhs
        V32 = band.apply(0.3, 1.0, U[:, :nrhs].float().contiguous(), transpose=True)
        assert float((V32.double() - one[:, :nrhs]).abs().max()) <= 2e-6 * top, nrhs
