"""Mixed-precision analyses with 33..128 local scalars or members (the
tournament-position Jacobi and the tiled refinement) against the FP64 oracle:
tile edges of every size class in both forms, mixtures of both forms and of
empty points on one lattice, every Gram arithmetic, and wide spectra."""
import numpy as np
import pytest

import oracle
from paper_2308_03972_gb300 import inputs
from _helpers import U_RMS, W_REST, norm_rel, turbulent_state

pytestmark = pytest.mark.gpu
TAU0, CS, MU = 0.55, 0.2, 6.16e-7
SIGMA = 0.1 * U_RMS
# Binary32 storage of f - w (|f - w| <= 0.05) and binary32 sums over the
# members: 5e-8 of max |f| up to 32 terms, times sqrt(128 / 32) at 128.
TOL = 1e-7


def _check(gpu, nx, ny, k, nox, noy, d_cut, sigma=SIGMA, tol=TOL, products=None, rho=False, spacing=None):
    f = turbulent_state(oracle, nx, ny, k, seed=k + nox, pert=0.1)
    w = np.asarray(W_REST)[:, None, None, None]
    f = ((f - w).astype(np.float32).astype(np.float64)) + w
    ix, iy = inputs.uniform_obs_points(nx, ny, nox, noy)
    if spacing:
        ix, iy = inputs.uniform_obs_points(spacing * nox, spacing * noy, nox, noy)
    rng = np.random.default_rng(k)
    _, u, v = oracle.moments(f)
    yu = u.mean(2)[iy, ix] + sigma * rng.standard_normal(len(ix))
    yv = v.mean(2)[iy, ix] + sigma * rng.standard_normal(len(ix))
    yr = 1.0 + 1e-3 * rng.standard_normal(len(ix))
    with gpu.Ensemble(nx, ny, k, TAU0, CS, MU, gpu.LBM_MIXED, f0=f) as e:
        if products is not None:
            e.set_products(products)
        e.sweep_stats(True)
        if rho:
            e.observe_rho(ix, iy, yu, yv, yr, sigma, sigma, 1e-3)
        else:
            e.observe(ix, iy, yu, yv, sigma, sigma)
        e.analyze(d_cut, 1.05)
        got = e.get_f()
        hist = e.sweep_stats(False, read=True)
        e.sync()
    pts = np.sort(rng.choice(nx * ny, min(24, nx * ny), replace=False)).astype(np.int32)
    if rho:
        ref = oracle.letkf_analyze_vars(f, ix, iy, np.stack([yu, yv, yr], 1), [sigma, sigma, 1e-3], d_cut, 1.05,
                                        points=pts)
    else:
        ref = oracle.letkf_analyze(f, ix, iy, yu, yv, sigma, sigma, d_cut, 1.05, points=pts)
    y, x = pts // nx, pts % nx
    assert np.all(np.isfinite(got))
    err = norm_rel(got[:, y, x, :], ref[:, y, x, :])
    assert err <= tol, err
    return hist


@pytest.mark.parametrize("k", [33, 47, 48, 49, 63, 64, 65, 79, 80, 81, 96, 97, 111, 112, 113, 127, 128])
def test_ensemble_space_sizes(gpu, k):
    hist = _check(gpu, 16, 10, k, 16, 10, 40.0)  # 320 scalars everywhere
    assert int(hist.sum()) == 160


@pytest.mark.parametrize("k,nox,noy", [(41, 5, 4), (64, 9, 2), (65, 8, 4), (100, 7, 7), (128, 9, 7), (128, 8, 6),
                                       (127, 6, 5), (128, 9, 2)])
def test_observation_space_sizes(gpu, k, nox, noy):
    """All points in range: p = 2 nox noy < k scalars at every grid point."""
    assert 32 < 2 * nox * noy < k
    hist = _check(gpu, 4 * nox, 4 * noy, k, nox, noy, 100.0)
    assert int(hist.sum()) == 16 * nox * noy


@pytest.mark.parametrize("k,d_cut", [(40, 3.5), (64, 4.0), (90, 5.5)])
def test_mixed_forms_and_empty_points(gpu, k, d_cut):
    """Observation points on every cell of one corner: local counts from none
    to above k across one lattice."""
    hist = _check(gpu, 31, 26, k, 10, 9, d_cut, spacing=1)
    assert 0 < int(hist.sum()) < 31 * 26


@pytest.mark.parametrize("name", ["FP64", "FP32", "TF32", "BF16"])
def test_gram_arithmetic(gpu, name):
    tol = {"FP64": TOL, "FP32": 1e-6, "TF32": 2e-4, "BF16": 2e-3}[name]
    _check(gpu, 16, 10, 64, 16, 10, 6.0, tol=tol, products=getattr(gpu, "LBM_PROD_" + name))


def test_density_observations(gpu):
    _check(gpu, 20, 18, 50, 10, 9, 4.0, rho=True)


@pytest.mark.parametrize("shrink", [0.3, 0.1, 0.02])
@pytest.mark.parametrize("k,nox,noy", [(64, 16, 10), (128, 9, 7)])
def test_wide_spectra(gpu, k, nox, noy, shrink):
    """Smaller observation errors widen the spectrum by 1 / shrink^2. The
    general mixed-precision bound."""
    hist = _check(gpu, 16 if nox == 16 else 18, 10 if nox == 16 else 14, k, nox, noy, 100.0, sigma=shrink * SIGMA,
                  tol=1e-6)
    assert int(hist.sum()) == (160 if nox == 16 else 252)
