"""The double-binary32 Gram of the mixed analysis against FP64 products and
the FP64 oracle: odd numbers of grid points and of local scalars (the scratch
arrays behind them stay aligned), long local lists, points with few or no
observations, density, ensemble sizes around the kernels' widths."""
import numpy as np
import pytest

import oracle
from paper_2308_03972_gb300 import inputs
from _helpers import U_RMS, W_REST, norm_rel, turbulent_state

pytestmark = pytest.mark.gpu
TAU0, CS, MU = 0.55, 0.2, 6.16e-7
SIGMA = 0.1 * U_RMS


@pytest.mark.parametrize("nx,ny,k,nox,noy,d_cut,rho", [
    (20, 20, 16, 20, 20, 100.0, False),  # 400 points in range everywhere: two stages
    (27, 25, 5, 27, 25, 100.0, False),   # 675 points: three stages; 15 entries
    (23, 11, 9, 23, 11, 3.0, True),      # 253 grid points: the last block holds five
    (20, 20, 31, 20, 20, 100.0, False),  # 496 entries
    (20, 20, 32, 20, 20, 4.5, True),
    (18, 17, 33, 18, 17, 6.0, False),    # 561 entries: a second pass of 49
    (31, 26, 8, 6, 5, 1.6, False),       # some points see nothing
    (20, 13, 128, 20, 13, 100.0, False),  # 260 points, 8256 entries
])
def test_gram_matches_fp64_products_and_oracle(gpu, nx, ny, k, nox, noy, d_cut, rho):
    f = turbulent_state(oracle, nx, ny, k, seed=k + nox, pert=0.1)
    w = np.asarray(W_REST)[:, None, None, None]
    f = ((f - w).astype(np.float32).astype(np.float64)) + w
    ix, iy = inputs.uniform_obs_points(nx, ny, nox, noy)
    rng = np.random.default_rng(k)
    _, u, v = oracle.moments(f)
    yo = np.stack([u.mean(2)[iy, ix], v.mean(2)[iy, ix], np.ones(len(ix))], 1)
    sig = np.array([SIGMA, 1.5 * SIGMA, 1e-3])
    yo = yo + sig * rng.standard_normal(yo.shape)
    out = {}
    with gpu.Ensemble(nx, ny, k, TAU0, CS, MU, gpu.LBM_MIXED) as e:
        for mode in (gpu.LBM_PROD_DF32, gpu.LBM_PROD_FP64):
            e.set_f(f)
            e.set_products(mode)
            if rho:
                e.observe_rho(ix, iy, *np.ascontiguousarray(yo.T), *sig)
            else:
                e.observe(ix, iy, yo[:, 0].copy(), yo[:, 1].copy(), sig[0], sig[1])
            e.analyze(d_cut, 1.05)
            out[mode] = e.get_f()
        e.sync()
    # Binary32 storage of f - w (|f - w| < 0.05) separates the two.
    assert np.max(np.abs(out[gpu.LBM_PROD_DF32] - out[gpu.LBM_PROD_FP64])) / np.max(np.abs(f)) <= 2e-8
    nv = 3 if rho else 2
    pts = np.sort(rng.choice(nx * ny, 24, replace=False)).astype(np.int32)
    ref = oracle.letkf_analyze_vars(f, ix, iy, yo[:, :nv].copy(), list(sig[:nv]), d_cut, 1.05, points=pts)
    y, x = pts // nx, pts % nx
    # 5e-8 up to 32 members (the binary32 floor of the analysis), times sqrt(128 / 32).
    assert norm_rel(out[gpu.LBM_PROD_DF32][:, y, x, :], ref[:, y, x, :]) <= (5e-8 if k <= 32 else 1e-7)
