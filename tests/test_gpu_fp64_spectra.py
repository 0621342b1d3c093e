"""FP64 analyses whose local problems have wide spectra (small observation
errors), in observation space: what the eigensolve leaves off the diagonal
grows with ||A||_F and enters the matrix functions to second order."""
import numpy as np
import pytest

import oracle
from paper_2308_03972_gb300 import inputs
from _helpers import TOL_FP64, U_RMS, norm_rel, turbulent_state
from _svd import svd_analysis

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("run_len", [0, 8])
@pytest.mark.parametrize("nx,ny,k,nox,noy,d_cut", [(32, 24, 64, 4, 4, 16.0), (24, 20, 48, 4, 3, 100.0), (24, 20, 64, 6, 5, 100.0)])
@pytest.mark.parametrize("shrink", [3.0, 0.1, 0.02, 0.005])
def test_wide_spectra_match_oracle(gpu, nx, ny, k, nox, noy, d_cut, shrink, run_len):
    sigma = 0.1 * shrink * U_RMS
    f = turbulent_state(oracle, nx, ny, k, seed=k + nox, pert=0.1)
    ix, iy = inputs.uniform_obs_points(nx, ny, nox, noy)
    rng = np.random.default_rng(k)
    _, u, v = oracle.moments(f)
    yu = u.mean(2)[iy, ix] + sigma * rng.standard_normal(len(ix))
    yv = v.mean(2)[iy, ix] + sigma * rng.standard_normal(len(ix))
    with gpu.Ensemble(nx, ny, k, 0.55, 0.2, 0.0, gpu.LBM_FP64, f0=f) as e:
        e.set_run_length(run_len)
        e.observe(ix, iy, yu, yv, sigma, sigma)
        e.analyze(d_cut, 1.05)
        got = e.get_f()
        e.sync()
    Y = np.stack([u[iy, ix], v[iy, ix]], 1).reshape(-1, k)
    Y = (Y - Y.mean(1, keepdims=True)) / sigma
    spread = 1.05 * np.linalg.norm(Y @ Y.T) / (k - 1)  # ||A||_F / a at unit weights
    assert shrink > 1.0 or spread > 100.0
    # The FP64 bound, the rounding of eigenvalues of that size relative to a
    # (16 units), and the cube of what the eigensolve may leave.
    tol = TOL_FP64 + 16 * np.finfo(float).eps * spread + (3e-8 * spread) ** 3
    for p in rng.choice(nx * ny, 48, replace=False):
        x, y = int(p % nx), int(p // nx)
        ref = svd_analysis(oracle, f, ix, iy, yu, yv, sigma, d_cut, 1.05, x, y)
        assert norm_rel(got[:, y, x, :], ref) <= tol
