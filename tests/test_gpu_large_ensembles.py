"""Mixed-precision analyses in observation space of ensembles whose
perturbations do not fit shared memory beside the n x n matrices (n local
scalars, more members than that), against FP64."""
import numpy as np
import pytest

import oracle
from paper_2308_03972_gb300 import inputs
from _helpers import U_RMS, W_REST, norm_rel, turbulent_state
from _svd import svd_analysis

pytestmark = pytest.mark.gpu
SIGMA = 0.1 * U_RMS
BETA = 1.05


@pytest.mark.parametrize("k,nox,noy", [
    (200, 9, 7),                               # 126 scalars, staged
    (750, 9, 7), (751, 9, 7), (1000, 10, 6), (2044, 9, 7),  # 128 columns: staged up to 750 members
    (1463, 10, 5), (1464, 10, 5), (2044, 10, 5),            # 112: up to 1463
    (2044, 7, 6),                              # 96: the largest ensemble of the observation operator
])
def test_large_ensemble_matches_fp64(gpu, k, nox, noy):
    nx, ny, d_cut = nox, noy, 100.0
    f = turbulent_state(oracle, nx, ny, k, seed=k + nox, pert=0.1)
    w = np.asarray(W_REST)[:, None, None, None]
    f = ((f - w).astype(np.float32).astype(np.float64)) + w
    ix, iy = inputs.uniform_obs_points(nx, ny, nox, noy)
    rng = np.random.default_rng(k)
    _, u, v = oracle.moments(f)
    yu = u.mean(2)[iy, ix] + SIGMA * rng.standard_normal(len(ix))
    yv = v.mean(2)[iy, ix] + SIGMA * rng.standard_normal(len(ix))
    with gpu.Ensemble(nx, ny, k, 0.55, 0.2, 0.0, gpu.LBM_MIXED, f0=f) as e:
        e.observe(ix, iy, yu, yv, SIGMA, SIGMA)
        e.analyze(d_cut, BETA)
        got = e.get_f()
        e.sync()
    # 5e-8 of max |f| for binary32 sums up to 32 members, growing as their square root.
    tol = 5e-8 * np.sqrt(max(k, 32) / 32.0)
    for x, y in ((0, 0), (nx - 1, 0), (2, ny - 1), (nx // 2, ny // 2)):
        ref = svd_analysis(oracle, f, ix, iy, yu, yv, SIGMA, d_cut, BETA, x, y)
        assert norm_rel(got[:, y, x, :], ref) <= tol
