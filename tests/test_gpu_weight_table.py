"""Localisation weights from the table by squared distance and, where the
table would be too long, evaluated in the kernels: both against the FP64
oracle, in every analysis kernel that reads them."""
import numpy as np
import pytest

import oracle
from paper_2308_03972_gb300 import inputs
from _helpers import TOL_FP64, U_RMS, norm_rel, turbulent_state

pytestmark = pytest.mark.gpu
SIGMA = 0.1 * U_RMS


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("nx,ny,k,nox,noy,d_cut", [
    (1100, 8, 4, 20, 1, 300.0),   # 361,201 squared distances within reach: evaluated
    (1100, 8, 4, 20, 1, 250.0),   # 251,001: from the table, which the lattice's own 302,516 would not fit
    (1100, 8, 48, 11, 1, 255.4),  # the last d_cut below 2^18 entries; p < k, runs
    (1100, 8, 48, 11, 1, 255.6),  # the first above
    (21, 18, 24, 5, 4, 3.3),      # the whole lattice's distances, some points see nothing
    (8, 40, 6, 1, 8, 100.0),      # distances up to 416
])
def test_weights_match_oracle(gpu, prec, nx, ny, k, nox, noy, d_cut):
    f = turbulent_state(oracle, nx, ny, k, seed=nx + k, pert=0.1)
    ix, iy = inputs.uniform_obs_points(nx, ny, nox, noy)
    rng = np.random.default_rng(k)
    _, u, v = oracle.moments(f)
    yu = u.mean(2)[iy, ix] + SIGMA * rng.standard_normal(len(ix))
    yv = v.mean(2)[iy, ix] + SIGMA * rng.standard_normal(len(ix))
    p = gpu.LBM_FP64 if prec == "fp64" else gpu.LBM_MIXED
    with gpu.Ensemble(nx, ny, k, 0.55, 0.2, 6.16e-7, p, f0=f) as e:
        e.observe(ix, iy, yu, yv, SIGMA, SIGMA)
        e.analyze(d_cut, 1.05)
        got = e.get_f()
        e.sync()
    pts = np.sort(rng.choice(nx * ny, min(40, nx * ny), replace=False)).astype(np.int32)
    ref = oracle.letkf_analyze(f, ix, iy, yu, yv, SIGMA, SIGMA, d_cut, 1.05, points=pts)
    y, x = pts // nx, pts % nx
    # The bounds of both precisions everywhere else in these tests.
    assert norm_rel(got[:, y, x, :], ref[:, y, x, :]) <= (TOL_FP64 if prec == "fp64" else 1e-6)
