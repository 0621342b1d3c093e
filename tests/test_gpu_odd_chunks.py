"""Mixed analyses in chunks of an odd number of grid points, alternating
between the two scratch buffers: the second starts aligned whatever the first
one's size."""
import numpy as np
import pytest

import oracle
from paper_2308_03972_gb300 import inputs
from _helpers import U_RMS, W_REST, norm_rel, turbulent_state

pytestmark = pytest.mark.gpu
SIGMA = 0.1 * U_RMS


@pytest.mark.parametrize("k", [104, 122])  # 154,436 and 187,124 bytes a point: chunks of 2,607 and 2,151
def test_odd_chunks_match_oracle(gpu, k):
    nx = ny = 64
    bytes_per_point = 128 * 128 * 4 + 128 * 12 + 4 + k * (k + 1) * 8  # basis, list of 128, count, Gram and b
    chunk = (384 << 20) // bytes_per_point
    assert chunk % 2 == 1 and chunk < nx * ny
    f = turbulent_state(oracle, nx, ny, k, seed=k, pert=0.1)
    w = np.asarray(W_REST)[:, None, None, None]
    f = ((f - w).astype(np.float32).astype(np.float64)) + w
    ix, iy = inputs.uniform_obs_points(nx, ny, 8, 8)
    rng = np.random.default_rng(k)
    _, u, v = oracle.moments(f)
    yu = u.mean(2)[iy, ix] + SIGMA * rng.standard_normal(len(ix))
    yv = v.mean(2)[iy, ix] + SIGMA * rng.standard_normal(len(ix))
    with gpu.Ensemble(nx, ny, k, 0.55, 0.2, 0.0, gpu.LBM_MIXED, f0=f) as e:
        e.observe(ix, iy, yu, yv, SIGMA, SIGMA)
        e.analyze(100.0, 1.05)
        got = e.get_f()
        e.sync()
    pts = np.sort(rng.choice(nx * ny, 48, replace=False)).astype(np.int32)
    ref = oracle.letkf_analyze(f, ix, iy, yu, yv, SIGMA, SIGMA, 100.0, 1.05, points=pts)
    y, x = pts // nx, pts % nx
    # 5e-8 of max |f| up to 32 members, times sqrt(128 / 32).
    assert norm_rel(got[:, y, x, :], ref[:, y, x, :]) <= 1e-7
