"""u = j / rho is the correctly rounded quotient: on states whose sums are exact
in FP64 the device's moments, mean velocity and spectrum use numpy's quotients."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("nx,ny,k", [(16, 12, 5), (33, 7, 64)])
def test_velocity_is_the_rounded_quotient(gpu, prec, nx, ny, k):
    rng = np.random.default_rng(nx + k)
    # g = f - w: multiples of 2^-26 below 2^-6, sums of nine exact; f stored in
    # FP64 is the same with power-of-two weights in place of w.
    g = rng.integers(-(1 << 20), 1 << 20, (9, ny, nx, k)) * 2.0 ** -26
    if prec == "fp64":
        f = g + np.array([0.25] + [0.125] * 4 + [0.0625] * 4)[:, None, None, None]
        rho = f.sum(0)
    else:
        f = g + np.array([4 / 9] + [1 / 9] * 4 + [1 / 36] * 4)[:, None, None, None]
        rho = 1.0 + g.sum(0)
    u = (g[1] - g[2] + g[5] - g[6] + g[7] - g[8]) / rho
    v = (g[3] - g[4] + g[5] - g[6] - g[7] + g[8]) / rho
    p = gpu.LBM_FP64 if prec == "fp64" else gpu.LBM_MIXED
    with gpu.Ensemble(nx, ny, k, 0.55, 0.2, 0.0, p, f0=f) as e:
        r_gpu, u_gpu, v_gpu = e.moments_host()
    assert np.array_equal(r_gpu, rho) and np.array_equal(u_gpu, u) and np.array_equal(v_gpu, v)
    if prec == "fp64":
        with gpu.Ensemble(nx, ny, 1, 0.55, 0.2, 0.0, p, f0=np.ascontiguousarray(f[..., :1])) as e:
            um, vm = e.mean_velocity()
        assert np.array_equal(um, u[..., 0]) and np.array_equal(vm, v[..., 0])
