"""FP64 analysis of single grid points, for ensembles and spectra beyond the
oracle's eigensolver."""
import numpy as np


def svd_analysis(oracle, f, ix, iy, yo_u, yo_v, sigma, d_cut, beta, x, y):
    """LETKF analysis of grid point (x, y) in FP64 through the singular values
    of Yh [p][k] (C = a I + Yh^T Yh). Returns [9][k]."""
    ny, nx, k = f.shape[1:]
    _, u, v = oracle.moments(f)
    Y = np.stack([u[iy, ix], v[iy, ix]], 1).reshape(-1, k)
    d = np.stack([yo_u, yo_v], 1).ravel() - Y.mean(1)
    idx, r = oracle.local_obs(nx, ny, x, y, ix, iy, sigma, sigma, d_cut)
    lw = np.sqrt(r)
    Yh = lw[:, None] * (Y - Y.mean(1, keepdims=True))[idx]
    a = (k - 1) / beta
    U, s, Vt = np.linalg.svd(Yh, full_matrices=False)
    wbar = Vt.T @ (s / (a + s * s) * (U.T @ (lw * d[idx])))
    X = f[:, y, x, :]
    xm = X.mean(1, keepdims=True)
    dX = X - xm
    root = dX / np.sqrt(a) + (dX @ Vt.T) * (1.0 / np.sqrt(a + s * s) - 1.0 / np.sqrt(a)) @ Vt
    return xm + (dX @ wbar)[:, None] + np.sqrt(k - 1.0) * root
