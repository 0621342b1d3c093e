"""Words of mixed-precision analyses and of the equilibrium: a checksum of every
lattice row's result (stored binary32 posteriors), for inputs that are the same
to the bit on any machine (uniform random numbers and sums of them, no libm). A
kernel that sums in another order, or in other formats, changes some of them.

``python analysis_words.py FILE`` writes them for the package on ``sys.path``.
"""
from __future__ import annotations

import sys
import zlib

import numpy as np

W = np.array([4 / 9] + [1 / 9] * 4 + [1 / 36] * 4)
SIGMA = 0.003

# name: nx, ny, members, observation lattice, d_cut, run length, Gram products, density observed
CASES = {
    "dense_16": (256, 256, 16, (32, 32), 32.0, 8, "DF32", False),
    "dense_32": (256, 128, 32, (16, 8), 32.0, 8, "DF32", False),
    "density_24": (96, 64, 24, (24, 16), 9.0, 8, "DF32", True),
    "dense_64": (128, 64, 64, (16, 8), 24.0, 8, "DF32", False),
    "fp64_products_40": (64, 48, 40, (16, 12), 9.0, 8, "FP64", False),
    "members_128": (48, 32, 128, (12, 8), 40.0, 8, "DF32", False),
    "scalars_32": (96, 96, 64, (12, 12), 8.5, 0, "DF32", False),
    "scalars_32_of_128": (96, 64, 128, (12, 8), 8.5, 0, "DF32", False),
    "scalars_60": (96, 96, 96, (12, 12), 12.0, 8, "DF32", False),
    "scalars_100": (96, 96, 128, (12, 12), 16.0, 8, "DF32", False),
}


def posterior(binding, name):
    """The stored binary32 state g = f - w after one analysis, [ny][nx][9][k]."""
    import torch

    nx, ny, k, (nox, noy), d_cut, run_len, products, rho = CASES[name]
    rng = np.random.Generator(np.random.PCG64(nx * 1000 + k))
    g = (rng.random((9, ny, nx, 1), dtype=np.float32) - np.float32(0.5)) * np.float32(2.0 ** -6)
    g = g + (rng.random((9, ny, nx, k), dtype=np.float32) - np.float32(0.5)) * np.float32(2.0 ** -7)
    w = W[:, None, None, None]
    ix, iy = np.meshgrid(np.arange(nox) * (nx // nox), np.arange(noy) * (ny // noy))
    ix, iy = ix.ravel().astype(np.int32), iy.ravel().astype(np.int32)
    yu, yv, yr = ((rng.random((3, len(ix))) - 0.5) * 0.02)
    f = torch.as_tensor(g.astype(np.float64) * w * 9 + w).cuda()
    with binding.Ensemble(nx, ny, k, 0.55, 0.2, 0.0, binding.LBM_MIXED) as e:
        e.set_f(f)
        e.set_run_length(run_len)
        e.set_products(getattr(binding, "LBM_PROD_" + products))
        if rho:
            e.observe_rho(ix, iy, yu, yv, 1.0 + yr, SIGMA, SIGMA, SIGMA)
        else:
            e.observe(ix, iy, yu, yv, SIGMA, SIGMA)
        e.analyze(d_cut, 1.05)
        out = e.get_f()
        e.sync()
    return np.ascontiguousarray((out - w).astype(np.float32).transpose(1, 2, 0, 3))


EQUILIBRIA = ("equilibrium_fp64", "equilibrium_fp64_rho", "equilibrium_mixed", "equilibrium_mixed_rho")


def equilibrium(binding, name):
    """f after set_equilibrium, [ny][nx][9][k]; its first row at rest."""
    nx, ny, k = 250, 41, 24
    rng = np.random.Generator(np.random.PCG64(7))
    u, v = (rng.random((2, ny, nx, k)) - 0.5) * 0.2
    u[0] = v[0] = 0.0
    rho = 1.0 + (rng.random((ny, nx, k)) - 0.5) * 0.1 if name.endswith("_rho") else None
    prec = binding.LBM_FP64 if "fp64" in name else binding.LBM_MIXED
    with binding.Ensemble(nx, ny, k, 0.55, 0.2, 0.0, prec) as e:
        e.set_equilibrium(rho, u, v)
        out = e.get_f()
        e.sync()
    return np.ascontiguousarray(out.transpose(1, 2, 0, 3))


def rows(binding, name):
    if name in EQUILIBRIA:
        return ["%08x" % zlib.crc32(r.tobytes()) for r in equilibrium(binding, name)]
    return ["%08x" % zlib.crc32(r.tobytes()) for r in posterior(binding, name)]


def load(path):
    with open(path) as fh:
        return {t[0]: t[1:] for t in (line.split() for line in fh) if t}


if __name__ == "__main__":
    from paper_2308_03972_gb300 import binding

    with open(sys.argv[1], "w") as fh:
        for name in (*CASES, *EQUILIBRIA):
            fh.write(" ".join([name] + rows(binding, name)) + "\n")
