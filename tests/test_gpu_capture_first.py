"""A context's first analysis and first diagnostic inside a stream capture:
what needs no buffers beyond those of the observation step is captured, and
the replayed graph gives what plain calls give."""
import numpy as np
import pytest

import oracle
from paper_2308_03972_gb300 import inputs
from _helpers import U_RMS, turbulent_state

pytestmark = pytest.mark.gpu
SIGMA = 0.1 * U_RMS


@pytest.mark.parametrize("k,run_len", [(24, 0), (8, 8)])  # observation space, cold; ensemble space
def test_first_fp64_analysis_in_a_capture(gpu, k, run_len):
    import torch

    nx, ny = 24, 20
    f = turbulent_state(oracle, nx, ny, k, seed=5)
    ix, iy = inputs.uniform_obs_points(nx, ny, 4, 4)
    yu, yv = f[1, iy, ix, 0] * 0.1, f[2, iy, ix, 0] * 0.1
    out = []
    s = torch.cuda.Stream()
    for captured in (False, True):
        with torch.cuda.stream(s):
            with gpu.Ensemble(nx, ny, k, 0.55, 0.2, 0.0, gpu.LBM_FP64, f0=f) as e:
                e.set_run_length(run_len)
                e.observe(ix, iy, yu, yv, SIGMA, SIGMA)
                if captured:
                    s.synchronize()
                    g = torch.cuda.CUDAGraph()
                    with torch.cuda.graph(g, stream=s):
                        e.analyze(6.0, 1.05)
                    g.replay()
                else:
                    e.analyze(6.0, 1.05)
                out.append(e.get_f())
                e.sync()
    assert np.array_equal(out[0], out[1])


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
def test_first_spectrum_in_a_capture(gpu, prec):
    import torch

    nx, ny, k = 40, 36, 9
    f = turbulent_state(oracle, nx, ny, k, seed=6)
    p = gpu.LBM_FP64 if prec == "fp64" else gpu.LBM_MIXED
    nsh = gpu.spectrum_shells(nx, ny)
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        with gpu.Ensemble(nx, ny, k, 0.55, 0.2, 0.0, p, f0=f) as e:
            E = torch.zeros(nsh, dtype=torch.float64, device="cuda")
            s.synchronize()
            g = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g, stream=s):
                e.energy_spectrum(E)
            for _ in range(2):
                E.zero_()
                g.replay()
            s.synchronize()
            got = E.cpu().numpy()
            assert np.array_equal(got, e.energy_spectrum())
            del g
