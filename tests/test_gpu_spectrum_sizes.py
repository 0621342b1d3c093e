"""Energy spectrum of long rows and columns (few members per block, large
prime factors), up to the largest lattices that the diagnostic takes, with
fewer shells than the lattice has, against the FP64 oracle."""
import numpy as np
import pytest

import oracle
from _helpers import U_RMS

pytestmark = pytest.mark.gpu


def _ensemble(gpu, nx, ny, k, seed):
    rng = np.random.default_rng(seed)
    u, v = (U_RMS * rng.standard_normal((2, ny, nx, k)))
    f = oracle.set_equilibrium(np.ones_like(u), u, v)
    return f, gpu.Ensemble(nx, ny, k, 0.55, 0.2, 0.0, gpu.LBM_FP64, f0=f)


@pytest.mark.parametrize("nx,ny,k,nsh", [
    (4, 4000, 2, 100),    # 56 * 4000 + 8 * 100 bytes: within 227 KB
    (2, 4136, 1, 104),    # the longest column with 104 shells
    (3, 3875, 3, 900),
    (1614, 6, 2, 808),    # the longest row: 2 * 3 * 269
    (1613, 4, 1, 50),     # a prime
    (500, 428, 9, 200),   # four members per block
    (16, 1024, 5, 513),
])
def test_long_rows_and_columns_match_oracle(gpu, nx, ny, k, nsh):
    f, e = _ensemble(gpu, nx, ny, k, nx + ny)
    with e:
        got = e.energy_spectrum(np.zeros(nsh))
        e.sync()
    ref = oracle.energy_spectrum(f)[:nsh]
    # White noise: shells of similar size. The bound of the other lattices.
    assert np.max(np.abs(got[:len(ref)] - ref)) <= 1e-12 * ref.max()


@pytest.mark.parametrize("nx,ny,nsh", [(2, 4136, 105), (1615, 4, 8)])
def test_larger_lattices_are_refused(gpu, nx, ny, nsh):
    _, e = _ensemble(gpu, nx, ny, 1, 3)
    with e:
        with pytest.raises(gpu.LbmError) as err:
            e.energy_spectrum(np.zeros(nsh))
        assert err.value.code == gpu.LBM_EINVAL
