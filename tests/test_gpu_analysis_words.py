"""The mixed-precision analysis and the equilibrium give the same words for the
same inputs: row checksums against those of the plainest kernels (the Gram from
the observation rows in order, the refinement one column per lane with its FP64
corrections, every direction of the equilibrium by itself). Kernel (A) starts
from the Gram rounded to binary32, so one changed word there, or in the state
that the Gram is formed of, changes the basis and with it the roundings of the
point's whole transform."""
import os
import sys

import pytest

sys.path.insert(0, os.path.join(os.path.dirname(os.path.abspath(__file__)), "golden"))
import analysis_words  # noqa: E402

pytestmark = pytest.mark.gpu
EXPECTED = analysis_words.load(os.path.join(os.path.dirname(os.path.abspath(__file__)), "golden", "analysis_words.txt"))


@pytest.mark.parametrize("name", sorted(analysis_words.CASES) + list(analysis_words.EQUILIBRIA))
def test_words(gpu, name):
    got = analysis_words.rows(gpu, name)
    assert len(got) == len(EXPECTED[name])
    assert [i for i, (a, b) in enumerate(zip(got, EXPECTED[name])) if a != b] == []
