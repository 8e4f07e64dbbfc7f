"""What Theta takes: sequences, arrays of any shape with p entries, and what NumPy makes doubles of."""
from fractions import Fraction

import numpy as np
import pytest

import paper_2008_07437_gb300 as geo


@pytest.mark.parametrize("s2,nu", [
    ((1.0, 2.0), (0.5, 1.0)),
    ([1, 2], [Fraction(1, 2), 1]),
    (np.array([1.0, 2.0], dtype=np.float32), np.array([0.5, 1.0])[::1]),
    (np.array([[1.0], [2.0]]), np.array([[0.5], [1.0]])),
    (np.arange(4.0)[1::1][:2], np.array([0.5, 9.0, 1.0])[::2]),
])
def test_entries(s2, nu):
    th, keep = geo.Theta(s2, 0.1, nu, 0.25).to_c()
    assert th.p == 2 and th.a == 0.1
    assert [th.sigma2[0], th.sigma2[1]] == [1.0, 2.0]
    assert [th.nu[0], th.nu[1]] == [0.5, 1.0]
    assert [th.beta[k] for k in range(4)] == [1.0, 0.25, 0.25, 1.0]
