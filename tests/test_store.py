"""Reading a state back into complex float: values that are not finite come back as
they were loaded."""
import numpy as np
import pytest

from paper_1906_06327_gb300.rotgp import Solver

pytestmark = pytest.mark.gpu


def test_infinities_come_back_as_loaded():
    n = (40, 30)
    psi = np.zeros((31, 41), np.complex64)
    psi[10, 10] = 1.0
    psi[11, 12] = complex(np.inf, 2.0)
    psi[13, 14] = complex(-np.inf, np.nan)
    s = Solver(n, (0.3, 0.3), dt=1e-3, g=1.0)
    s.set_psi(psi)
    got = s.get_psi(fp64=False)
    assert np.array_equal(got.view(np.float32), psi.view(np.float32), equal_nan=True)

