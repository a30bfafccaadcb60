"""Real couplings where b_t times the field is NaN: the rule is s' = +1 iff delta >= 0, so the spin is
-1.  An infinite b_t = fl32(beta_t c) meets the zero field of an isolated spin, or b_t = 0 the infinite
field of a bias beyond float32."""
import numpy as np
import pytest

from gpu_helpers import pim

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("case", ["infinite_slope", "infinite_bias"])
@pytest.mark.parametrize("n,R", [(17, 5), (64, 32), (100, 130), (256, 33), (300, 65), (700, 129)])
def test_nan_is_down(n, R, case):
    P = pim()
    g = np.random.default_rng(n)
    J = np.triu(g.standard_normal((n, n)), 1)
    nan = np.arange(n) % 5 == 3  # the spins whose product is NaN
    h = np.zeros(n)
    if case == "infinite_slope":
        J[nan, :] = J[:, nan] = 0.0
        c, beta = 1e39, np.array([1.0, 3.0], np.float32)
    else:
        h[nan] = 1e39
        c, beta = 1.0, np.zeros(2, np.float32)
    hd = P.pim_create(J + J.T, h if h.any() else None, c)
    try:
        P.pim_set_schedule(hd, beta, np.full(2, 0.25, np.float32), 0.5)
        for sweeps in (1, 2):
            P.pim_anneal(hd, R, sweeps, 3, init_spins=np.ones((R, n), np.int8))
            final = P.pim_final_state(hd, n)
            assert np.all(final[:, nan] == -1)
            assert np.any(final[:, ~nan] == 1)
    finally:
        P.pim_destroy(hd)
