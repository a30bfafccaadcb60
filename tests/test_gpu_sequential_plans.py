"""Sequential kernel: every layout its plan picks (4, 8, 16 or 32 field registers per lane or fields
in shared memory; J in shared memory or not; table in shared memory or not; one or several replicas
per block) gives the oracle's run, at the edges of the layouts."""
import numpy as np
import pytest

import oracle
from workloads import Instance, eta_power, linear_beta, random_spins, sk_pm1

from gpu_helpers import assert_same, collect, pim

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,R,scale", [
    (1, 3, 1), (31, 5, 1), (32, 5, 16), (33, 160, 1), (128, 4, 1), (129, 4, 1), (256, 310, 1),
    (257, 3, 1), (470, 3, 1), (512, 3, 16), (513, 3, 1), (1024, 2, 1), (1025, 2, 4)])
def test_layouts(n, R, scale):
    P = pim()
    T = 3 if n < 300 else 2
    J = (sk_pm1(n, 2).J.astype(np.int32) * scale).astype(np.int8)
    h = np.random.default_rng(n).integers(-3, 4, n).astype(np.int32)
    inst = Instance("sk", n, J, h, 1.0 / (scale * np.sqrt(n)), 2)
    beta = linear_beta(T)
    eta = eta_power(beta)
    init = random_spins(n, R, seed=1) if n % 2 else None
    hd = P.pim_create(inst.J, h, inst.c)
    try:
        P.pim_set_schedule(hd, beta, eta, 0.2, "uniform")
        P.pim_anneal_sequential(hd, R, T, 6, init_spins=init, target=-0.3 * n * scale)
        got = collect(hd, n)
    finally:
        P.pim_destroy(hd)
    want = oracle.anneal_sequential_sweeps(inst.J, h, inst.c, beta, eta, 0.2, replicas=R, seed=6, noise="uniform",
                                           target=-0.3 * n * scale, init=init)
    assert_same(got, want, label=f"n={n}")
