"""Sequential kernel with more replicas than one wave of blocks: the plan leaves the tables out of shared
memory or takes smaller blocks, and every replica's run stays what it is alone and in the oracle; sizes
around the tails of a row of couplings."""
import numpy as np
import pytest

import oracle
from workloads import Instance, eta_power, linear_beta, sk_pm1

from gpu_helpers import assert_same, collect, pim

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,R", [(513, 1400), (640, 700), (641, 3000), (769, 1400), (896, 400), (897, 1400), (1024, 4000), (1025, 1400), (1280, 2500), (1281, 1000), (2049, 1300)])
def test_replica_count_changes_nothing(n, R):
    P = pim()
    T = 2
    h = np.random.default_rng(n).integers(-3, 4, n).astype(np.int32)
    inst = Instance("sk", n, sk_pm1(n, 4).J, h, 1.0 / np.sqrt(n), 4)
    beta = linear_beta(T)
    eta = eta_power(beta)
    hd = P.pim_create(inst.J, h, inst.c)
    try:
        P.pim_set_schedule(hd, beta, eta, 0.2, "uniform")
        runs = []
        for replicas in (2, 300, R):
            P.pim_anneal_sequential(hd, replicas, T, 6, target=-0.3 * n)
            runs.append(collect(hd, n))
    finally:
        P.pim_destroy(hd)
    assert_same(runs[0], oracle.anneal_sequential_sweeps(inst.J, h, inst.c, beta, eta, 0.2, replicas=2, seed=6,
                                                         noise="uniform", target=-0.3 * n))
    assert_same({k: v[:2] for k, v in runs[1].items()}, runs[0])
    assert_same({k: v[:300] for k, v in runs[2].items()}, runs[1])
