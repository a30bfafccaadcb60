"""Fused integer kernels: a replica's run does not depend on the kernel and the tile height that
the replica count selects (few tiles: the latency kernel with 32, 64 or 128 replicas per CTA; many:
the throughput kernel, without and with its queue), at the edges of their chunks and tiles, and
equals the oracle's."""
import numpy as np
import pytest

import oracle
from workloads import Instance, eta_power, linear_beta, maxcut_er, random_spins, sk_pm1

from gpu_helpers import assert_same, collect, oracle_run, pim

pytestmark = pytest.mark.gpu

COUNTS = (20, 4000, 9600, 19000, 38000, 60000)  # replicas: about 1, 30, 75, 150, 300, 470 tiles of 128


def _instance(n, field):
    inst = (sk_pm1 if n % 2 else maxcut_er)(n, 3)
    if field:
        h = np.random.default_rng(n).integers(-5, 6, n).astype(np.int32)
        inst = Instance(inst.kind, n, inst.J, h, inst.c, 3)
    return inst


@pytest.mark.parametrize("field", [False, True])
@pytest.mark.parametrize("n", [1, 16, 17, 64, 65, 100, 128, 129, 200, 255, 256])
def test_replicas_agree_across_kernels(n, field):
    P = pim()
    inst = _instance(n, field)
    T = 9
    beta = linear_beta(T)
    kw = dict(noise="uniform", act="lut", lut_levels=6) if n % 3 == 0 else {}
    hd = P.pim_create(inst.J, inst.h if field else None, inst.c)
    try:
        P.pim_set_schedule(hd, beta, eta_power(beta), 0.6, **kw)
        first = oracle_run(inst, beta, eta_power(beta), 0.6, replicas=COUNTS[0], seed=8, target=-n / 2, **kw)
        for R in COUNTS:
            P.pim_anneal(hd, R, T, 8, target=-n / 2)
            got = collect(hd, n)
            assert_same({k: v[:COUNTS[0]] for k, v in got.items()}, first, label=f"R={R}")
            if R == COUNTS[1]:
                more = got
            elif R > COUNTS[1]:
                for k in more:
                    assert np.array_equal(got[k][:COUNTS[1]], more[k]), (R, k)
    finally:
        P.pim_destroy(hd)


@pytest.mark.parametrize("n,R,field", [(40, 33, True), (128, 64, False), (200, 129, False), (256, 31, True)])
def test_resume_and_given_spins(n, R, field):
    """A split run with given spins equals the oracle's whole run; no sweeps gives the energy only."""
    P = pim()
    inst = _instance(n, field)
    T = 11
    beta = linear_beta(T)
    init = random_spins(n, R, seed=5)
    hd = P.pim_create(inst.J, inst.h if field else None, inst.c)
    try:
        P.pim_set_schedule(hd, beta, eta_power(beta), 0.5)
        P.pim_anneal(hd, R, 0, 4, init_spins=init)
        assert np.array_equal(P.pim_energies(hd)["final_E"], oracle.energy(inst.J, inst.h, init))
        P.pim_anneal(hd, R, 5, 4, init_spins=init)
        P.pim_anneal(hd, R, 6, 4, t_begin=5, flags=P.PIM_CONTINUE)
        got = collect(hd, n)
    finally:
        P.pim_destroy(hd)
    assert_same(got, oracle_run(inst, beta, eta_power(beta), 0.5, replicas=R, seed=4, init=init))
