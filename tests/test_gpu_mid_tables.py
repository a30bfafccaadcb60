"""Mid-N integer kernel: threshold tables on both sides of a half of the shared-memory table area
(copied one step ahead), the whole area (loaded by the deciding threads) and past it (global memory),
units of all kinds in one batch, odd and even numbers of steps, split runs."""
import numpy as np
import pytest

from workloads import Instance, eta_power, linear_beta, sk_pm1

from gpu_helpers import assert_same, collect, oracle_run, pim

pytestmark = pytest.mark.gpu


def _instance(n, imax):
    """SK couplings and a bias on spin 0 that sets the largest |field| to `imax` (0: no bias; -2: no
    bias and couplings +-2)."""
    inst = sk_pm1(n, 3)
    if imax == 0:
        return inst
    if imax < 0:
        return Instance(inst.kind, n, -imax * inst.J, inst.h, inst.c, 3)
    h = np.zeros(n, np.int32)
    h[0] = imax - int(np.abs(inst.J[0]).sum())
    return Instance(inst.kind, n, inst.J, h, inst.c, 3)


# table words of a step: 2 imax + 1, rounded up to a multiple of 4
CASES = [(300, 0), (300, 1023), (300, 1024), (300, 2047), (300, 2048), (512, 0), (513, 0), (700, 1023), (600, -2),
         (1000, 0), (1024, 0)]


@pytest.mark.parametrize("shared", [False, True])
@pytest.mark.parametrize("T", [1, 2, 7])
def test_tables_in_one_batch(T, shared):
    """Every kind of unit follows another on the same SM, and each equals the oracle's run; with and
    without units whose table is too large for shared memory."""
    P = pim()
    beta = linear_beta(T) if T > 1 else np.array([0.7])
    insts = [_instance(n, imax) for n, imax in CASES if not shared or imax < 2048]
    R = (3, 130)[T % 2]
    hd = []
    try:
        for k in range(200):  # more units than SMs
            inst = insts[k % len(insts)]
            h = P.pim_create(inst.J, inst.h if inst.h.any() else None, inst.c)
            hd.append(h)
            P.pim_set_schedule(h, beta, eta_power(beta), 0.6)
        P.pim_anneal_batch(hd, [R] * len(hd), T, 5, instance_ids=[0] * len(hd))
        want = [oracle_run(inst, beta, eta_power(beta), 0.6, replicas=R, seed=5) for inst in insts]
        for k, h in enumerate(hd):
            assert_same(collect(h, insts[k % len(insts)].n), want[k % len(insts)], label=f"unit {k}")
    finally:
        for h in hd:
            P.pim_destroy(h)


@pytest.mark.parametrize("n,imax", CASES)
def test_split_run(n, imax):
    P = pim()
    T = 9
    beta = linear_beta(T)
    inst = _instance(n, imax)
    hd = P.pim_create(inst.J, inst.h if imax > 0 else None, inst.c)
    try:
        P.pim_set_schedule(hd, beta, eta_power(beta), 0.5)
        P.pim_anneal(hd, 40, 4, 6)
        P.pim_anneal(hd, 40, 5, 6, t_begin=4, flags=P.PIM_CONTINUE)
        got = collect(hd, n)
    finally:
        P.pim_destroy(hd)
    assert_same(got, oracle_run(inst, beta, eta_power(beta), 0.5, replicas=40, seed=6))
