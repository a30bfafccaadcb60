"""Large-N kernel: the replica tiles of a launch wait for no other tile, so a replica's run is the same
however many tiles run beside it, in one launch or several, alone or from a plan's scratch."""
import numpy as np
import pytest

from oracle import pimi
from workloads import Instance, eta_power, linear_beta, maxcut_gauss, sk_pm1

from gpu_helpers import pim

pytestmark = pytest.mark.gpu


def _instance(kind, n):
    if kind == "real":
        base = maxcut_gauss(n, 3)
        return Instance("maxcut_gauss", n, pimi.round_bf16(base.J), np.zeros(n), base.c, 3)
    inst = sk_pm1(n, 3)
    if kind == "wide":  # couplings beyond E2M1: the streamed FP8 variant
        return Instance("sk", n, 5 * inst.J, inst.h, inst.c / 5, 3)
    return inst


# tiles of 128 replicas: one; a few and a ragged one; one more than fits a launch; several launches
@pytest.mark.parametrize("kind,n,R", [
    ("e2m1", 513, 100), ("e2m1", 513, 300), ("e2m1", 1201, 900), ("e2m1", 1201, 2000), ("wide", 300, 2500),
    ("wide", 700, 1300), ("wide", 1500, 1100), ("real", 300, 700), ("real", 1000, 1300)])
def test_tiles_do_not_matter(kind, n, R):
    P = pim()
    inst = _instance(kind, n)
    T = 7
    beta = linear_beta(T)
    hd = P.pim_create(inst.J, None, inst.c)
    try:
        P.pim_set_schedule(hd, beta, eta_power(beta), 0.5)
        P.pim_anneal(hd, 64, T, 5, flags=P.PIM_PATH_BIG)
        few, few_E = P.pim_final_state(hd, n), P.pim_energies(hd)
        P.pim_anneal(hd, R, T, 5, flags=P.PIM_PATH_BIG)
        many, many_E = P.pim_final_state(hd, n), P.pim_energies(hd)
        assert np.array_equal(many[:64], few)
        plan = P.pim_batch_create([hd], [R], instance_ids=[0], flags=P.PIM_PATH_BIG)
        try:
            P.pim_batch_run(plan, T, 5)
            assert np.array_equal(P.pim_final_state(hd, n), many)
        finally:
            P.pim_batch_destroy(plan)
        # energies of the last replica's own state, which lies in the last tile
        s = many[-1].astype(np.float64)
        want = -0.5 * s @ inst.J.astype(np.float64) @ s
        if kind == "real":  # FP32 sums of n^2 products of N(0, 1) couplings
            assert abs(many_E["final_E"][-1] - want) <= 1e-4 * n * np.sqrt(n)
        else:
            assert many_E["final_E"][-1] == want
            assert np.array_equal(many_E["best_E"][:64], few_E["best_E"])
            assert np.array_equal(many_E["best_t"][:64], few_E["best_t"])
    finally:
        P.pim_destroy(hd)
