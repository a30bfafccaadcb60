"""Fused real-valued kernel: energies are the same to the last bit in every tile height (32, 64 and 128
replicas per CTA), as doubles, not only their whole part."""
import numpy as np
import pytest

from oracle import pimi
from workloads import eta_power, linear_beta, maxcut_gauss

from gpu_helpers import pim

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 16, 63, 65, 128, 200, 256])
def test_energies_agree_to_the_last_bit(n):
    P = pim()
    T, R = 12, 100
    beta = linear_beta(T)
    J = pimi.round_bf16(maxcut_gauss(n, 4).J)
    h = pimi.round_bf16(np.random.default_rng(4).standard_normal(n))
    handles = []
    try:
        for _ in range(240):
            hd = P.pim_create(J, h, 2.0 / np.sqrt(n))
            handles.append(hd)
            P.pim_set_schedule(hd, beta, eta_power(beta), 0.7)
        P.pim_anneal(handles[0], R, T, 11, instance_id=3)  # tiles of 32
        alone = P.pim_energies(handles[0])
        assert np.any(alone["best_E"] != np.floor(alone["best_E"]))
        for count in (40, 60, 240):  # up to tiles of 128
            P.pim_anneal_batch(handles[:count], R, T, 11, instance_ids=[3] * count)
            for hd in (handles[0], handles[count - 1]):
                got = P.pim_energies(hd)
                for k in alone:
                    assert np.array_equal(got[k], alone[k]), (count, k)
    finally:
        for hd in handles:
            P.pim_destroy(hd)
