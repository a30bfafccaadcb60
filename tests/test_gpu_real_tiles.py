"""Fused real-valued kernel: every tile height (32, 64, 128 replicas) and capacity (64, 128, 256
spins) takes the same decisions and sums the same energies, bit for bit, at the edges of its
chunks and tiles, and the decisions of one sweep are the float64 oracle's beyond FP32 error.

A lone instance runs in tiles of 32 replicas; in a batch that fills the GPU several times over
the same instance runs in tiles of 128, in a batch in between in tiles of 64."""
import numpy as np
import pytest

import oracle
from oracle import pimi
from workloads import Instance, eta_power, linear_beta, maxcut_gauss, random_spins

from gpu_helpers import collect, pim

pytestmark = pytest.mark.gpu


def _instance(n, seed):
    J = pimi.round_bf16(maxcut_gauss(n, seed).J)
    h = pimi.round_bf16(np.random.default_rng(seed).standard_normal(n))
    return Instance("maxcut_gauss", n, J, h, 2.0 / np.sqrt(n), seed)


@pytest.mark.parametrize("act", ["tanh", "lut"])
@pytest.mark.parametrize("n", [1, 15, 16, 17, 63, 64, 65, 128, 129, 200, 256])
def test_tile_heights_agree(n, act):
    P = pim()
    T, R = 24, 100
    beta = linear_beta(T)
    inst = _instance(n, 4)
    handles = []
    try:
        for _ in range(240):
            hd = P.pim_create(inst.J, inst.h, inst.c)
            handles.append(hd)
            P.pim_set_schedule(hd, beta, eta_power(beta), 0.7, act=act, lut_levels=5)
        P.pim_anneal(handles[0], R, T, 11, instance_id=3)
        alone = collect(handles[0], n)
        for count in (40, 60, 240):
            P.pim_anneal_batch(handles[:count], R, T, 11, instance_ids=[3] * count)
            for hd in (handles[0], handles[count - 1]):
                got = collect(hd, n)
                for k in alone:
                    assert np.array_equal(got[k], alone[k]), (count, k)
    finally:
        for hd in handles:
            P.pim_destroy(hd)


@pytest.mark.parametrize("n,R", [(16, 32), (65, 33), (100, 128), (256, 65)])
@pytest.mark.parametrize("xi,eta_t", [(0.0, 0.0), (1.0, 0.45), (2.0, 3.0)])
def test_one_sweep_matches_oracle(n, R, xi, eta_t):
    """|delta_gpu - delta_oracle| <= b n 2^-23 row sum (FP32 fields through a Lipschitz-1 tanh)
    + 1e-6 (1 + xi + 4 eta) (tanhf and three float32 operations)."""
    P = pim()
    inst = _instance(n, 9)
    beta = np.full(2, 1.5, np.float32)
    eta = np.full(2, eta_t, np.float32)
    init = random_spins(n, R, seed=2)
    hd = P.pim_create(inst.J, inst.h, inst.c)
    try:
        P.pim_set_schedule(hd, beta, eta, xi)
        P.pim_anneal(hd, R, 1, 21, init_spins=init)
        got = P.pim_final_state(hd, n)
    finally:
        P.pim_destroy(hd)
    I = oracle.field(inst.J, inst.h, init)
    b = np.float32(np.float64(beta[0]) * inst.c)
    d = oracle.noise_draw16(21, 0, np.arange(R)[:, None], 0, np.arange(n)[None, :])
    delta = pimi.delta(oracle.activation(b, I), init, np.float32(xi), eta[0],
                       pimi.gaussian_quantiles()[d >> 4])
    row = np.abs(inst.J).sum(axis=1) + np.abs(inst.h)
    bound = float(b) * n * 2.0 ** -23 * row[None, :] + 1e-6 * (1 + xi + 4 * eta_t)
    differ = got != np.where(delta >= 0, 1, -1)
    assert np.all(np.abs(delta)[differ] <= np.broadcast_to(bound, delta.shape)[differ])
