"""pim_results_dev: the bits of a row past the last spin are 0, whichever kernel ran, also where the
result block held other bits before."""
import numpy as np
import pytest
import torch

from gpu_helpers import pim
from workloads import eta_power, linear_beta, maxcut_gauss, sk_pm1

pytestmark = pytest.mark.gpu

T = 4


def _run(P, inst, R, flags, target):
    """One run's best and final bit rows."""
    beta = linear_beta(T)
    hd = P.pim_create(inst.J, None, inst.c)
    try:
        P.pim_set_schedule(hd, beta, eta_power(beta), 0.5, "uniform")
        if target == "sequential":
            P.pim_anneal_sequential(hd, R, T, 9)
        else:
            P.pim_anneal(hd, R, T, 9, flags=flags)
        words = P.pim_state_words(hd)
        out = {k: torch.full((R * words,), -1, dtype=torch.int32, device="cuda") for k in ("best_bits", "final_bits")}
        P.pim_results_dev(hd, **out)
        torch.cuda.synchronize()
    finally:
        P.pim_destroy(hd)
    return {k: np.unpackbits(v.cpu().numpy().view(np.uint8).reshape(R, 4 * words), axis=1, bitorder="little")
            for k, v in out.items()}


# integer n <= 256: few replicas take the latency kernel, many the throughput kernel (40000 with its queue)
KINDS = [("sk", 64, 0), ("sk", 9600, 0), ("sk", 40000, 0), ("sk", 130, "mid"), ("sk", 130, "sequential"), ("gauss", 130, 0)]


@pytest.mark.parametrize("kind,R,path", KINDS)
@pytest.mark.parametrize("n", [1, 33, 72, 129, 200])
def test_fused_sizes(n, kind, R, path):
    P = pim()
    make = sk_pm1 if kind == "sk" else maxcut_gauss
    flags = P.PIM_PATH_MID if path == "mid" else 0
    full = 64 * ((n + 63) // 64)
    _run(P, make(full, 1), R, 0, path)  # leaves a result block of the same size full of spins
    for k, bits in _run(P, make(n, 2), R, flags, path).items():
        assert bits[:, :n].any() and not bits[:, n:].any(), k


@pytest.mark.parametrize("kind,path", [("sk", "mid"), ("sk", "big"), ("sk", "sequential"), ("gauss", "big")])
@pytest.mark.parametrize("n", [257, 328, 545])
def test_larger_sizes(n, kind, path):
    P = pim()
    make = sk_pm1 if kind == "sk" else maxcut_gauss
    flags = {"mid": P.PIM_PATH_MID, "big": P.PIM_PATH_BIG}.get(path, 0)
    full = 64 * ((n + 63) // 64)
    _run(P, make(full, 1), 130, flags, path)
    for k, bits in _run(P, make(n, 2), 130, flags, path).items():
        assert bits[:, :n].any() and not bits[:, n:].any(), k
