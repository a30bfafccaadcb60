"""pim_results_dev: every record arrives whole, into aligned and 4-byte-aligned tensors, on the
run's stream and on another, and a pinned host destination still works."""
import numpy as np
import pytest
import torch

from gpu_helpers import pim
from workloads import eta_power, linear_beta, sk_pm1

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,R", [(1, 1), (33, 7), (200, 129), (1100, 130)])
@pytest.mark.parametrize("where", ["same", "other", "pinned", "shifted"])
def test_records_arrive(n, R, where):
    P = pim()
    inst = sk_pm1(n, 1)
    T = 12
    beta = linear_beta(T)
    hd = P.pim_create(inst.J, None, inst.c)
    try:
        P.pim_set_schedule(hd, beta, eta_power(beta), 0.5)
        run = torch.cuda.Stream()
        read = torch.cuda.Stream() if where == "other" else run
        words = P.pim_state_words(hd)
        kw = dict(pin_memory=True) if where == "pinned" else dict(device="cuda")
        off = 1 if where == "shifted" else 0
        t = {k: torch.zeros(R + off, dtype=torch.float64, **kw)[off:] for k in ("best_E", "final_E")}
        t |= {k: torch.zeros(R + off, dtype=torch.int32, **kw)[off:] for k in ("best_t", "first_hit")}
        t |= {k: torch.zeros(R * words + off, dtype=torch.int32, **kw)[off:] for k in ("best_bits", "final_bits")}
        torch.cuda.synchronize()  # the tensors are filled before another stream writes them
        P.pim_anneal(hd, R, T, 3, target=-n, stream=run)
        P.pim_results_dev(hd, **t, stream=read)
        torch.cuda.synchronize()
        want = P.pim_energies(hd)
        for k in ("best_E", "final_E", "best_t", "first_hit"):
            assert np.array_equal(t[k].cpu().numpy(), want[k]), k
        for k, s in (("best_bits", P.pim_best_state(hd, n)), ("final_bits", P.pim_final_state(hd, n))):
            b = t[k].cpu().numpy().view(np.uint32).reshape(R, words)
            i = np.arange(n)
            assert np.array_equal(((b[:, i // 32] >> (i % 32)) & 1).astype(bool), s > 0), k
    finally:
        P.pim_destroy(hd)
