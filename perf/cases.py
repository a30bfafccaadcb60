"""Work that programs have this library do, for timing it: annealing calls through the public entry points.

A case is a dict of plain values:
  call      "oneshot"     host matrix in, host results out: create, schedule, anneal, read, destroy
            "anneal"      one instance that the program keeps, all records read on the device
            "batch"       pim_anneal_batch over instances that arrived together
            "plan"        a batch plan that the program keeps and runs again
            "sequential"  the conventional, spin-by-spin update of one instance
  problem   "maxcut" (J = -A, edge probability 1/2), "sk" (J = +-1), "gauss" (Max-Cut with
            N(0, 1) weights, real couplings), "mimo" (detection of 16-QAM over a Rayleigh
            channel, real couplings with a bias, n = 4 antennas), "uneven" (Max-Cut and SK
            of sizes in [64, n] and replica counts in [32, replicas])
  n, count, replicas, sweeps   spins, instances, replicas of each, sweeps of one pass
  field     an integer external field h in [-3, 3] beside the couplings
  noise     "gauss" or "uniform";  lut: levels of the staircase activation, 0 = tanh
  spins     the program gives the initial spins (else they come from the library's generator)
"""
import math

import numpy as np
import torch

from paper_2604_17109_gb300 import pim

SEED = 7  # Philox key of every run; a case's inputs come from the seed that prepare() gets


def _case(name, call, problem, n, count, replicas, sweeps, field=False, noise="gauss", lut=0, spins=False):
    c = dict(call=call, problem=problem, n=n, count=count, replicas=replicas, sweeps=sweeps,
             field=field, noise=noise, lut=lut, spins=spins)
    return dict(c, name=name) if name else c


def listed():
    return [
        # Detection requests that a base station's loop has in hand at once: 16 x 16 antennas,
        # the paper's 64 sweeps.  The smallest calls: their latency is what the user waits for.
        _case("mimo16_requests", "batch", "mimo", 64, 4, 32, 64),
        # The same for 64 x 64 antennas, a burst of requests.
        _case("mimo64_requests", "batch", "mimo", 256, 16, 32, 256),
        # One small graph, solved once from host arrays: what a first-time or scripted user calls.
        _case("oneshot_sk200", "oneshot", "sk", 200, 1, 128, 200),
        # The paper's Max-Cut size with its 64 trials: one small resident instance.
        _case("maxcut100", "anneal", "maxcut", 100, 1, 64, 1000),
        # An odd size and a ragged replica count with an external field, uniform noise and the
        # staircase activation of the hardware design.
        _case("field173_lut", "batch", "sk", 173, 24, 100, 300, field=True, noise="uniform", lut=8),
        # The benchmark's workload: 100 spin glasses, 1024 replicas, kept as a batch plan.
        _case("sk200_plan", "plan", "sk", 200, 100, 1024, 2000),
        # A batch of mid-size spin glasses, kept as a plan.
        _case("sk512_plan", "plan", "sk", 512, 152, 256, 200),
        # Mixed sizes and replica counts in one plan, as a solver service collects them.
        _case("uneven_plan", "plan", "uneven", 1024, 128, 512, 200),
        # One graph of odd size from given spins, too large for the small-instance kernels.
        _case("maxcut1201", "anneal", "maxcut", 1201, 1, 200, 200, spins=True),
        # The large integer benchmark instance.
        _case("sk4096", "anneal", "sk", 4096, 1, 256, 200),
        # The large real-valued benchmark instance, whose couplings exceed the L2 cache.
        _case("gauss8192", "anneal", "gauss", 8192, 1, 256, 40),
        # The conventional method that the parallel one is compared with.
        _case("sequential200", "sequential", "sk", 200, 1, 256, 100),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: the kinds above, sizes over their logarithm; total work at most that of
    the largest listed case."""
    kind = rng.choice(["mimo", "oneshot", "small", "field", "plan_small", "plan_mid", "uneven",
                       "large", "large_real", "sequential"])
    ints = rng.choice(["maxcut", "sk"])
    if kind == "mimo":
        return _case(None, "batch", "mimo", 4 * _log_int(rng, 8, 64), _log_int(rng, 1, 24),
                     rng.choice([16, 32, 64]), _log_int(rng, 48, 256))
    if kind == "oneshot":
        return _case(None, "oneshot", ints, _log_int(rng, 40, 400), 1, _log_int(rng, 32, 256),
                     _log_int(rng, 100, 400))
    if kind == "small":
        return _case(None, "anneal", ints, _log_int(rng, 40, 256), 1, _log_int(rng, 32, 512),
                     _log_int(rng, 200, 1000), spins=rng.random() < 0.5)
    if kind == "field":
        return _case(None, "batch", ints, _log_int(rng, 60, 700), _log_int(rng, 4, 40),
                     _log_int(rng, 32, 256), _log_int(rng, 100, 300), field=True,
                     noise=rng.choice(["gauss", "uniform"]), lut=rng.choice([0, 4, 8]))
    if kind == "plan_small":
        return _case(None, "plan", ints, _log_int(rng, 64, 255), _log_int(rng, 16, 100),
                     _log_int(rng, 64, 1024), _log_int(rng, 200, 2000))
    if kind == "plan_mid":
        return _case(None, "plan", ints, _log_int(rng, 257, 1024), _log_int(rng, 16, 152),
                     _log_int(rng, 64, 256), _log_int(rng, 50, 200))
    if kind == "uneven":
        return _case(None, "plan", "uneven", rng.randint(400, 1024), _log_int(rng, 32, 128),
                     512, _log_int(rng, 50, 200))
    if kind == "large":
        return _case(None, "anneal", ints, _log_int(rng, 1025, 4800), 1, _log_int(rng, 64, 256),
                     _log_int(rng, 50, 200), spins=rng.random() < 0.5)
    if kind == "large_real":
        return _case(None, "anneal", "gauss", _log_int(rng, 300, 8192), 1, _log_int(rng, 64, 256),
                     _log_int(rng, 20, 40))
    return _case(None, "sequential", ints, _log_int(rng, 60, 400), 1, _log_int(rng, 32, 256),
                 _log_int(rng, 50, 100))


def _shapes(case):
    """(n, replicas) of every instance; an uneven batch's follow from the case alone."""
    if case["problem"] != "uneven":
        return [(case["n"], case["replicas"])] * case["count"]
    g = np.random.default_rng([case["n"], case["count"]])
    n = g.integers(64, case["n"] + 1, case["count"])
    r = 32 * g.integers(1, case["replicas"] // 32 + 1, case["count"])
    # Up to 256 spins the last 16 of a bit row's 64 hold at least one (see _spin_words).
    n = np.where(n <= 256, n - (n - 1) % 64 + 48 + (n - 1) % 64 // 4, n)
    return [(int(a), int(b)) for a, b in zip(n, r)]


def _spin_words(bits, case):
    """The 16-bit words of bit rows that hold spins.  Rows are padded to 64 spins, and what the
    padding holds is not defined by every kernel, so a program does not look at it."""
    if case["problem"] == "uneven":
        return bits
    n = case["n"]
    return bits.view(torch.int16).reshape(-1, 4 * ((n + 63) // 64))[:, :(n + 15) // 16]


def _schedule(case):
    t = np.arange(case["sweeps"], dtype=np.float64) / max(case["sweeps"] - 1, 1)
    if case["problem"] == "mimo":  # beta = 1, noise falling as the paper's gamma rises
        return np.ones(t.size, np.float32), np.sqrt(1.0 / (5.0 * (0.01 + 0.99 * t))).astype(np.float32)
    beta = (0.1 + 2.9 * t).astype(np.float32)
    return beta, np.sqrt(beta.astype(np.float64) / 5.0).astype(np.float32)


def _couplings(problem, n, gen):
    """Symmetric couplings with a zero diagonal, drawn on the GPU, as a host array."""
    if problem == "gauss":
        w = torch.randn((n, n), generator=gen, device="cuda")
        w = w * (torch.rand((n, n), generator=gen, device="cuda") < 0.5)
        w = torch.triu(-w, 1)
    else:
        b = torch.rand((n, n), generator=gen, device="cuda") < 0.5
        w = torch.triu(torch.where(b, 1, -1) if problem == "sk" else -b.to(torch.int8), 1).to(torch.int8)
    return (w + w.T).cpu().numpy()


def _detection(nt, g):
    """Couplings, bias and schedule scale of one 16-QAM detection problem at 10 to 25 dB."""
    H = (g.standard_normal((nt, nt)) + 1j * g.standard_normal((nt, nt))) / np.sqrt(2.0)
    x = g.choice([-3.0, -1.0, 1.0, 3.0], nt) + 1j * g.choice([-3.0, -1.0, 1.0, 3.0], nt)
    y = H @ x
    es_n0 = 4.0 * 10.0 ** (g.uniform(10.0, 25.0) / 10.0)
    sigma = np.sqrt(np.mean(np.abs(y) ** 2) / es_n0 / 2.0)
    y = y + sigma * (g.standard_normal(nt) + 1j * g.standard_normal(nt))
    J, h, _ = pim.pim_mimo_formulate(H, y, 16, 1.0 / es_n0)
    return J, h, 2.0 / nt


def _problems(case, seed):
    """(J, h or None, scale, xi) of every instance."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    g = np.random.default_rng(seed)
    out = []
    for k, (n, _) in enumerate(_shapes(case)):
        p = case["problem"]
        if p == "mimo":
            out.append((*_detection(n // 4, g), 1.0))
            continue
        if p == "uneven":
            p = "maxcut" if k % 2 == 0 else "sk"
        h = g.integers(-3, 4, n).astype(np.int32) if case["field"] else None
        c = (1.0 if p == "sk" else 2.0) / math.sqrt(n)
        out.append((_couplings(p, n, gen), h, c, 0.5 if p == "sk" else 0.7))
    return out


def _spins(case, seed):
    g = np.random.default_rng([seed, 1])
    return np.where(g.random((case["replicas"], case["n"])) < 0.5, -1, 1).astype(np.int8)


def _stage(case, J, h, scale, xi):
    beta, eta = _schedule(case)
    inst = pim.pim_create(J, h, scale)
    pim.pim_set_schedule(inst, beta, eta, xi, case["noise"], "lut" if case["lut"] else "tanh",
                         case["lut"] or 4)
    return inst


class _State:
    """Handles that a program keeps between calls, and the tensors it reads results into."""

    def __init__(self, case, seed):
        self.case, self.insts, self.plan, self.spins = case, [], None, None
        self.problems = None
        if case["call"] == "oneshot":
            self.problems = _problems(case, seed)
            return
        self.insts = [_stage(case, *p) for p in _problems(case, seed)]
        shapes = _shapes(case)
        self.replicas = [r for _, r in shapes]
        if case["spins"]:
            self.spins = _spins(case, seed)
        if case["call"] == "plan":
            self.plan = pim.pim_batch_create(self.insts, self.replicas)
        rows = [0]
        words = [0]
        for inst, r in zip(self.insts, self.replicas):
            rows.append(rows[-1] + r)
            words.append(words[-1] + r * pim.pim_state_words(inst))
        self.out = {"best_E": torch.empty(rows[-1], dtype=torch.float64, device="cuda"),
                    "best_bits": torch.empty(words[-1], dtype=torch.int32, device="cuda")}
        if len(self.insts) == 1:  # a single instance's user reads every record
            self.out.update(
                final_E=torch.empty(rows[-1], dtype=torch.float64, device="cuda"),
                best_t=torch.empty(rows[-1], dtype=torch.int32, device="cuda"),
                first_hit=torch.empty(rows[-1], dtype=torch.int32, device="cuda"),
                final_bits=torch.empty(words[-1], dtype=torch.int32, device="cuda"))
        self.views = []
        for k in range(len(self.insts)):
            at = {}
            for name, t in self.out.items():
                o = words if name.endswith("bits") else rows
                at[name] = t[o[k]:o[k + 1]]
            self.views.append(at)
        self.result = {name: _spin_words(t, case) if name.endswith("bits") else t
                       for name, t in self.out.items()}

    def __del__(self):
        if self.plan is not None:
            pim.pim_batch_destroy(self.plan)
        for inst in self.insts:
            pim.pim_destroy(inst)


def prepare(case, seed):
    return _State(case, seed)


def run(state):
    c = state.case
    if c["call"] == "oneshot":
        out = {}
        for J, h, scale, xi in state.problems:
            inst = _stage(c, J, h, scale, xi)
            pim.pim_anneal(inst, c["replicas"], c["sweeps"], SEED, flags=pim.PIM_RESULTS_TO_HOST)
            out = dict(pim.pim_energies(inst), best=pim.pim_best_state(inst, c["n"]))
            pim.pim_destroy(inst)
        return out
    stream = torch.cuda.current_stream()
    if c["call"] == "plan":
        pim.pim_batch_run(state.plan, c["sweeps"], SEED, stream=stream)
    elif c["call"] == "batch":
        pim.pim_anneal_batch(state.insts, state.replicas, c["sweeps"], SEED, stream=stream)
    elif c["call"] == "sequential":
        pim.pim_anneal_sequential(state.insts[0], c["replicas"], c["sweeps"], SEED, stream=stream)
    else:
        pim.pim_anneal(state.insts[0], c["replicas"], c["sweeps"], SEED, init_spins=state.spins,
                       stream=stream)
    for inst, at in zip(state.insts, state.views):
        pim.pim_results_dev(inst, **at, stream=stream)
    return state.result


def work(case):
    """Couplings and bias in, the records that are read out; the fields' multiplies and adds
    (the spin-by-spin method needs a row of the couplings for a flipped spin only: its fields
    of one sweep stand for that)."""
    real = case["problem"] in ("gauss", "mimo")
    nbytes = flops = 0
    for n, r in _shapes(case):
        nbytes += n * n * (2 if real else 1) + (4 * n if case["field"] or case["problem"] == "mimo" else 0)
        nbytes += r * (8 + n / 8) * (2 if case["count"] == 1 else 1)
        nbytes += r * n if case["spins"] else 0
        flops += 2.0 * n * n * r * (1 if case["call"] == "sequential" else case["sweeps"])
    return {"bytes": int(nbytes), "flops": flops}


# ---- the same runs in plain torch, from the definitions in include/pim.h -------------------

_MASK = 0xFFFFFFFF


def _philox(c0, c1, c2, c3, seed):
    """Philox4x32-10 (Salmon et al., SC'11) on int64 tensors holding 32-bit words."""
    k0, k1 = seed & _MASK, seed >> 32

    def mul(m, c):  # 32 x 32 -> (high, low) without leaving 63 bits
        lo, hi = m * (c & 0xFFFF), m * (c >> 16)
        mid = hi + (lo >> 16)
        return mid >> 16, ((mid & 0xFFFF) << 16) | (lo & 0xFFFF)

    for _ in range(10):
        h0, l0 = mul(0xD2511F53, c0)
        h1, l1 = mul(0xCD9E8D57, c2)
        c0, c1, c2, c3 = h1 ^ c1 ^ k0, l1, h0 ^ c3 ^ k1, l0
        k0, k1 = (k0 + 0x9E3779B9) & _MASK, (k1 + 0xBB67AE85) & _MASK
    return torch.stack([c0, c1, c2, c3], -1)


def _draws(count, replicas, n, t):
    """16-bit draws [count, replicas, n] of step field t: word (i & 7) >> 1 of block i >> 3,
    the low half for even i."""
    dev = "cuda"
    shape = (count, replicas, (n + 7) // 8)
    blk = torch.arange(shape[2], device=dev).expand(shape)
    r = torch.arange(replicas, device=dev)[None, :, None].expand(shape)
    q = torch.arange(count, device=dev)[:, None, None].expand(shape)
    w = _philox(blk, r, torch.full(shape, t, dtype=torch.int64, device=dev), q, SEED)
    return torch.stack([w & 0xFFFF, w >> 16], -1).reshape(count, replicas, -1)[:, :, :n]


def _decider(case, scale, xi):
    """step t -> function (fields, spins, draws) -> new spins, the float32 rule of pim.h."""
    beta, eta = _schedule(case)
    m = torch.arange(4096, dtype=torch.float64, device="cuda")
    if case["noise"] == "uniform":
        z = ((2 * m - 4095) / 4096).float()
    else:
        z = torch.special.ndtri((m + 0.5) / 4096).float()
        z[2048:] = -z[:2048].flip(0)
    L = case["lut"]
    levels = torch.tensor([-1.0 + 2.0 * k / (L - 1) for k in range(L)], dtype=torch.float64, device="cuda") if L else None
    edges = torch.tensor([-1.0 + 2.0 * k / L for k in range(1, L)], dtype=torch.float64, device="cuda") if L else None

    def decide(t, I, s, d):
        x = float(np.float32(np.float64(beta[t]) * scale)) * I.double()
        tau = levels[torch.bucketize(x, edges, right=True)] if L else torch.tanh(x)
        a = tau.float() + torch.where(s > 0, float(np.float32(xi)), -float(np.float32(xi))).float()
        return torch.where(a + float(eta[t]) * z[d >> 4] >= 0, 1.0, -1.0)

    return decide


def exact(case, seed):
    """What run() returns, for the integer problems of one size (whole numbers throughout: the
    fields are exact in these sums).  A real-valued run has no such value: one decision that a
    rounding turns changes every later state.  Uneven batches take too long."""
    if case["problem"] in ("gauss", "mimo", "uneven"):
        return None
    cnt, n, R, T = case["count"], case["n"], case["replicas"], case["sweeps"]
    if cnt * n * R * T > 5e10 or (case["call"] == "sequential" and n * T > 3e4):
        return None
    probs = _problems(case, seed)
    J = torch.tensor(np.stack([p[0] for p in probs]), device="cuda").float()
    h = torch.tensor(np.stack([p[1] if p[1] is not None else np.zeros(n, np.int32) for p in probs]),
                     device="cuda").float()[:, None, :]
    decide = _decider(case, probs[0][2], probs[0][3])
    if case["spins"]:
        s = torch.tensor(_spins(case, seed), device="cuda").float()[None]
    else:
        s = torch.where(_draws(cnt, R, n, 0xFFFFFFFF) >> 15 > 0, 1.0, -1.0)
    best_E = torch.full((cnt, R), math.inf, dtype=torch.float64, device="cuda")
    best_t = torch.full((cnt, R), -1, dtype=torch.int32, device="cuda")
    best = s.clone()
    for t in range(T + 1):
        I = torch.matmul(s, J) + h
        E = -((s * (I + h)).double().sum(-1) / 2)
        better = E < best_E
        best_E = torch.where(better, E, best_E)
        best_t[better] = t
        best = torch.where(better[..., None], s, best)
        if t == T:
            break
        d = _draws(cnt, R, n, t)
        if case["call"] == "sequential":
            s = s.clone()
            for i in range(n):
                new = decide(t, I[..., i], s[..., i], d[..., i])
                I += (new - s[..., i])[..., None] * J[:, None, i, :]
                s[..., i] = new
        else:
            s = decide(t, I, s, d)

    def bits(x):  # bit i % 32 of word i // 32 set <=> spin i = +1, 2 ceil(n / 64) words
        pad = torch.zeros((cnt, R, 64 * ((n + 63) // 64)), dtype=torch.int64, device="cuda")
        pad[..., :n] = x > 0
        w = (pad.reshape(cnt, R, -1, 32) << torch.arange(32, device="cuda")).sum(-1)
        return _spin_words(torch.where(w >= 1 << 31, w - (1 << 32), w).to(torch.int32).reshape(-1), case)

    out = {"best_E": best_E.reshape(-1), "best_bits": bits(best)}
    hit = torch.full((cnt * R,), -1, dtype=torch.int32, device="cuda")
    if case["call"] == "oneshot":
        return {"best_E": best_E[0], "final_E": E[0], "best_t": best_t[0], "first_hit": hit,
                "best": best[0].to(torch.int8)}
    if cnt == 1:
        out.update(final_E=E.reshape(-1), best_t=best_t.reshape(-1), first_hit=hit, final_bits=bits(s))
    return out
