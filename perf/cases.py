"""The work that programs built on this package have it do, as measurable cases.

A case is one pass through the public entry points (``paper_1202_6163_gb300.pf``)
the way a particle-filter program calls them, in one of five forms:

``single``      one filter: optionally the effective sample size, one cumulative
                resampler, optionally the gather of the states or the in-place move
``all_four``    one filter through all four resamplers and the gather
``metropolis``  one filter through the Metropolis resampler
``batched``     many filters of uneven size in one call
``bootstrap``   whole steps of many bootstrap filters (draw, propagate, weight,
                resample where the effective sample size asks for it)

Sizes are those of this repository's configurations, tests and benchmark, and odd
ones between them.  ``exact`` gives the 64-bit values of the outputs that are
computed numbers; ancestors are whole numbers and rows moved by them are copies,
so they have none.
"""
import math

import numpy as np
import torch

from paper_1202_6163_gb300 import pf, workloads

KINDS = {"multinomial": pf.PF_MULTINOMIAL, "stratified": pf.PF_STRATIFIED, "systematic": pf.PF_SYSTEMATIC,
         "metropolis": pf.PF_METROPOLIS}

# The linear-Gaussian test model's noise, observation density and resampling rule.
LG_D = 4
LG_THRESHOLD = 0.5


def listed():
    return [
        # The smallest configuration: P = 1024, states x 4, every resampler in turn (Metropolis
        # B = 64) and the gather.  Five calls whose cost is launches and serial phases.
        {"name": "all_four_1024", "form": "all_four", "P": 1024, "law": "gaussian", "s": 1.0, "B": 64, "dim": 4},
        # An ordinary filter of odd size taking its resampling step: effective sample size,
        # systematic resampling, gather of four-dimensional states.
        {"name": "filter_step_20011", "form": "single", "kind": "systematic", "P": 20011, "law": "gaussian", "s": 1.0,
         "lead": 0, "ess": True, "move": "gather", "dim": 4},
        # The benchmark's filter, P = 2^20, through the scheme most filters use ...
        {"name": "systematic_1m", "form": "single", "kind": "systematic", "P": 1 << 20, "law": "gaussian", "s": 1.0,
         "lead": 0, "ess": False, "move": "none", "dim": 0},
        # ... through the paper's multinomial binary search ...
        {"name": "multinomial_1m", "form": "single", "kind": "multinomial", "P": 1 << 20, "law": "gaussian", "s": 1.0,
         "lead": 0, "ess": False, "move": "none", "dim": 0},
        # ... and through the paper's Metropolis resampler at the benchmark's B.
        {"name": "metropolis_1m", "form": "metropolis", "P": 1 << 20, "law": "gaussian", "s": 1.0, "B": 32},
        # A filter that cannot hold a second copy of its states: stratified resampling of an
        # unaligned odd-sized slice, the ancestors made fit for in-place moves, the rows moved.
        {"name": "stratified_inplace_3m", "form": "single", "kind": "stratified", "P": 3000017, "law": "gaussian",
         "s": 2.0, "lead": 1, "ess": False, "move": "inplace", "dim": 16},
        # A large multinomial resampling, odd size: random reads from more than L2 keeps close.
        {"name": "multinomial_16m", "form": "single", "kind": "multinomial", "P": (1 << 24) - 5, "law": "gaussian",
         "s": 1.0, "lead": 0, "ess": False, "move": "none", "dim": 0},
        # The large-filter configuration: P = 2^24 with one log-weight in a hundred raised by 10,
        # effective sample size, systematic resampling, gather of eight-dimensional states.
        {"name": "heavy_tail_step_16m", "form": "single", "kind": "systematic", "P": 1 << 24, "law": "heavy", "s": 1.0,
         "lead": 0, "ess": True, "move": "gather", "dim": 8},
        # The largest single filter: beyond what one cooperative launch holds.
        {"name": "stratified_100m", "form": "single", "kind": "stratified", "P": 100000000, "law": "gaussian", "s": 1.0,
         "lead": 0, "ess": False, "move": "none", "dim": 0},
        # Particle MCMC: 4096 filters of 256 to 65536 particles (sizes log-uniform, drawn from
        # the layout's own seed) resampled in one call.
        {"name": "batched_systematic_4096", "form": "batched", "kind": "systematic", "F": 4096, "P_lo": 256,
         "P_hi": 65536, "layout": 0, "B": 0},
        # The same through the Metropolis resampler.
        {"name": "batched_metropolis_4096", "form": "batched", "kind": "metropolis", "F": 4096, "P_lo": 256,
         "P_hi": 65536, "layout": 0, "B": 32},
        # Particle MCMC from the start: 256 bootstrap filters of 2^16 particles drawn and taken
        # through two steps, resampling between them where the weights ask for it.
        {"name": "bootstrap_256x65536", "form": "bootstrap", "kind": "systematic", "F": 256, "P": 65536, "T": 2},
    ]


def _log_uniform(rng, lo, hi):
    return int(math.exp(rng.uniform(math.log(lo), math.log(hi))))


def draw(rng):
    form = rng.choice(["single", "single", "single", "single", "large", "all_four", "metropolis", "batched", "batched",
                       "bootstrap"])
    cumulative = rng.choice(["systematic", "stratified", "multinomial"])
    if form == "single":
        move = rng.choice(["none", "none", "gather", "inplace"])
        lead = rng.choice([0, 0, 1, 2, 3])
        law = rng.choice(["gaussian", "gaussian", "heavy", "dirichlet"])
        # numpy draws the Dirichlet weights, at the sizes the paper simulates
        P = _log_uniform(rng, 256, (1 << 16) if law == "dirichlet" else (1 << 24))
        s = {"gaussian": rng.choice([0.25, 1.0, 2.0, 4.0]), "heavy": 1.0,
             "dirichlet": rng.choice([10.0, 1.0, 0.1, 0.01])}[law]
        return {"form": "single", "kind": cumulative, "P": P, "law": law, "s": s, "lead": lead,
                "ess": lead == 0 and rng.random() < 0.5, "move": move,
                "dim": 0 if move == "none" else rng.choice([1, 3, 4, 8, 16])}
    if form == "large":
        return {"form": "single", "kind": cumulative,
                "P": _log_uniform(rng, 1 << 24, 40000000 if cumulative == "multinomial" else 100000000),
                "law": "gaussian", "s": 1.0, "lead": rng.choice([0, 0, 1, 2, 3]), "ess": False, "move": "none",
                "dim": 0}
    if form == "all_four":
        return {"form": "all_four", "P": _log_uniform(rng, 256, 1 << 17), "law": "gaussian",
                "s": rng.choice([0.25, 1.0, 2.0]), "B": rng.choice([8, 32, 64]), "dim": rng.choice([4, 8, 16])}
    if form == "metropolis":
        # B < 0: the step count from the bias bound, found on the device
        bound = rng.random() < 0.5
        return {"form": "metropolis", "P": _log_uniform(rng, 256, (1 << 16) if bound else (1 << 21)),
                "law": "gaussian", "s": rng.choice([0.25, 1.0]), "B": -1 if bound else rng.choice([8, 32, 128])}
    if form == "batched":
        kind = rng.choice(["systematic", "stratified", "multinomial", "metropolis"])
        hi = rng.choice([4096, 16384, 65536])
        return {"form": "batched", "kind": kind, "F": _log_uniform(rng, 16, 4096), "P_lo": 256, "P_hi": hi,
                "layout": rng.randrange(1 << 16), "B": rng.choice([8, 32]) if kind == "metropolis" else 0}
    return {"form": "bootstrap", "kind": cumulative, "F": _log_uniform(rng, 4, 256), "P": _log_uniform(rng, 1000, 65536),
            "T": rng.choice([2, 2, 4])}


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------
def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _logw(case, seed, lead=0):
    """The case's P log-weights, `lead` floats past a 16-byte boundary."""
    P = case["P"]
    buf = torch.empty(P + lead, device="cuda")
    lw = buf[lead:]
    if case["law"] == "dirichlet":
        lw.copy_(torch.from_numpy(workloads.dirichlet_logw(P, case["s"], seed=seed)))
        return lw
    g = _generator(seed)
    lw.copy_(torch.randn(P, device="cuda", generator=g))
    if case["law"] == "heavy":
        lw += 10.0 * (torch.rand(P, device="cuda", generator=g) < 0.01)
    else:
        lw *= case["s"]
    return lw


def _i32(n):
    return torch.zeros(n, dtype=torch.int32, device="cuda")


def prepare(case, seed):
    st = {"case": case, "seed": seed}
    form = case["form"]
    if form == "batched":
        off, _ = workloads.batched_layout(case["F"], case["P_lo"], case["P_hi"], seed=case["layout"])
        _, spreads = workloads.batched_layout(case["F"], seed=seed)
        total = int(off[-1])
        sizes = torch.from_numpy(np.diff(off)).cuda()
        scale = torch.repeat_interleave(torch.from_numpy(spreads.astype(np.float32)).cuda(), sizes)
        st["lw"] = torch.randn(total, device="cuda", generator=_generator(seed)) * scale
        st["offsets"] = torch.from_numpy(off).cuda()
        st["seeds"] = torch.from_numpy(workloads.batched_seeds(case["F"], base=seed).view(np.int64)).cuda()
        st["anc"] = _i32(total)
        return st
    if form == "bootstrap":
        F, P, T = case["F"], case["P"], case["T"]
        a = workloads.lg_params(F, seed=seed)
        y = workloads.lg_observations(a, T=T, D=LG_D, seed=seed + 1)
        st["a"] = torch.from_numpy(a).cuda()
        st["y"] = torch.from_numpy(y).cuda()
        st["step_seeds"] = torch.from_numpy(workloads.lg_step_seeds(T, F, base=1000 + seed).view(np.int64)).cuda()
        st["offsets"] = torch.arange(F + 1, dtype=torch.int64, device="cuda") * P
        st["x"] = [torch.empty((F, P, LG_D), device="cuda") for _ in range(2)]
        st["lw"] = torch.empty((F, P), device="cuda")
        st["loglik"] = torch.empty(F, dtype=torch.float64, device="cuda")
        st["log_sum"] = torch.empty(F, dtype=torch.float64, device="cuda")
        st["ess"] = torch.empty(F, device="cuda")
        st["resample"] = _i32(F)
        st["anc"] = _i32(F * P)
        return st
    P = case["P"]
    st["lw"] = _logw(case, seed, case.get("lead", 0))
    if form == "metropolis":
        st["anc"] = _i32(P)
        return st
    if form == "all_four":
        st["anc"] = {k: _i32(P) for k in KINDS}
    else:
        st["anc"] = _i32(P)
        if case["ess"]:
            st["ess"] = torch.zeros(1, device="cuda")
            st["log_sum"] = torch.zeros(1, dtype=torch.float64, device="cuda")
        if case["move"] == "inplace":
            st["perm"] = _i32(P)
    if case["dim"]:
        st["states"] = torch.randn((P, case["dim"]), device="cuda", generator=_generator(seed + 1))
        if case.get("move") != "inplace":
            st["moved"] = torch.empty_like(st["states"])
    return st


# ---------------------------------------------------------------------------
# One pass
# ---------------------------------------------------------------------------
def run(st):
    case, seed = st["case"], st["seed"]
    form = case["form"]
    if form == "batched":
        pf.pf_resample_batched(KINDS[case["kind"]], st["lw"], st["offsets"], case["F"], case["B"], st["seeds"],
                               st["anc"])
        return {"ancestors": st["anc"]}
    if form == "bootstrap":
        F, P = case["F"], case["P"]
        kind = KINDS[case["kind"]]
        x, nx = st["x"]
        pf.pf_lg_init(F, P, LG_D, workloads.LG_M0, workloads.LG_P0, seed, x, st["lw"], st["loglik"], st["log_sum"],
                      st["ess"], st["resample"])
        for t in range(1, case["T"] + 1):
            if t > 1:
                pf.pf_resample_batched_masked(kind, st["lw"], st["offsets"], F, 0, st["step_seeds"][t - 1],
                                              st["resample"], st["anc"])
            pf.pf_lg_step(F, P, LG_D, st["a"], workloads.LG_Q, workloads.LG_R, LG_THRESHOLD, st["y"][t - 1], t, seed,
                          st["anc"], x, nx, st["lw"], st["loglik"], st["log_sum"], st["ess"], st["resample"])
            x, nx = nx, x
        return {"states": x, "previous_states": nx, "logw": st["lw"], "loglik": st["loglik"],
                "log_sum": st["log_sum"], "ess": st["ess"], "resample": st["resample"]}
    P, lw = case["P"], st["lw"]
    if form == "metropolis":
        pf.pf_resample_metropolis(lw, P, case["B"], seed, st["anc"])
        return {"ancestors": st["anc"]}
    if form == "all_four":
        for name, kind in KINDS.items():
            pf.RESAMPLERS[kind](lw, P, case["B"], seed, st["anc"][name])
        pf.pf_gather(st["states"], P, 4 * case["dim"], st["anc"]["systematic"], P, st["moved"])
        return {"ancestors": st["anc"], "states": st["moved"]}
    out = {}
    if case["ess"]:
        pf.pf_ess(lw, P, st["ess"], st["log_sum"])
        out["ess"], out["log_sum"] = st["ess"], st["log_sum"]
    pf.RESAMPLERS[KINDS[case["kind"]]](lw, P, 0, seed, st["anc"])
    out["ancestors"] = st["anc"]
    if case["move"] == "gather":
        pf.pf_gather(st["states"], P, 4 * case["dim"], st["anc"], P, st["moved"])
        out["states"] = st["moved"]
    elif case["move"] == "inplace":
        pf.pf_permute(st["anc"], P, st["perm"])
        pf.pf_gather_inplace(st["states"], P, 4 * case["dim"], st["perm"])
        out["permuted"], out["states"] = st["perm"], st["states"]
    return out


def work(case):
    """Bytes: each input read once, each output written once.  Operations: one
    exponential and one addition per weight summed, one comparison per ancestor;
    for Metropolis a draw, a ratio and a comparison per chain step; for a bootstrap
    step the noise, the transition and the observation density per dimension."""
    form = case["form"]
    if form == "bootstrap":
        n, D = case["F"] * case["P"], LG_D
        steps = case["T"]
        # states out at each step and at the draw, in at each step; log-weights in and out
        return {"bytes": n * 4 * (D + steps * (2 * D + 2)), "flops": n * (steps + 1) * D * 10}
    if form == "batched":
        # log-uniform sizes: the mean of the law
        lo, hi = case["P_lo"], case["P_hi"]
        n = case["F"] * (hi - lo) / math.log(hi / lo)
    else:
        n = case["P"]
    if form == "metropolis" or case.get("kind") == "metropolis":
        return {"bytes": 8 * n, "flops": 4 * n * max(case["B"], 1)}
    if form == "all_four":
        return {"bytes": n * (4 + 4 * 4 + 8 * case["dim"]), "flops": n * (3 * 3 + 4 * case["B"])}
    b = 8 * n
    if case.get("move") == "gather":
        b += n * 8 * case["dim"]
    elif case.get("move") == "inplace":
        # the permuted ancestors, and the rows that change slots (at least one in four) in and out
        b += n * 4 + n * 2 * case["dim"]
    return {"bytes": b, "flops": 3 * n}


# ---------------------------------------------------------------------------
# 64-bit values
# ---------------------------------------------------------------------------
def _mulhilo(a, m):
    """High and low 32 bits of a * m for int64 tensors holding 32-bit values."""
    lo = (a & 0xFFFF) * m
    hi = (a >> 16) * m
    low = lo + ((hi & 0xFFFF) << 16)
    return (hi >> 16) + (low >> 32), low & 0xFFFFFFFF


def _philox(c, key):
    """Philox-4x32-10 on int64 tensors of 32-bit words."""
    k0, k1 = key & 0xFFFFFFFF, (key >> 32) & 0xFFFFFFFF
    c0, c1, c2, c3 = c
    for _ in range(10):
        h0, l0 = _mulhilo(c0, 0xD2511F53)
        h1, l1 = _mulhilo(c2, 0xCD9E8D57)
        c0, c1, c2, c3 = h1 ^ c1 ^ k0, l1, h0 ^ c3 ^ k1, l0
        k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
    return c0, c1, c2, c3


def _normals(F, P, t, seed):
    """The model's four N(0,1) draws per particle at time t, [F, P, 4] float64."""
    j = torch.arange(P, dtype=torch.int64, device="cuda").expand(F, P)
    f = torch.arange(F, dtype=torch.int64, device="cuda")[:, None].expand(F, P)
    w = _philox((j, torch.full_like(j, t), f, torch.full_like(j, 6)), seed)
    u = [((v >> 9) * 2 + 1).double() * 2.0 ** -24 for v in w]
    z = []
    for u0, u1 in ((u[0], u[1]), (u[2], u[3])):
        rad, ang = torch.sqrt(-2.0 * torch.log(u0)), 2.0 * math.pi * u1
        z += [rad * torch.cos(ang), rad * torch.sin(ang)]
    return torch.stack(z, dim=2)


def exact(case, seed):
    form = case["form"]
    if form == "single" and case["ess"]:
        lw = _logw(case, seed).double()
        m = lw.max()
        w = torch.exp(lw - m)
        out = {"ess": (w.sum() ** 2 / (w * w).sum()).reshape(1), "log_sum": (m + torch.log(w.sum())).reshape(1),
               "ancestors": None}
        if case["move"] == "inplace":
            out["permuted"] = None
        if case["move"] != "none":
            out["states"] = None
        return out
    if form == "bootstrap" and case["T"] == 2:
        # the states of the first step, which follow no ancestors; what follows the
        # resampling after it depends on whole-number choices
        F, P = case["F"], case["P"]
        a = torch.from_numpy(workloads.lg_params(F, seed=seed)).cuda().double()[:, None, None]
        x0 = workloads.LG_M0 + math.sqrt(workloads.LG_P0) * _normals(F, P, 0, seed)
        x1 = a * x0 + math.sqrt(workloads.LG_Q) * _normals(F, P, 1, seed)
        return {"states": None, "previous_states": x1, "logw": None, "loglik": None, "log_sum": None, "ess": None,
                "resample": None}
    return None
