"""The performance cases: what a program that uses the sampler has it do.

One pass is what such a program runs between two looks at its chains: some
sweeps (or block-move passes, or training steps) through the public Python
interface, then the results read back into host buffers that the program
keeps.  Chains, parameter grids and ladders are those of
paper_2511_20911_gb300/workloads.py and of bench.py, in sizes that keep one
pass at a few milliseconds.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2511_20911_gb300 as crbm
from paper_2511_20911_gb300 import workloads

EXACT, PAPER, BITPLANE = "exact", "paper", "bitplane"


def listed():
    return [
        # A quick look at a handful of chains on the smallest lattice in use (36 spins, 64 chains, one
        # point, every sweep measured): launch and half-step latency, almost no parallel work.
        dict(name="small", kind="sweep", L=6, cols=6, chains=64, n_beta=1, n_h=1, mode=EXACT, measure=1, sq=0,
             sweeps=200),
        # The 18 x 18 parameter grid (3 couplings x 16 beta x 16 h x 16 chains) with its observables every
        # 10 sweeps and its structure-factor sums every 100: the sampler's main use.
        dict(name="grid", kind="sweep", L=18, cols=18, chains=12288, n_beta=16, n_h=16, mode=EXACT, measure=10,
             sq=100, sweeps=500),
        # The same grid in the arithmetic of the paper's FPGA, to compare with its results.
        dict(name="grid_paper", kind="sweep", L=18, cols=18, chains=12288, n_beta=16, n_h=16, mode=PAPER, measure=10,
             sq=100, sweeps=500),
        # The same grid with bit-plane uniforms, the mode for the most spin updates a second.
        dict(name="grid_bitplane", kind="sweep", L=18, cols=18, chains=12288, n_beta=16, n_h=16, mode=BITPLANE,
             measure=10, sq=0, sweeps=500),
        # Ground-state search by replica exchange at L = 18: three phase points x 32 ladders of 32 rungs,
        # measured after every sweep against target energies, exchanges every second sweep.
        dict(name="ladders", kind="ladder", L=18, ladders=96, swap=2, measure=1, mode=EXACT, sweeps=400),
        # The laterally confined strip (18 periodic rows, 12 open columns): the general-lattice sweep.
        dict(name="strip", kind="lattice", L=18, cols=12, rows_periodic=True, cols_periodic=False, chains=1536,
             mode=EXACT, measure=10, sweeps=200),
        # Parallel tempering on mixed sizes, odd ones among them, in one launch.
        dict(name="batch", kind="batch", sizes="6,9,12,18,24,48", ladders=8, sweeps=100),
        # A lattice too large for shared memory, spins and hidden units in device memory.
        dict(name="stream", kind="stream", L=384, cols=384, chains=768, mode=EXACT, measure=10, sweeps=20),
        # The same layout with bit-plane uniforms on a ragged rectangle and a chain count that fills no
        # whole number of 64-chain words.
        dict(name="stream_bitplane", kind="stream", L=250, cols=198, chains=1000, mode=BITPLANE, measure=10,
             sweeps=20),
        # Gibbs sweeps mixed with learned block moves, a pass after every 4 sweeps, L = 18 at the
        # evaluation points.
        dict(name="mixed", kind="mixed", L=18, chains=4096, sweeps=40, every=4),
        # Training the block proposal on the sampler's own chains.
        dict(name="train", kind="train", L=18, chains=4096, steps=4, batch=4096),
        # Loss and gradient of the proposal's net on examples the program holds.
        dict(name="loss_grad", kind="loss_grad", L=18, n=2048),
    ]


def _log_int(rng, lo, hi, step=1):
    """An integer multiple of `step` in [lo, hi], spread over the logarithm."""
    x = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    return max(lo, min(hi, int(round(x / step)) * step))


def _cap(spins, chains, sweeps, budget):
    """Sweeps such that spins x chains x sweeps stays within the budget."""
    return max(1, min(sweeps, int(budget / (spins * chains))))


def draw(rng):
    kind = rng.choice(["sweep", "sweep", "sweep", "ladder", "lattice", "batch", "stream", "stream", "mixed", "train",
                       "loss_grad"])
    if kind == "sweep":
        L = _log_int(rng, 4, 64, 2)
        cols = L if rng.random() < 0.6 else _log_int(rng, 4, 64, 2)
        n_beta, n_h = rng.randint(1, 16), rng.randint(1, 16)
        chains = _log_int(rng, 33, 12288)
        mode = rng.choice([EXACT, EXACT, PAPER, BITPLANE])
        sq = rng.choice([0, 50, 100]) if mode != BITPLANE and cols == L and L <= 32 else 0
        return dict(kind=kind, L=L, cols=cols, chains=chains, n_beta=n_beta, n_h=n_h, mode=mode,
                    measure=rng.choice([1, 5, 10]), sq=sq,
                    sweeps=_cap(L * cols, chains, _log_int(rng, 1, 500), 1.2e9))
    if kind == "ladder":
        L = _log_int(rng, 6, 36, 2)
        ladders = _log_int(rng, 1, 128)
        return dict(kind=kind, L=L, ladders=ladders, swap=rng.choice([1, 2, 5, 10]), measure=rng.choice([1, 2, 10]),
                    mode=rng.choice([EXACT, EXACT, PAPER, BITPLANE]),
                    sweeps=_cap(L * L, 32 * ladders, _log_int(rng, 10, 400), 5e8))
    if kind == "lattice":
        L, cols = _log_int(rng, 4, 40), _log_int(rng, 4, 40)
        rows_p, cols_p = rng.choice([(True, False), (False, True), (False, False), (True, True)])
        if rows_p and cols_p and L % 2 == 0 and cols % 2 == 0:
            L -= 1 if L > 4 else -1  # an even periodic lattice is not what this kind stands for
        chains = _log_int(rng, 33, 4096)
        return dict(kind=kind, L=L, cols=cols, rows_periodic=rows_p, cols_periodic=cols_p, chains=chains,
                    mode=rng.choice([EXACT, EXACT, PAPER]), measure=rng.choice([1, 10]),
                    sweeps=_cap(L * cols, chains, _log_int(rng, 10, 200), 1.5e8))
    if kind == "batch":
        sizes = rng.sample([6, 8, 9, 10, 12, 15, 18, 24, 30, 36, 48], rng.randint(2, 6))
        ladders = rng.randint(1, 8)
        return dict(kind=kind, sizes=",".join(str(x) for x in sorted(sizes)), ladders=ladders,
                    sweeps=rng.randint(10, 100))
    if kind == "stream":
        L, cols = _log_int(rng, 64, 384, 2), _log_int(rng, 64, 384, 2)
        chains = _log_int(rng, 64, 1024)
        return dict(kind=kind, L=L, cols=cols, chains=chains, mode=rng.choice([EXACT, PAPER, BITPLANE]),
                    measure=rng.choice([1, 10]), sweeps=_cap(L * cols, chains, rng.randint(2, 20), 1.2e9))
    if kind == "mixed":
        L = _log_int(rng, 10, 48, 2)
        chains = _log_int(rng, 64, 4096)
        return dict(kind=kind, L=L, chains=chains, sweeps=_cap(L * L, chains, rng.randint(4, 40), 3e8),
                    every=rng.choice([1, 2, 4, 8]))
    if kind == "train":
        return dict(kind=kind, L=rng.choice([10, 12, 18, 24]), chains=_log_int(rng, 256, 4096),
                    steps=rng.randint(1, 4), batch=_log_int(rng, 100, 4096))
    return dict(kind=kind, L=rng.choice([10, 12, 18, 24]), n=_log_int(rng, 100, 2048))


# ------------------------------------------------------------------ inputs


def _modes(case):
    return dict(precision=crbm.CRBM_PRECISION_PAPER if case["mode"] == PAPER else crbm.CRBM_PRECISION_EXACT,
                rng=crbm.CRBM_RNG_BITPLANE if case["mode"] == BITPLANE else crbm.CRBM_RNG_LANE)


def _host(shape, dtype):
    """A pinned host buffer, as a program that reads its chains back often keeps one."""
    t = torch.empty(shape, dtype=dtype, pin_memory=True)
    return t.numpy()


def _buffers(s):
    return dict(spins=_host((s.n_chains, s.L, s.L_cols), torch.int8), sums=_host((s.n_chains, crbm.CRBM_NSUM), torch.int64))


def _grid_points(case):
    """J'/J in {0.5, 1, 2} (one of them for a single point) x beta in [0.1, 5] x h in [0, 4]."""
    ratios = (0.5, 1.0, 2.0) if case["n_beta"] * case["n_h"] > 1 else (1.0,)
    betas = np.linspace(0.1, 5.0, case["n_beta"]) if case["n_beta"] > 1 else np.array([2.0])
    hs = workloads.q4(np.linspace(0.0, 4.0, case["n_h"])) if case["n_h"] > 1 else np.array([0.5])
    pts = [(r, b, h) for r in ratios for b in betas for h in hs]
    return dict(J=[1.0] * len(pts), Jp=[float(r) for r, _, _ in pts], h=[float(h) for _, _, h in pts],
                beta=[float(b) for _, b, _ in pts]), len(pts)


def _contiguous(chains, points):
    return (np.arange(chains, dtype=np.int64) * points // chains).astype(np.int32)


# (J', h, energy per spin in units of J): the Neel, dimer and ferromagnetic ground states
_PHASES = [(1.0, 0.0, -1.5), (2.5, 0.0, -1.25), (1.0, 7.0, -4.5)]


def _ladder_state(case, seed):
    L, ladders = case["L"], case["ladders"]
    betas = 0.25 * 32.0 ** (np.arange(32) / 31.0)
    params = dict(J=[1.0] * 96, Jp=[p[0] for p in _PHASES for _ in range(32)], h=[p[1] for p in _PHASES for _ in range(32)],
                  beta=[float(b) for _ in _PHASES for b in betas])
    cp = np.concatenate([np.arange(32, dtype=np.int32) + 32 * (k * 3 // ladders) for k in range(ladders)])
    s = crbm.Sampler(L, params, 32 * ladders, chain_param=cp, seed=seed, measure_every=case["measure"],
                     swap_every=case["swap"], **_modes(case))
    s.set_targets([int(round(16 * p[2] * L * L)) for p in _PHASES for _ in range(32)])
    return dict(s=s, **_buffers(s))


def _proposal_sampler(case, seed, points):
    L, chains = case["L"], case["chains"]
    w = workloads.proposal_eval_workload(L, chains) if points == "eval" else workloads.proposal_training_workload(L, chains)
    s = crbm.Sampler(L, w["params"], chains, chain_param=w["chain_param"], seed=seed, measure_every=0)
    s.sweep(20)
    return s


def _examples(case, seed):
    """Configurations with domains of the up-up-down and Neel patterns (what the chains near the
    plateau look like), random block origins, and the training points' beta and h."""
    L, n = case["L"], case["n"]
    rng = np.random.default_rng(seed)
    r = np.arange(L)
    uud = np.where((r[None, :] % 3) == 2, -1, 1).repeat(L, 0).reshape(L, L)
    neel = np.where((r[:, None] + r[None, :]) % 2 == 0, 1, -1)
    base = np.stack([uud, neel]).astype(np.int8)[rng.integers(0, 2, n)]
    flips = np.where(rng.random((n, L, L)) < 0.1, -1, 1).astype(np.int8)
    spins = np.ascontiguousarray(base * flips)
    origins = rng.integers(0, L, (n, 2)).astype(np.int32)
    beta_h = np.stack([rng.choice([1.5, 2.0, 2.5, 3.0], n), rng.choice([2.5, 2.75, 3.0, 3.25, 3.5], n)], 1).astype(np.float32)
    return spins, origins, beta_h


def _net_weights(seed):
    """Weights of a partly trained net: the initial scales, the last layer and the biases away from zero."""
    rng = np.random.default_rng(seed + 1)
    w = np.zeros(crbm.NET_PARAMS, np.float64)
    w[:864] = rng.normal(0.0, math.sqrt(2 / 54), 864)
    w[864:880] = rng.normal(0.0, 0.05, 16)
    w[880:3184] = rng.normal(0.0, math.sqrt(2 / 144), 2304)
    w[3184:3200] = rng.normal(0.0, 0.05, 16)
    w[3200:3344] = rng.normal(0.0, 0.1, 144)
    w[3344] = 0.02
    return w.astype(np.float32)


def _state(case, seed):
    kind = case["kind"]
    if kind == "sweep":
        params, points = _grid_points(case)
        s = crbm.Sampler(case["L"], params, case["chains"], chain_param=_contiguous(case["chains"], points), seed=seed,
                         measure_every=case["measure"], sq_every=case["sq"], L_cols=0 if case["cols"] == case["L"] else case["cols"],
                         **_modes(case))
        return dict(s=s, **_buffers(s))
    if kind == "ladder":
        return _ladder_state(case, seed)
    if kind == "lattice":
        w = workloads.strip_workload(chains_per_point=1)
        points = len(w["params"]["J"])
        s = crbm.Sampler(case["L"], w["params"], case["chains"], chain_param=_contiguous(case["chains"], points), seed=seed,
                         periodic=case["rows_periodic"], L_cols=case["cols"],
                         periodic_cols=crbm.CRBM_BC_PERIODIC if case["cols_periodic"] else crbm.CRBM_BC_OPEN,
                         measure_every=case["measure"], **_modes(case))
        return dict(s=s, **_buffers(s))
    if kind == "batch":
        sizes = [int(x) for x in case["sizes"].split(",")]
        members = []
        for m in workloads.tempering_batch_workload(sizes, case["ladders"]):
            members.append(crbm.Sampler(m["L"], m["params"], m["n_chains"], chain_param=m["chain_param"],
                                        seed=m["seed"] + seed, measure_every=10, swap_every=m["swap_every"]))
        return dict(batch=crbm.Batch(members), members=[dict(s=s, **_buffers(s)) for s in members])
    if kind == "stream":
        params = dict(J=[1.0] * 3, Jp=[1.0] * 3, h=[0.0, 1.0, 2.0], beta=[1.0] * 3)
        s = crbm.Sampler(case["L"], params, case["chains"], chain_param=_contiguous(case["chains"], 3), seed=seed,
                         measure_every=case["measure"], layout=crbm.CRBM_LAYOUT_STREAM,
                         L_cols=0 if case["cols"] == case["L"] else case["cols"], **_modes(case))
        return dict(s=s, **_buffers(s))
    if kind == "mixed":
        s = _proposal_sampler(case, seed, "eval")
        p = crbm.Proposal(seed=1)
        p.weights = _net_weights(3)
        return dict(s=s, p=p, **_buffers(s))
    if kind == "train":
        return dict(s=_proposal_sampler(case, seed, "train"), p=crbm.Proposal(seed=seed % 1000))
    spins, origins, beta_h = _examples(case, seed)
    p = crbm.Proposal(seed=1)
    p.weights = _net_weights(seed)
    return dict(p=p, spins=spins, origins=origins, beta_h=beta_h)


def prepare(case, seed):
    return dict(_state(case, seed), case=case)


# -------------------------------------------------------------------- pass


def _read(st):
    return dict(spins=st["s"].get_spins(out=st["spins"]), sums=st["s"].observables(out=st["sums"]))


def run(state):
    case, kind = state["case"], state["case"]["kind"]
    if kind == "batch":
        state["batch"].sweep(case["sweeps"])
        return [dict(_read(m), slots=m["s"].permutation()) for m in state["members"]]
    if kind == "train":
        losses = state["p"].train(state["s"], steps=case["steps"], batch=case["batch"], lr=1e-2, sweeps_between=2)
        return dict(losses=losses, weights=state["p"].weights)
    if kind == "loss_grad":
        loss, grad = state["p"].loss_grad(state["spins"], state["origins"], state["beta_h"])
        return dict(loss=loss, grad=grad)
    s = state["s"]
    if kind == "mixed":
        state["p"].sweep_mixed(s, case["sweeps"], every=case["every"])
        return dict(spins=s.get_spins(out=state["spins"]))
    s.sweep(case["sweeps"])
    out = _read(state)
    if kind == "ladder":
        out.update(slots=s.permutation(), hits=s.first_hits())
    if kind == "sweep" and case["sq"]:
        out["correlations"] = s.correlations()
    return out


# -------------------------------------------------------------------- work
# "flops" counts the integer multiply operations of the uniforms (a Philox-4x32-10
# call is 20 products of 32 x 32 -> 64 bits, two operations each) and the
# floating operations of the nets.

_CALLS = {EXACT: 4.0, PAPER: 2.0, BITPLANE: 1.0}  # per chain and cell of 4 spins and 10 filters
_NET = 2.0 * (16 * 64 * 54 + 16 * 36 * 144 + 16 * 144)  # one forward pass of the net on one block


def _sweep_work(spins, chains, sweeps, calls):
    state = 2 * chains * spins / 8.0
    return state + chains * (spins + 88.0), 40.0 * calls * chains * sweeps * spins / 4.0


def work(case):
    kind = case["kind"]
    if kind == "batch":
        b = f = 0.0
        for L in (int(x) for x in case["sizes"].split(",")):
            x, y = _sweep_work(L * L, 32 * case["ladders"], case["sweeps"], 4.0)
            b, f = b + x, f + y
        return {"bytes": b, "flops": f}
    if kind == "ladder":
        b, f = _sweep_work(case["L"] ** 2, 32 * case["ladders"], case["sweeps"], _CALLS[case["mode"]])
        return {"bytes": b, "flops": f}
    if kind in ("sweep", "lattice", "stream"):
        b, f = _sweep_work(case["L"] * case["cols"], case["chains"], case["sweeps"], _CALLS[case["mode"]])
        if case.get("sq"):
            b += 8.0 * case["L"] * case["cols"] * min(case["chains"], 3 * case["n_beta"] * case["n_h"])
        return {"bytes": b, "flops": f}
    if kind == "mixed":
        b, f = _sweep_work(case["L"] ** 2, case["chains"], case["sweeps"], 4.0)
        passes = -(-case["sweeps"] // case["every"])
        return {"bytes": b, "flops": f + passes * case["chains"] * max(1, case["L"] // 8) ** 2 * _NET}
    if kind == "train":
        b, f = _sweep_work(case["L"] ** 2, case["chains"], 2 * case["steps"], 4.0)
        return {"bytes": case["steps"] * case["batch"] * 116 / 8.0 + 7 * 4.0 * crbm.NET_PARAMS,
                "flops": f + 3 * case["steps"] * case["batch"] * _NET}
    return {"bytes": case["n"] * (case["L"] ** 2 + 16.0) + 8.0 * crbm.NET_PARAMS, "flops": 3 * case["n"] * _NET}


# ------------------------------------------------------------------- exact


class _Bf16(torch.autograd.Function):
    """Rounding of a double to bfloat16 (nearest even), gradients straight through."""

    @staticmethod
    def forward(ctx, x):
        return x.to(torch.float32).to(torch.bfloat16).to(torch.float64)

    @staticmethod
    def backward(ctx, g):
        return g


def exact(case, seed):
    """The net's loss and gradient in 64 bits (weights and activations rounded to bfloat16, as the
    method defines them); the other kinds return whole numbers, or train on the chains' own states."""
    if case["kind"] != "loss_grad":
        return None
    spins, origins, beta_h = (torch.from_numpy(x) for x in _examples(case, seed))
    L, n = case["L"], case["n"]
    k = torch.arange(10)
    rows, cols = (origins[:, :1].long() - 3 + k) % L, (origins[:, 1:].long() - 3 + k) % L
    patch = spins.double()[torch.arange(n)[:, None, None], rows[:, :, None], cols[:, None, :]]
    # inside the block, by position on the lattice (a patch may wrap onto its own block)
    in_r = ((rows - origins[:, :1].long()) % L) < 4
    in_c = ((cols - origins[:, 1:].long()) % L) < 4
    mask = (in_r[:, :, None] & in_c[:, None, :]).double()
    pr = (((origins[:, :1].long() + 1) & 1) + k) & 1
    pc = (((origins[:, 1:].long() + 1) & 1) + k) & 1
    plane = torch.ones(n, 10, 10, dtype=torch.float64)
    x = torch.stack([patch * (1 - mask), mask, plane * pr[:, :, None], plane * pc[:, None, :],
                     plane * beta_h[:, 0, None, None].double(), plane * beta_h[:, 1, None, None].double()], 1)
    target = (patch[:, 3:7, 3:7] > 0).double()
    w = _Bf16.apply(torch.from_numpy(_net_weights(seed)).double()).requires_grad_(True)
    conv = torch.nn.functional.conv2d
    a1 = _Bf16.apply(conv(x, w[:864].view(16, 6, 3, 3), w[864:880]).relu())
    a2 = _Bf16.apply(conv(a1, w[880:3184].view(16, 16, 3, 3), w[3184:3200]).relu())
    logit = conv(a2, w[3200:3344].view(1, 16, 3, 3), w[3344:3345])[:, 0]
    loss = torch.nn.functional.binary_cross_entropy_with_logits(logit, target)
    loss.backward()
    return dict(loss=loss.item(), grad=w.grad.numpy())
