"""What this library is measured on: the calls its users make, over the sizes they make them at.

Every case is one pass through a public entry point of the binding (paper_2501_17267_gb300.sg):
annealing (SA), parallel tempering (PT), a batch of uneven instances, a burst of solve
requests to the server, the fragment meta-heuristic with both of its optimisers, and
energies of given configurations.  Instances are tile-planted, or random integer couplings
where the general-coupling path is meant; seeds give the instances, the runs' draws, and
the configurations.
"""
import math

import numpy as np
import torch

from paper_2501_17267_gb300 import sg

F6 = (0.0, 0.0, 1.0)
UNIFORM = (1.0 / 3.0, 1.0 / 3.0, 1.0 / 3.0)

# One Metropolis attempt: six multiply-adds of the local field, the compare, and its share
# of the draw (two ten-round generator blocks, two multiplies and four xors a round, give
# the leading bytes of 32 attempts).
OPS_PER_ATTEMPT = 13.0 + 2 * 10 * 6 / 32.0


def listed():
    return [
        # one small lattice, few replicas: nothing but the latency of 2000 dependent half sweeps
        dict(name="sa_smallest", kind="sa", L=4, I=1, R=8, S=1000, beta0=0.1, beta1=3.0, schedule="linear",
             couplings="planted", spins="host"),
        # many replicas of one lattice, for the distribution of the gap
        dict(name="sa_replicas", kind="sa", L=16, I=1, R=1024, S=1000, beta0=0.1, beta1=3.0, schedule="linear",
             couplings="planted", spins="device"),
        # the time-to-gap protocol: 20 instances of one size in one call, 20 runs each, a short
        # geometric schedule
        dict(name="sa_protocol", kind="sa", L=50, I=20, R=20, S=76, beta0=1.22, beta1=13.6, schedule="geometric",
             couplings="f6", spins="none"),
        # couplings of a user's own (|J| <= 2, absent bonds), a ragged number of replicas
        dict(name="sa_general", kind="sa", L=24, I=1, R=100, S=200, beta0=0.1, beta1=3.0, schedule="linear",
             couplings="general", spins="device"),
        # 512 instances of uneven size and length in one call (sweeps a tenth of the workload's)
        dict(name="sa_uneven", kind="uneven", I=512, R=64, sides="8,12,16,24,32,48", sweeps="10,100,1000",
             beta0=0.1, beta1=3.0),
        # tempering of one small lattice: latency of the sweep and its exchange
        dict(name="pt_small", kind="pt", L=16, I=1, K=32, S=1000, beta0=0.2, beta1=3.0, spins="device"),
        # the throughput workload: 16 large lattices (a fifth of its sweeps)
        dict(name="pt_batch", kind="pt", L=64, I=16, K=32, S=2000, beta0=0.2, beta1=3.0, spins="device"),
        # a ladder longer than one word of 32 slots
        dict(name="pt_wide", kind="pt", L=32, I=4, K=48, S=300, beta0=0.2, beta1=3.0, spins="device"),
        # requests of both kinds and mixed sizes arriving together, each to a gap of 1 % or its cap
        dict(name="serve_burst", kind="serve", n=96, sides="8,16,24,32,40,48,56,64", large=1, R=32, K=32, cap=1000,
             chunk=100),
        # the linear-time meta-heuristic on 20 lattices, cubes annealed
        dict(name="fragments", kind="fragment", L=50, I=20, l=5, S=20, beta0=0.5, beta1=6.0, spins="device"),
        # the same with exact cube minima
        dict(name="fragments_exact", kind="tropical", L=12, I=4, l=3, spins="device"),
        # scoring configurations a user holds on the device
        dict(name="energies", kind="energy", L=64, n=1000),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _even(v):
    return max(2, v - v % 2)


def draw(rng):
    kind = rng.choice(["sa", "sa", "general", "uneven", "pt", "pt", "serve", "fragment", "tropical", "energy"])
    if kind in ("sa", "general"):
        general = kind == "general"
        L = _even(_log(rng, 4, 32 if general else 96))
        I, R = _log(rng, 1, 3 if general else 20), _log(rng, 1, 128 if general else 1024)
        S = _log(rng, 5, 1000)
        most = 5e8 if general else 2e10  # attempts
        S = int(max(3, min(S, most / (I * R * L ** 3))))
        R = int(max(1, min(R, most / (I * S * L ** 3))))
        geo = rng.random() < 0.5
        return dict(kind="sa", L=L, I=I, R=R, S=S, beta0=0.5 if geo else 0.1, beta1=8.0 if geo else 3.0,
                    schedule="geometric" if geo else "linear",
                    couplings="general" if general else rng.choice(["planted", "f6"]),
                    spins=rng.choice(["none", "host", "device"]) if I * R * L ** 3 < 5e7 else "none")
    if kind == "uneven":
        sides = sorted(set(_even(_log(rng, 4, 48)) for _ in range(rng.randint(2, 6))))
        sweeps = sorted(set(_log(rng, 5, 500) for _ in range(rng.randint(1, 3))))
        I, R = _log(rng, 8, 256), _log(rng, 8, 128)
        I = int(max(8, min(I, 1e11 / (max(sides) ** 3 * max(sweeps) * R))))  # attempts
        return dict(kind="uneven", I=I, R=R, sides=",".join(map(str, sides)),
                    sweeps=",".join(map(str, sweeps)), beta0=0.1, beta1=3.0)
    if kind == "pt":
        L, I, K = _even(_log(rng, 4, 64)), _log(rng, 1, 20), _log(rng, 2, 64)
        S = int(max(3, min(_log(rng, 20, 2000), 5e10 / (I * 32 * ((K + 31) // 32) * L ** 3))))
        return dict(kind="pt", L=L, I=I, K=K, S=S, beta0=0.2, beta1=3.0,
                    spins=rng.choice(["none", "host", "device"]) if I * K * L ** 3 < 5e7 else "none")
    if kind == "serve":
        sides = sorted(set(8 * rng.randint(1, 8) for _ in range(rng.randint(2, 8))))
        return dict(kind="serve", n=_log(rng, 4, 96), sides=",".join(map(str, sides)), large=0,
                    R=rng.choice([16, 32, 40]), K=rng.choice([16, 32]), cap=rng.choice([300, 1000]), chunk=100)
    if kind == "fragment":
        l = rng.choice([3, 5, 7])
        L = l * _even(rng.randint(2, 50 // l))
        return dict(kind="fragment", L=L, I=_log(rng, 1, 12), l=l, S=_log(rng, 2, 20 if l < 7 else 8), beta0=0.5,
                    beta1=6.0, spins=rng.choice(["none", "host", "device"]))
    if kind == "tropical":
        L = rng.choice([6, 12, 18])
        return dict(kind="tropical", L=L, I=rng.randint(1, {6: 12, 12: 4, 18: 1}[L]), l=3,
                    spins=rng.choice(["none", "host", "device"]))
    L = _even(_log(rng, 4, 64))
    return dict(kind="energy", L=L, n=int(max(1, min(_log(rng, 1, 4000), 2.6e8 / L ** 3))))


def _instance(L, couplings, seed):
    if couplings == "general":
        J3 = np.random.default_rng(seed).integers(-2, 3, size=(L ** 3, 3), dtype=np.int8)
        return sg.Instance.from_couplings(L, J3, e_gs=-3 * L ** 3)
    return sg.Instance.create(L, seed, F6 if couplings == "f6" else UNIFORM)


def _targets(how, insts, rows):
    """Where a call puts the spins: nowhere, fresh host arrays, or one device tensor an instance."""
    if how == "device":
        return [torch.empty((rows, i.N), dtype=torch.int8, device="cuda") for i in insts]
    return "host" if how == "host" else None


def _uneven(case, seed):
    """(side, sweeps) of each instance, uniform over the case's choices."""
    rng = np.random.default_rng(seed)
    Ls = rng.choice([int(v) for v in case["sides"].split(",")], size=case["I"])
    Ss = rng.choice([int(v) for v in case["sweeps"].split(",")], size=case["I"])
    return [(int(a), int(b)) for a, b in zip(Ls, Ss)]


def _energy_inputs(case, seed):
    L, n = case["L"], case["n"]
    J3 = np.random.default_rng(seed).integers(0, 2, size=(L ** 3, 3), dtype=np.int8) * 2 - 1
    gen = torch.Generator(device="cuda").manual_seed(seed)
    spins = torch.randint(0, 2, (n, L ** 3), dtype=torch.int8, device="cuda", generator=gen) * 2 - 1
    return J3.astype(np.int8), spins


def prepare(case, seed):
    kind = case["kind"]
    base = seed * 2 ** 20  # instance seeds of different cases' seeds do not meet
    if kind == "sa":
        insts = [_instance(case["L"], case["couplings"], base + k) for k in range(case["I"])]
        params = [dict(replicas=case["R"], sweeps=case["S"], beta0=case["beta0"], beta1=case["beta1"],
                       schedule=case["schedule"], seed=seed, instance_id=k) for k in range(case["I"])]
        return dict(case=case, insts=insts, params=params, spins=_targets(case["spins"], insts, case["R"]))
    if kind == "uneven":
        shapes = _uneven(case, seed)
        insts = [_instance(L, "planted", base + k) for k, (L, _) in enumerate(shapes)]
        params = [dict(replicas=case["R"], sweeps=S, beta0=case["beta0"], beta1=case["beta1"], schedule="linear",
                       seed=seed, instance_id=k) for k, (_, S) in enumerate(shapes)]
        return dict(case=case, insts=insts, params=params, spins=None)
    if kind == "pt":
        insts = [_instance(case["L"], "planted", base + k) for k in range(case["I"])]
        params = [dict(temps=case["K"], sweeps=case["S"], beta_min=case["beta0"], beta_max=case["beta1"], seed=seed,
                       instance_id=k) for k in range(case["I"])]
        return dict(case=case, insts=insts, params=params, spins=_targets(case["spins"], insts, case["K"]))
    if kind == "serve":
        rng = np.random.default_rng(seed)
        sides = [int(v) for v in case["sides"].split(",")]
        reqs = []
        for k in range(case["n"]):
            L = 128 if k < case["large"] else int(rng.choice(sides))
            sa = bool(rng.random() < 0.5)
            reqs.append(sg.request(sg.SG_REQ_SA if sa else sg.SG_REQ_PT, L, base + k,
                                   case["R"] if sa else case["K"], 0.1 if sa else 0.2, 3.0, 0.01, case["cap"],
                                   run_seed=seed + k))
        server = sg.Server(8 << 30, max_active=256, chunk_sweeps=case["chunk"])
        return dict(case=case, server=server, reqs=reqs)
    if kind in ("fragment", "tropical"):
        insts = [_instance(case["L"], "f6", base + k) for k in range(case["I"])]
        params = [dict(l=case["l"], sweeps=case.get("S", 0), beta0=case.get("beta0", 1.0),
                       beta1=case.get("beta1", 1.0), seed=seed, instance_id=k) for k in range(case["I"])]
        return dict(case=case, insts=insts, params=params, spins=_targets(case["spins"], insts, 1))
    J3, spins = _energy_inputs(case, seed)
    return dict(case=case, inst=sg.Instance.from_couplings(case["L"], J3), spins=spins)


def run(state):
    kind = state["case"]["kind"]
    if kind in ("sa", "uneven"):
        res = sg.sa_run_batch(state["insts"], state["params"], spins=state["spins"])
        out = dict(E=np.concatenate([r["E"] for r in res]), eps=np.concatenate([r["eps"] for r in res]))
    elif kind == "pt":
        res = sg.pt_run_batch(state["insts"], state["params"], spins=state["spins"])
        out = dict(E=np.concatenate([r["E"] for r in res]), perm=np.concatenate([r["perm"] for r in res]),
                   accepts=np.concatenate([r["accepts"] for r in res]),
                   minE=np.array([r["minE"] for r in res], dtype=np.int64),
                   min_eps=np.array([r["min_eps"] for r in res]))
    elif kind in ("fragment", "tropical"):
        res = sg.fragment_run_batch(state["insts"], state["params"], spins=state["spins"],
                                    tropical=kind == "tropical")
        out = dict(E=np.array([r["E"] for r in res], dtype=np.int64), eps=np.array([r["eps"] for r in res]))
    elif kind == "serve":
        server = state["server"]
        tickets = [server.submit(q) for q in state["reqs"]]
        res = [server.poll(t) for t in tickets]
        return dict(status=np.array([r["status"] for r in res]), reached=np.array([r["reached"] for r in res]),
                    sweeps=np.array([r["sweeps"] for r in res], dtype=np.int64),
                    minE=np.array([r["minE"] for r in res], dtype=np.int64),
                    e_gs=np.array([r["e_gs"] for r in res], dtype=np.int64),
                    min_eps=np.array([r["min_eps"] for r in res]))
    else:
        return sg.energy(state["inst"], state["spins"])
    if state["spins"] is not None:
        out["spins"] = [r["spins"] for r in res]
    return out


def work(case):
    """Couplings (three bytes a site) and outputs once; the operations of every attempt."""
    kind = case["kind"]
    if kind == "uneven":
        sides = [int(v) for v in case["sides"].split(",")]
        sweeps = [int(v) for v in case["sweeps"].split(",")]
        N = case["I"] * sum(L ** 3 for L in sides) / len(sides)
        return dict(bytes=3 * N + 16 * case["I"] * case["R"],
                    flops=OPS_PER_ATTEMPT * N * case["R"] * sum(sweeps) / len(sweeps))
    if kind == "serve":  # at least one chunk of every request
        sides = [int(v) for v in case["sides"].split(",")]
        N = (case["n"] - case["large"]) * sum(L ** 3 for L in sides) / len(sides) + case["large"] * 128 ** 3
        return dict(bytes=3 * N + 40 * case["n"],
                    flops=OPS_PER_ATTEMPT * N * 0.5 * (case["R"] + case["K"]) * min(case["chunk"], case["cap"]))
    L = case["L"]
    N = L ** 3
    if kind == "energy":
        return dict(bytes=3 * N + N * case["n"] + 8 * case["n"], flops=6.0 * N * case["n"])
    I = case["I"]
    rows = case.get("R") or case.get("K") or 1
    out = 16 * I * rows + (0 if case["spins"] == "none" else I * rows * N)
    if kind in ("sa", "pt"):
        return dict(bytes=3 * N * I + out, flops=OPS_PER_ATTEMPT * I * N * rows * case["S"])
    V = case["l"] ** 3
    cubes = I * N // V
    if kind == "fragment":  # wave w anneals the V - w spins still free, 32 reads a cube
        return dict(bytes=3 * N * I + out, flops=OPS_PER_ATTEMPT * cubes * 32.0 * case["S"] * V * (V + 1) / 2)
    # exact cube minima: spins eliminated one after another, each leaving a table over the
    # l^2 (or fewer) spins it still touches: two additions and a minimum an entry
    free = sum(3.0 * 2 ** min(f - k - 1, case["l"] ** 2) for f in range(1, V + 1) for k in range(f))
    return dict(bytes=3 * N * I + out, flops=cubes * free)


def exact(case, seed):
    """Energies straight from their definition (Eq. 1), in 64 bits.  The other cases return
    whole numbers that follow from the draws bit by bit, and gaps made from those."""
    if case["kind"] != "energy":
        return None
    L, n = case["L"], case["n"]
    J3, spins = _energy_inputs(case, seed)
    J = torch.from_numpy(J3).cuda().view(L, L, L, 3).to(torch.float64)
    out = []
    for a in range(0, n, 64):
        s = spins[a:a + 64].view(-1, L, L, L).to(torch.float64)
        E = sum((J[..., d] * s * torch.roll(s, -1, dims=3 - d)).sum(dim=(1, 2, 3)) for d in range(3))
        out.append(E.to(torch.int64).cpu().numpy())
    return np.concatenate(out)
