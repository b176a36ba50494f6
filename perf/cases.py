"""The calls that a variational Monte Carlo program makes of this library, at the sizes it makes them.

``listed()`` names them, ``draw(rng)`` gives more of the same ranges, ``prepare`` makes the inputs
and the handle that the program has in hand, ``run`` is one pass through the public entry points,
``work`` the least bytes and operations of a pass, and ``exact`` the same results in 64 bits from
plain torch.

A VMC program alternates between sampling |psi|^2 (value-only forwards, many per optimisation
step), the local energies of the samples (value, gradient and Laplacian together) and the gradient
of the loss in the parameters (summed over the walkers, or per walker for the natural gradient).
Parameters are a run's initial ones, and walkers are Metropolis samples of the |psi|^2 that they
give, drawn here by plain torch so that they follow from the seed alone.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_2307_14123_gb300 import Ansatz, AnsatzBatch
from paper_2307_14123_gb300 import binding
from paper_2307_14123_gb300 import fixtures as fx

DEVICE = "cuda"
N_RBF, CUTOFF = 16, 10.0
SWEEPS = 80  # Metropolis sweeps from the placement by charge to the walkers of a case
MIXED = ("H2O", "NH3", "C2H4", "C6H6")  # the molecules of a batch
CG_ITERS = 200


def listed():
    return [
        # Local energies of a full batch of walkers, once per optimisation step: the main call.
        _case("energy_n2", "energy", "N2", 4096, 128, 3, 16),
        # The same call on a few walkers (a debugging run, the last part of a sample, one
        # molecule of many): an odd count that leaves most of the chip idle.
        _case("energy_n2_few", "energy", "N2", 77, 128, 3, 16),
        # The forward of every sampling sweep and of every wave-function ratio: value only.
        _case("eval_n2", "eval", "N2", 4096, 128, 3, 16),
        # The gradient of the loss, once per optimisation step of a first-order optimiser.
        _case("grad_n2", "grad", "N2", 4096, 128, 3, 16),
        # Per-walker gradients, the input of the natural gradient; a ragged count.
        _case("walker_grads_h2o", "walker_grads", "H2O", 501, 128, 3, 8),
        # The natural-gradient direction from those gradients.
        _case("natural_n2", "natural", "N2", 1024, 128, 3, 16),
        # Ten sampling sweeps of a small molecule in 64 bits: launches and latency.
        _case("sample_lih", "sample", "LiH", 512, 32, 2, 1, precision="fp64"),
        # A whole training step of a small molecule: sampler, energies, weights, per-walker
        # gradients, natural gradient, update.
        _case("train_lih", "train", "LiH", 1024, 64, 2, 1),
        # One step of training one ansatz shape on several molecules at once: energies, loss
        # weights and gradients of uneven molecules (10, 10, 16 and 42 electrons).
        _case("batch_mixed", "batch", "mixed", 1000, 128, 3, 8),
        # A larger molecule and network in the mixed-precision mode: the most work.
        _case("energy_c4h4_bf16", "energy", "C4H4", 1024, 256, 4, 32, precision="bf16"),
        # The same class of molecule in FP32, on fewer walkers.
        _case("energy_c4h4", "energy", "C4H4", 333, 256, 4, 32),
        # The other ansatz options together: one determinant of all electrons, iterated edge
        # embeddings, initial embeddings from the nuclei.
        _case("energy_c2h4_options", "energy", "C2H4", 1001, 128, 3, 8, full_det=1, edge_update=1, el_init=1),
    ]


def _case(name, op, molecule, walkers, width, layers, dets, precision="fp32", full_det=0, edge_update=0, el_init=0):
    return {"name": name, "op": op, "molecule": molecule, "walkers": walkers, "width": width, "layers": layers,
            "dets": dets, "precision": precision, "full_det": full_det, "edge_update": edge_update,
            "el_init": el_init}


def draw(rng):
    """One more case: an operation, a molecule, a precision and log-uniform sizes of the listed
    ranges, with at most the work of the largest listed case (64-bit work, which runs about
    fifty times slower, at most a hundredth of it)."""
    most = work(next(c for c in listed() if c["name"] == "energy_c4h4_bf16"))["flops"]
    while True:
        op = rng.choice(["energy"] * 4 + ["eval"] * 2 + ["grad"] * 2 + ["walker_grads", "natural", "batch", "sample"])
        precision = rng.choice(["fp32"] * 5 + ["bf16", "fp64"])
        molecule = rng.choice(["LiH", "H2O", "NH3", "N2", "C2H4", "C4H4", "C6H6"])
        width = rng.choice([32, 64, 96, 128, 128, 128, 192, 256])
        layers, dets = rng.randint(2, 4), rng.choice([1, 4, 8, 16, 16, 32])
        walkers = int(round(math.exp(rng.uniform(math.log(40), math.log(4096)))))
        options = rng.random() < 0.25 and molecule not in ("C6H6",)
        flags = [rng.randint(0, 1) if options else 0 for _ in range(3)]
        if op == "batch":
            molecule, flags, width, dets = "mixed", [0, 0, 0], rng.choice([64, 128]), rng.choice([4, 8])
            precision = "fp32"
        if op == "sample":
            precision, molecule = "fp64", rng.choice(["LiH", "H2O"])
            width, layers, dets = 32, 2, rng.choice([1, 2, 4])
            walkers = max(64, walkers // 4)
        if op == "natural":
            precision = "fp32"
            walkers = max(64, walkers // 2)
        if op == "walker_grads":
            walkers = max(16, walkers // 8)
        if precision == "bf16":
            width = max(64, width // 64 * 64)
            if op in ("walker_grads", "grad"):
                precision = "fp32"  # the mode changes the forward's GEMMs only
        if precision == "fp64":
            width, molecule, dets = min(width, 64), rng.choice(["LiH", "H2O"]), min(dets, 4)
        case = _case("", op, molecule, walkers, width, layers, dets, precision, *flags)
        del case["name"]
        f = work(case)["flops"]
        state = work(case)["bytes"]
        if f <= most * (0.01 if precision == "fp64" else 0.5) and state < 4e9:
            return case


# ----------------------------------------------------------------------------
# Inputs
# ----------------------------------------------------------------------------
def _parts(case):
    """(molecule, walkers) of every molecule of a case: one, or the batch's four, the larger ones
    with fewer walkers."""
    if case["molecule"] != "mixed":
        return [(case["molecule"], case["walkers"])]
    share = {"H2O": 1.0, "NH3": 1.0, "C2H4": 0.5, "C6H6": 0.25}
    return [(m, max(1, int(case["walkers"] * share[m]))) for m in MIXED]


def _cfg(case):
    return fx.AnsatzCfg(case["width"], case["layers"], case["dets"], N_RBF, CUTOFF, full_det=case["full_det"],
                        edge_update=case["edge_update"], el_init=case["el_init"])


def _layout(case, system):
    """Blocks of the flat parameter vector: (name, shape, how it is drawn)."""
    D, K, Q, M = case["width"], case["dets"], N_RBF, system.n_nuc
    out = ([("W_e1", (D, 3 * M), "matrix"), ("b_e1", (D,), "zero"), ("W_e2", (D, D), "matrix"), ("b_e2", (D,), "zero")]
           if case["el_init"] else [("E_spin", (2, D), "normal")])
    for l in range(case["layers"]):
        out.append((f"W_h{l}", (D, D), "matrix"))
        for t in range(3):
            if case["edge_update"] and l:
                out += [(f"U{t}{l}", (Q, Q), "matrix"), (f"c{t}{l}", (Q,), "zero")]
            out += [(f"W1{t}{l}", (D, Q), "matrix"), (f"b1{t}{l}", (D,), "zero"), (f"W2{t}{l}", (D, D), "matrix"),
                    (f"b2{t}{l}", (D,), "zero")]
        out += [(f"Y{l}", (M, D), "normal"), (f"W_g{l}", (D, 3 * D), "matrix"), (f"b_g{l}", (D,), "zero")]
    for s, n in enumerate((system.n_up, system.n_down)):
        n = K * (system.n_elec if case["full_det"] else n)
        out += [(f"W_o{s}", (n, D), "matrix"), (f"b_o{s}", (n,), "zero"), (f"omega{s}", (n, M), "one"),
                (f"zeta{s}", (n, M), "exponent")]
    return out + [("c", (K,), "one"), ("W_J1", (D, D), "matrix"), ("b_J1", (D,), "zero"), ("w_J2", (1, D), "matrix")]


def _count(case, system):
    return sum(math.prod(shape) for _, shape, _ in _layout(case, system))


def _dtype(case):
    return torch.float64 if case["precision"] == "fp64" else torch.float32


def _params(case, system, rng):
    """Xavier matrices, normal embeddings, no biases, exponents in (0.5, 2)."""
    out = []
    for _, shape, kind in _layout(case, system):
        n = math.prod(shape)
        if kind == "zero":
            out.append(np.zeros(n))
        elif kind == "one":
            out.append(np.ones(n))
        elif kind == "exponent":
            out.append(rng.uniform(0.5, 2.0, n))
        else:
            std = 1.0 if kind == "normal" else math.sqrt(2.0 / sum(shape))
            out.append(std * rng.standard_normal(n))
    return torch.as_tensor(np.concatenate(out), device=DEVICE).to(_dtype(case))


def _walkers(case, system, theta, B, rng):
    """B Metropolis samples of |psi|^2, SWEEPS sweeps from the placement by charge."""
    N = system.n_elec
    start = system.R[fx.electron_slots(system)][None] + rng.standard_normal((B, N, 3))
    dtype = _dtype(case)
    r = torch.as_tensor(start, device=DEVICE).to(dtype)
    with torch.no_grad():
        th = _blocks(case, system, theta)
        size = _chunk(case, system, 1)
        steps = rng.standard_normal((SWEEPS, B, N, 3), dtype=np.float32)
        logu = np.log(rng.random((SWEEPS, B)))
        for b in range(0, B, size):
            x = r[b:b + size]
            now = _log_psi(case, system, th, x)[0]
            for k in range(SWEEPS):
                y = x + 0.6 / math.sqrt(N) * torch.as_tensor(steps[k, b:b + size], device=DEVICE).to(dtype)
                new = _log_psi(case, system, th, y)[0]
                yes = torch.as_tensor(logu[k, b:b + size], device=DEVICE) < 2 * (new - now).double()
                x = torch.where(yes[:, None, None], y, x)
                now = torch.where(yes, new, now)
            r[b:b + size] = x
    return r


def _loss_weights(case, B, rng):
    """Weights of the loss gradient: centred, clipped energy deviations of a few Ha, times 2 / B."""
    e = np.clip(rng.laplace(scale=1.5, size=B), -7.5, 7.5)
    return torch.as_tensor(2.0 / B * (e - e.mean()), device=DEVICE).to(_dtype(case))


@functools.lru_cache(maxsize=64)
def _system(name):
    return fx.molecule(name)


def _inputs(case, seed):
    """Everything of a case that follows from its seed: parameters and walkers per molecule, and
    the walker weights or per-walker gradients that the operation takes."""
    rng = np.random.Generator(np.random.Philox(seed))
    out = {"theta": [], "r": [], "w": []}
    for name, B in _parts(case):
        system = _system(name)
        if case["op"] == "natural":
            # per-walker gradients: directions of quickly falling weight under walker noise
            P, rank = _count(case, system), 64
            gen = torch.Generator(device=DEVICE).manual_seed(int(rng.integers(1 << 40)))
            left = torch.randn(B, rank, device=DEVICE, generator=gen)
            left *= 0.9 ** torch.arange(rank, device=DEVICE)
            out["G"] = torch.randn(B, P, device=DEVICE, generator=gen).mul_(0.2)
            for a in range(0, P, 1 << 16):
                n = min(P, a + (1 << 16)) - a
                right = torch.randn(rank, n, device=DEVICE, generator=gen)
                for k in range(rank):  # rank by rank: no library product decides the inputs
                    out["G"][:, a:a + n].addcmul_(left[:, k:k + 1], right[k:k + 1])
        else:
            theta = _params(case, system, rng)
            out["theta"].append(theta)
            out["r"].append(_walkers(case, system, theta, B, rng))
        out["w"].append(_loss_weights(case, B, rng))
    return out


def prepare(case, seed):
    s = _inputs(case, seed)
    systems = [_system(m) for m, _ in _parts(case)]
    s["op"], s["seed"], s["steps"] = case["op"], seed, 0
    if case["op"] == "batch":
        s["h"] = AnsatzBatch(systems, [_cfg(case)] * len(systems), case["precision"], device=DEVICE)
    else:
        s["h"] = Ansatz(systems[0], _cfg(case), case["precision"], device=DEVICE)
    if case["op"] in ("sample", "train"):
        s["logabs"], _ = s["h"].ansatz_eval(s["theta"][0], s["r"][0])
    return s


def run(s):
    h, op = s["h"], s["op"]
    if op == "natural":
        return h.natural_gradient(s["G"], s["w"][0], -0.1, CG_ITERS)[0]
    if op == "batch":
        logabs, sign, e_loc = h.local_energy(s["theta"], s["r"])
        w, _ = h.vmc_loss_weights(e_loc)
        return logabs, sign, e_loc, h.grad_logpsi(s["theta"], s["r"], w)
    theta, r = s["theta"][0], s["r"][0]
    if op == "energy":
        return h.local_energy(theta, r)
    if op == "eval":
        return h.ansatz_eval(theta, r)
    if op == "grad":
        return h.grad_logpsi(theta, r, s["w"][0])
    if op == "walker_grads":
        return h.grad_logpsi(theta, r, mode=1)
    if op == "sample":
        accepted = h.mcmc_step(theta, r, s["logabs"], 10, 0.2, s["seed"], s["steps"])
        s["steps"] += 10
        return r, s["logabs"], accepted
    stats = binding.vmc_train_step(h, theta, r, s["logabs"], 1e-3, max_norm=0.05, seed=s["seed"],
                                   step_counter=s["steps"], cg_iters=CG_ITERS)
    s["steps"] += 1
    return theta, r, s["logabs"], stats["e_sum2"]


# ----------------------------------------------------------------------------
# Work
# ----------------------------------------------------------------------------
def _flops(case, system, jets):
    """Operations of one walker's forward: value only, or with all derivatives."""
    N, M, D, K, Q, L = system.n_elec, system.n_nuc, case["width"], case["dets"], N_RBF, case["layers"]
    C, e = (3 * N + 2, 3) if jets else (1, 1)
    pairs = N * (N - 1) // 2 + N * M
    filters = L * pairs * e * (2 * Q * D + 2 * D * D)
    nodes = (L if case["el_init"] else L - 1) * N * C * 2 * D * D
    messages = L * 2 * N * (N - 1) * C * D
    update = L * N * 2 * D * D * (2 * C + (5 if jets else 1))
    blocks = [system.n_elec] if case["full_det"] else [n for n in (system.n_up, system.n_down) if n]
    orbitals = sum(2 * C * D * K * n * n for n in blocks)
    dets = K * sum(2 / 3 * n ** 3 + (2 * n ** 3 * (3 * N + 2) if jets else 0) for n in blocks)
    return filters + nodes + messages + update + orbitals + dets


def work(case):
    size = 8 if case["precision"] == "fp64" else 4
    flops = nbytes = 0.0
    for name, B in _parts(case):
        system = _system(name)
        N3, P = 3 * system.n_elec, _count(case, system)
        value, energy = _flops(case, system, False), _flops(case, system, True)
        op = case["op"]
        if op == "natural":
            flops += float(B) * B * P + 4.0 * B * P  # a symmetric product, and two passes over the gradients
            nbytes += size * (B * P + B + P)
            continue
        nbytes += size * (P + B * N3)
        if op in ("energy", "batch", "train"):
            flops += B * energy
            nbytes += B * (2 * size + 1)
        if op == "eval":
            flops += B * value
            nbytes += B * (size + 1)
        if op in ("grad", "batch", "walker_grads", "train"):
            flops += 3.0 * B * value
            nbytes += size * P * (B if op == "walker_grads" else 1) + size * B
        if op in ("sample", "train"):
            flops += (10 if op == "sample" else 1) * B * value
            nbytes += size * B * (N3 + 2)
        if op == "train":
            flops += float(B) * B * P + 4.0 * B * P
    return {"bytes": nbytes, "flops": flops}


# ----------------------------------------------------------------------------
# The same results in plain torch
# ----------------------------------------------------------------------------
def exact(case, seed):
    op = case["op"]
    if op in ("sample", "train"):
        return None  # accepted moves, counters and a solver's path: no value of their own
    s = _inputs(case, seed)
    if op == "natural":
        return _natural(s["G"], s["w"][0].double())
    res = []
    for (name, B), theta, r, w in zip(_parts(case), s["theta"], s["r"], s["w"]):
        system = _system(name)
        theta, r = theta.double(), r.double()
        th = _blocks(case, system, theta)
        if op == "eval":
            size = _chunk(case, system, 2)
            with torch.no_grad():
                return torch.cat([_log_psi(case, system, th, r[b:b + size])[0] for b in range(0, B, size)]), None
        if op in ("energy", "batch"):
            size = _chunk(case, system, 2 * (3 * system.n_elec + 2))
            with torch.no_grad():
                both = [_local_energy(case, system, th, r[b:b + size]) for b in range(0, B, size)]
            logabs, e_loc = (torch.cat(x) for x in zip(*both))
            if op == "energy":
                return logabs, None, e_loc
            w = _clipped_weights(e_loc)
        if op == "walker_grads":
            return _walker_grads(case, system, theta, r)
        theta.requires_grad_(True)
        size = _chunk(case, system, 8)
        for b in range(0, B, size):
            value = _log_psi(case, system, _blocks(case, system, theta), r[b:b + size])[0]
            (value * w[b:b + size].double()).sum().backward()
        if op == "grad":
            return theta.grad
        res.append((logabs, None, e_loc, theta.grad))
    return tuple([x[k] if k != 1 else None for x in res] for k in range(4))


def _natural(G, w):
    """(Gc^T Gc / B + lam 1)^-1 Gc^T w through the B x B matrix; lam is 0.1 of its mean eigenvalue."""
    B, P = G.shape
    gram = torch.zeros(B, B, dtype=torch.float64, device=G.device)
    means = []
    for a in range(0, P, 1 << 16):
        g = G[:, a:a + (1 << 16)].double()
        means.append(g.mean(0))
        g = g - means[-1]
        gram += g @ g.T
    gram /= B
    lam = 0.1 * gram.diagonal().mean()
    x = torch.linalg.solve(gram + lam * torch.eye(B, dtype=torch.float64, device=G.device), w)
    return torch.cat([(G[:, a:a + (1 << 16)].double() - means[k]).T @ x for k, a in enumerate(range(0, P, 1 << 16))])


def _clipped_weights(e):
    """2 / B times the centred energies, clipped to five mean deviations around the median."""
    v = e.sort().values
    B = e.numel()
    mid = 0.5 * (v[(B - 1) // 2] + v[B // 2])
    half = 5 * (e - mid).abs().mean()
    c = e.clamp(mid - half, mid + half)
    return 2.0 / B * (c - c.mean())


def _walker_grads(case, system, theta, r):
    def one(th, x):
        return _log_psi(case, system, _blocks(case, system, th), x[None])[0][0]

    size = max(1, min(64, _chunk(case, system, 16)))
    grads = torch.func.vmap(torch.func.grad(one), in_dims=(None, 0))
    return torch.cat([grads(theta, r[b:b + size]).float() for b in range(0, len(r), size)])


def _chunk(case, system, channels):
    """Walkers at a time, for about 1 GB in the largest intermediate."""
    N = system.n_elec
    per = case["width"] * N * max(N, channels) + case["dets"] * channels * N * N
    return max(1, min(8192, int(1.2e8 / per)))


def _blocks(case, system, theta):
    out, o = {}, 0
    for name, shape, _ in _layout(case, system):
        n = math.prod(shape)
        out[name] = theta[o:o + n].reshape(shape)
        o += n
    return out


def _geometry(system, r):
    """Distances and unit vectors electron-electron (1 on the diagonal) and electron-nucleus."""
    N = r.shape[1]
    eye = torch.eye(N, dtype=r.dtype, device=r.device)
    v = r[:, :, None] - r[:, None]
    d = (v.square().sum(-1) + eye).sqrt()
    vn = r[:, :, None] - torch.as_tensor(system.R, dtype=r.dtype, device=r.device)
    dn = vn.square().sum(-1).sqrt()
    return d, v / d[..., None], dn, vn / dn[..., None], 1 - eye


def _features(d):
    width = CUTOFF / (N_RBF - 1)
    x = (d[..., None] - width * torch.arange(N_RBF, dtype=d.dtype, device=d.device)) / width
    e = torch.exp(-0.5 * x * x)
    return e, -x / width * e, (x * x - 1) / (width * width) * e


def _spins(system):
    up, N = system.n_up, system.n_elec
    return [slice(0, up)] + ([slice(up, N)] if N > up else [])


def _norm(system, a, t):
    """One over the number of edges of type t of an electron of spin a."""
    n = (system.n_up, system.n_down)
    return 1.0 / (max(1, n[a] - 1) if t == 0 else max(1, n[1 - a]) if t == 1 else system.n_nuc)


def _lin(x, W, b=None):
    y = x @ W.T
    return y if b is None else y + b


def _cusp_strength(system, like):
    s = torch.arange(system.n_elec, device=like.device) < system.n_up
    return torch.where(s[:, None] == s[None], 0.25, 0.5).to(like.dtype)


def _log_psi(case, system, th, r):
    """log|psi| and its sign of every walker."""
    d, _, dn, _, off = _geometry(system, r)
    spins, L = _spins(system), case["layers"]
    if case["el_init"]:
        x = (r[:, :, None] - torch.as_tensor(system.R, dtype=r.dtype, device=r.device)).flatten(2)
        f = _lin(torch.tanh(_lin(x, th["W_e1"], th["b_e1"])), th["W_e2"], th["b_e2"])
    else:
        f = torch.cat([th["E_spin"][a].expand(r.shape[0], (system.n_up, system.n_down)[a], -1)
                       for a in range(len(spins))], 1)
    ee = {(a, b): _features(d[:, spins[a], spins[b]])[0] for a in range(len(spins)) for b in range(a, len(spins))}
    en = _features(dn)[0]
    for l in range(L):
        z = _lin(f, th[f"W_h{l}"])

        def filt(e, t):
            return _lin(torch.tanh(_lin(e, th[f"W1{t}{l}"], th[f"b1{t}{l}"])), th[f"W2{t}{l}"], th[f"b2{t}{l}"])

        if case["edge_update"] and l:
            ee = {k: e + torch.tanh(_lin(e, th[f"U{int(k[0] != k[1])}{l}"], th[f"c{int(k[0] != k[1])}{l}"]))
                  for k, e in ee.items()}
            en = en + torch.tanh(_lin(en, th[f"U2{l}"], th[f"c2{l}"]))
        m = [[z.new_zeros(z[:, sp].shape) for sp in spins] for _ in range(2)]
        for (a, b), e in ee.items():
            w = filt(e, int(a != b))
            if a == b:
                w = w * off[spins[a], spins[a], None]
            else:
                m[1][b] = (w * z[:, spins[a], None]).sum(1) * _norm(system, b, 1)
            m[int(a != b)][a] = (w * z[:, None, spins[b]]).sum(2) * _norm(system, a, int(a != b))
        nuc = (filt(en, 2) * th[f"Y{l}"]).sum(2) * _norm(system, 0, 2)
        f = f + torch.tanh(_lin(torch.cat([torch.cat(x, 1) for x in m] + [nuc], -1), th[f"W_g{l}"], th[f"b_g{l}"]))
    A = []
    for a, sp in enumerate(spins):
        env = (th[f"omega{a}"] * torch.exp(-th[f"zeta{a}"] * dn[:, sp, None])).sum(-1)
        A.append((_lin(f[:, sp], th[f"W_o{a}"], th[f"b_o{a}"]) * env).unflatten(-1, (case["dets"], -1)).transpose(1, 2))
    sign, logdet = 1, 0
    for M in [torch.cat(A, 2)] if case["full_det"] else A:
        s, x = torch.linalg.slogdet(M)
        sign, logdet = sign * s, logdet + x
    sign, logdet = sign * torch.sign(th["c"]), logdet + th["c"].abs().log()
    top = logdet.detach().max(-1, keepdim=True).values
    psi = (sign * torch.exp(logdet - top)).sum(-1)
    out = top[:, 0] + psi.abs().log() + _lin(torch.tanh(_lin(f.sum(1), th["W_J1"], th["b_J1"])), th["w_J2"])[:, 0]
    cusp = -_cusp_strength(system, r) / (1 + d) * off
    return out + 0.5 * cusp.sum((1, 2)), torch.sign(psi)


# A function of the walker's coordinates is carried as (value, derivatives in all 3N coordinates,
# Laplacian); a function of one distance as (value, first, second derivative).
def _tanh_1d(a):
    t = torch.tanh(a[0])
    s = 1 - t * t
    return t, s * a[1], s * a[2] - 2 * t * s * a[1].square()


def _tanh_jet(a):
    t = torch.tanh(a[0])
    s = 1 - t * t
    return t, s.unsqueeze(-2) * a[1], s * a[2] - 2 * t * s * a[1].square().sum(-2)


def _lin_jet(x, W, b=None):
    return (_lin(x[0], W, b),) + tuple(_lin(y, W) for y in x[1:])


def _local_energy(case, system, th, r):
    """log|psi| and the local energy of every walker."""
    B, N, _ = r.shape
    d, u, dn, un, off = _geometry(system, r)
    spins, L, K, D = _spins(system), case["layers"], case["dets"], case["width"]
    own = torch.eye(N, dtype=r.dtype, device=r.device)  # electron i's coordinates among all

    def scatter(x):
        """[.., N, 3, n] derivatives of electron i's rows in its own coordinates -> [.., N, 3N, n]"""
        return (own[:, :, None, None] * x[:, :, None]).flatten(2, 3)

    def own_part(x):
        """Electron i's own three of the 3N derivatives of its rows."""
        return torch.einsum("bikcn,ik->bicn", x.unflatten(2, (N, 3)), own)

    if case["el_init"]:
        x = (r[:, :, None] - torch.as_tensor(system.R, dtype=r.dtype, device=r.device)).flatten(2)
        W = th["W_e1"].unflatten(1, (-1, 3)).sum(1).T  # every nucleus' vector moves with r_i
        a = _lin(x, th["W_e1"], th["b_e1"])
        t = torch.tanh(a)
        s = 1 - t * t
        f = (t, scatter(s[:, :, None] * W), -2 * t * s * W.square().sum(0))
        f = _lin_jet(f, th["W_e2"], th["b_e2"])
    else:
        v = torch.cat([th["E_spin"][a].expand(B, (system.n_up, system.n_down)[a], -1) for a in range(len(spins))], 1)
        f = (v, torch.zeros(B, N, 3 * N, D, dtype=r.dtype, device=r.device), torch.zeros_like(v))
    ee = {(a, b): _features(d[:, spins[a], spins[b]]) for a in range(len(spins)) for b in range(a, len(spins))}
    en = _features(dn)
    for l in range(L):
        z = _lin_jet(f, th[f"W_h{l}"])

        def filt(e, t):
            return _lin_jet(_tanh_1d(_lin_jet(e, th[f"W1{t}{l}"], th[f"b1{t}{l}"])), th[f"W2{t}{l}"], th[f"b2{t}{l}"])

        def iterate(e, t):
            h = _tanh_1d(_lin_jet(e, th[f"U{t}{l}"], th[f"c{t}{l}"]))
            return tuple(x + y for x, y in zip(e, h))

        if case["edge_update"] and l:
            ee = {k: iterate(e, int(k[0] != k[1])) for k, e in ee.items()}
            en = iterate(en, 2)
        m = [[torch.zeros_like(x) for x in f] for _ in range(2)]

        def message(i, j, w, t, nu):
            """Messages of electrons i from electrons j."""
            w0, w1, w2 = w
            U = u[:, i, j, :, None]
            push = w1[..., None, :] * U * z[0][:, None, j, None]  # [b, i, j, 3, n]
            mv = torch.einsum("bijn,bjn->bin", w0, z[0][:, j])
            mj = torch.einsum("bijn,bjkn->bikn", w0, z[1][:, j])
            mj = mj + (own[i, :, None, None] * push.sum(2)[:, :, None]).flatten(2, 3)
            part = torch.zeros_like(mj).unflatten(2, (N, 3))
            part[:, :, j] = push
            mj = mj - part.flatten(2, 3)
            zj = z[1][:, j].unflatten(2, (N, 3))
            dz = zj[:, :, i].transpose(1, 2) - torch.einsum("bjkcn,jk->bjcn", zj, own[j])[:, None]
            ml = (torch.einsum("bijn,bjn->bin", w0, z[2][:, j]) + 2 * (w1[..., None, :] * U * dz).sum((2, 3))
                  + 2 * ((w2 + 2 * w1 / d[:, i, j, None]) * z[0][:, None, j]).sum(2))
            for x, y in zip(m[t], (mv, mj, ml)):
                x[:, i] += nu * y

        for (a, b), e in ee.items():
            w = filt(e, int(a != b))
            if a == b:
                w = tuple(x * off[spins[a], spins[a], None] for x in w)
            else:
                message(spins[b], spins[a], tuple(x.transpose(1, 2) for x in w), 1, _norm(system, b, 1))
            message(spins[a], spins[b], w, int(a != b), _norm(system, a, int(a != b)))
        w0, w1, w2 = (x * th[f"Y{l}"] * _norm(system, 0, 2) for x in filt(en, 2))
        nuc = (w0.sum(2), scatter((w1[..., None, :] * un[..., None]).sum(2)), (w2 + 2 * w1 / dn[..., None]).sum(2))
        x = _tanh_jet(_lin_jet([torch.cat(y, -1) for y in zip(m[0], m[1], nuc)], th[f"W_g{l}"], th[f"b_g{l}"]))
        f = tuple(x0 + y for x0, y in zip(f, x))

    A = []  # per spin the rows of the matrices [b, K, rows, cols], derivatives [b, K, 3N, rows, cols]
    for a, sp in enumerate(spins):
        zeta, dd, uu = th[f"zeta{a}"], dn[:, sp, None], un[:, sp]
        g = th[f"omega{a}"] * torch.exp(-zeta * dd)
        env, env1 = g.sum(-1), -torch.einsum("biom,bimx->bixo", g * zeta, uu)
        env2 = (g * (zeta * zeta - 2 * zeta / dd)).sum(-1)
        p = _lin_jet([x[:, sp] for x in f], th[f"W_o{a}"], th[f"b_o{a}"])
        mine = torch.einsum("bikxo,ik->bixo", p[1].unflatten(2, (N, 3)), own[sp])
        jac = p[1] * env[:, :, None] + (own[sp, :, None, None] * (p[0][:, :, None] * env1)[:, :, None]).flatten(2, 3)
        lap = p[2] * env + 2 * (mine * env1).sum(2) + p[0] * env2
        A.append(((p[0] * env).unflatten(-1, (K, -1)).transpose(1, 2),
                  jac.unflatten(-1, (K, -1)).permute(0, 3, 2, 1, 4), lap.unflatten(-1, (K, -1)).transpose(1, 2)))
    if case["full_det"]:
        A = [tuple(torch.cat(x, -2) for x in zip(*A))]
    sign, logdet, grad, lapl = 1, 0, 0, 0
    for v, jac, lap in A:
        s, x = torch.linalg.slogdet(v)
        inv = torch.linalg.inv(v)
        T = inv[:, :, None] @ jac
        sign, logdet = sign * s, logdet + x
        grad = grad + T.diagonal(dim1=-2, dim2=-1).sum(-1)
        lapl = lapl + (inv * lap.transpose(-1, -2)).sum((-1, -2)) - (T * T.transpose(-1, -2)).sum((-1, -2, -3))
    logdet = logdet + th["c"].abs().log()
    top = logdet.max(-1, keepdim=True).values
    q = sign * torch.sign(th["c"]) * torch.exp(logdet - top)
    psi = q.sum(-1)
    q = q / psi[:, None]
    logabs = top[:, 0] + psi.abs().log()
    g = (q[..., None] * grad).sum(1)
    lapl = (q * (lapl + grad.square().sum(-1))).sum(1) - g.square().sum(-1)
    J = _tanh_jet(_lin_jet([x.sum(1) for x in f], th["W_J1"], th["b_J1"]))
    J = [_lin(x, th["w_J2"])[..., 0] for x in J]
    cs = _cusp_strength(system, r) * off
    c1, c2 = cs / (1 + d) ** 2, -2 * cs / (1 + d) ** 3
    logabs = logabs + J[0] - 0.5 * (cs / (1 + d)).sum((1, 2))
    g = g + J[1] + (c1[..., None] * u).sum(2).flatten(1)
    lapl = lapl + J[2] + (c2 + 2 * c1 / d).sum((1, 2))
    Z = torch.as_tensor(system.Z, dtype=r.dtype, device=r.device)
    R = torch.as_tensor(system.R, dtype=r.dtype, device=r.device)
    rep = sum(float(Z[i] * Z[j] / (R[i] - R[j]).norm()) for i in range(len(Z)) for j in range(i))
    V = 0.5 * (off / d).sum((1, 2)) - (Z / dn).sum((1, 2)) + rep
    return logabs, -0.5 * (lapl + g.square().sum(-1)) + V
