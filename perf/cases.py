"""What a user of the decoder runs, as cases that can be timed and compared.

Sizes are those of the repository's own workloads (bench.py, ragged_bench.py,
serve_bench.py, variants_bench.py, cnn_bench.py, early_stop.py, the parity
configuration of the tests), with sweeps shortened where the full length would
only repeat the same work; draw() spreads sizes, chain counts, code sizes
(odd, even and ragged) and error rates over the ranges between them.

Error rates lie in [0.08, 0.18] (the range around the paper's threshold that
the workloads use); independent flips in [0.03, 0.10], the torus below 0.15.

Inputs are synthetic i.i.d. errors as in every workload here: sampled from the
seed with torch on the GPU and turned into syndromes by the parities of the
code, without the library's own generator.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1302_2669_gb300 as P

DEV = "cuda"
SERVE_LS = (9, 13, 17, 25)
RAGGED_LS = (5, 9, 13, 17, 25)
CHANNELS = (2, 64, 64, 64, 64, 2)
PAULI_ENERGY = (2, 3, 1)


def listed():
    return [
        # One syndrome by itself in host memory, a request outside any batch:
        # latency of the chains, launches and copies.
        {"name": "single_L13", "kind": "decode", "L": 13, "n": 1, "R": 4, "sweeps": 169, "burn": 42, "stages": 4,
         "a0": 0.3, "p": 0.12, "host": True},
        # The parity configuration: 200 syndromes of the smallest common code.
        {"name": "small_L5", "kind": "decode", "L": 5, "n": 200, "R": 4, "sweeps": 2000, "burn": 0, "stages": 0,
         "a0": 1.0, "p": 0.15, "host": False},
        # The benchmark's decode (64 chains per syndrome, annealed burn-in) at
        # a twentieth of its sweeps: the throughput of large batches.
        {"name": "batch_L13", "kind": "decode", "L": 13, "n": 16384, "R": 16, "sweeps": 1000, "burn": 200,
         "stages": 16, "a0": 0.1, "p": 0.13, "host": False},
        # Serving: a burst of requests of mixed sizes through the server.
        {"name": "serve_512", "kind": "serve", "n": 512, "R": 4, "p": 0.12},
        # A captured ragged batch of five code sizes, sweeps L^2.
        {"name": "ragged_32768", "kind": "plan", "n": 32768, "R": 4, "p": 0.14},
        # Decoding with the network's early stop.
        {"name": "early_L17", "kind": "early", "L": 17, "n": 8192, "R": 4, "sweeps": 1000, "burn": 200, "stages": 16,
         "a0": 0.1, "chunk": 100, "p": 0.10},
        # Thermodynamic integration over 21 temperatures.
        {"name": "ti_L9", "kind": "ti", "L": 9, "n": 4096, "R": 4, "sweeps": 400, "burn": 100, "stages": 4, "a0": 0.3,
         "p": 0.10, "n_beta": 21},
        # A general Pauli channel: random scan, the paper's Sec. IV as written.
        {"name": "general_L9", "kind": "general", "L": 9, "n": 4096, "R": 4, "sweeps": 200, "burn": 50, "stages": 4,
         "a0": 0.3, "p": 0.10},
        # Independent bit and phase flips.
        {"name": "flips_L9", "kind": "flips", "L": 9, "n": 16384, "R": 4, "sweeps": 400, "burn": 100, "stages": 4,
         "a0": 0.3, "p": 0.05},
        # The toric code's 16 classes, sampling the errors included (a Monte
        # Carlo estimate of the logical error rate draws and decodes).
        {"name": "toric_L8", "kind": "toric", "L": 8, "n": 16384, "R": 4, "sweeps": 400, "burn": 100, "stages": 4,
         "a0": 0.3, "p": 0.08},
        # The early-stop network: inference on a large batch, and loss and
        # gradient of a training batch.
        {"name": "forward_L17", "kind": "forward", "L": 17, "n": 8192, "p": 0.12},
        {"name": "gradient_L17", "kind": "gradient", "L": 17, "n": 1024, "p": 0.12},
    ]


# Chain updates (proposals, accepted or not) of a drawn case at most: those of
# the largest listed case of the same scan; random scan runs one proposal per
# thread where the colour sweeps run 32.
MAX_UPDATES = 16384 * 64 * 1000 * 312
MAX_UPDATES_SCAN = 4096 * 16 * 200 * 144


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["decode", "decode", "decode", "serve", "plan", "early", "ti", "general", "flips", "toric",
                       "forward", "gradient"])
    p = round(rng.uniform(0.08, 0.18), 4)
    if kind == "serve":
        return {"kind": kind, "n": _logint(rng, 40, 1500), "R": rng.choice([2, 4]), "p": round(rng.uniform(0.08, 0.14), 4)}
    if kind == "plan":
        return {"kind": kind, "n": _logint(rng, 500, 32768), "R": rng.choice([2, 4, 5]), "p": p}
    if kind in ("forward", "gradient"):
        L = rng.randint(5, 25)
        hi = min(8192 if kind == "forward" else 1024, (8192 if kind == "forward" else 1024) * 17 * 17 // (L * L))
        return {"kind": kind, "L": L, "n": _logint(rng, 3, hi), "p": p}
    stages = rng.choice([0, 4, 16])
    burn = rng.randint(stages, 10 * stages) if stages else rng.choice([0, rng.randint(1, 100)])
    sweeps = burn + _logint(rng, 50, 1000)
    c = {"kind": kind, "R": rng.choice([1, 2, 3, 4, 4, 8, 16]), "sweeps": sweeps, "burn": burn, "stages": stages,
         "a0": rng.choice([0.1, 0.3]) if stages else 1.0, "p": p}
    factor, top = 1, MAX_UPDATES
    if kind == "decode":
        c["L"] = rng.randint(3, 25)
    elif kind == "early":
        c.update(L=rng.randint(7, 19), R=4, chunk=rng.randint(30, 200), p=round(rng.uniform(0.08, 0.13), 4))
    elif kind == "ti":
        c.update(L=rng.randint(3, 13), R=rng.choice([2, 4]), n_beta=rng.choice([11, 21]))
        factor = c["n_beta"] - 1
    elif kind == "general":
        c.update(L=rng.randint(3, 13), R=rng.choice([2, 4]))
        top = MAX_UPDATES_SCAN
    elif kind == "flips":
        c.update(L=rng.randint(3, 17), R=rng.choice([2, 4, 8]), p=round(rng.uniform(0.03, 0.10), 4))
    elif kind == "toric":
        c.update(L=2 * rng.randint(2, 8), R=rng.choice([1, 4]), p=round(rng.uniform(0.05, 0.12), 4))
    per = max(1, _chains(c) * c["sweeps"] * factor * _n_stab(c))
    # "n" below the pass limits of both the work and the largest batch in use
    c["n"] = _logint(rng, 1, max(2, min(16384, top // per)))
    if kind == "decode":
        c["host"] = c["n"] < 64 and rng.random() < 0.5
    return c


def _n_stab(c):
    L = c["L"]
    return 2 * L * L if c["kind"] == "toric" else 2 * L * (L - 1)


def _chains(c):
    return (16 if c["kind"] == "toric" else 4) * c["R"]


# ---------------------------------------------------------------------------
# Inputs: i.i.d. errors and their syndromes, from the seed
# ---------------------------------------------------------------------------
def _generator(seed, salt=0):
    g = torch.Generator(device=DEV)
    g.manual_seed((int(seed) * 1000003 + salt) & 0x7FFFFFFFFFFF)
    return g


def _sample_planar(seed, n, L, probs, salt=0):
    """n syndromes [n][2L(L-1)] uint8 of errors X, Y, Z with probabilities probs."""
    out = torch.empty((n, 2 * L * (L - 1)), dtype=torch.uint8, device=DEV)
    g = _generator(seed, salt + 100 * L)
    m, step = 2 * L - 1, 4096
    r = torch.arange(m, device=DEV)
    qubit = ((r[:, None] + r[None, :]) % 2 == 0)
    for a in range(0, n, step):
        b = min(n, a + step)
        x, z = _errors(g, (b - a, m, m), probs)
        x, z = x & qubit, z & qubit
        px, pz = _neighbour_parity(x), _neighbour_parity(z)
        out[a:b, :L * (L - 1)] = pz[:, 1::2, 0::2].reshape(b - a, -1)
        out[a:b, L * (L - 1):] = px[:, 0::2, 1::2].reshape(b - a, -1)
    return out


def _errors(g, shape, probs):
    if len(probs) == 1:        # independent flips
        return (torch.rand(shape, generator=g, device=DEV) < probs[0],
                torch.rand(shape, generator=g, device=DEV) < probs[0])
    u = torch.rand(shape, generator=g, device=DEV)
    px, py, pz = probs
    return u < px + py, (u >= px) & (u < px + py + pz)


def _neighbour_parity(f):
    """Parity of the four grid neighbours (cells outside the grid count 0)."""
    s = torch.zeros_like(f)
    s[:, 1:] ^= f[:, :-1]
    s[:, :-1] ^= f[:, 1:]
    s[:, :, 1:] ^= f[:, :, :-1]
    s[:, :, :-1] ^= f[:, :, 1:]
    return s


def _general_probs(p, e):
    """p_P = (1 - p) r^e_P with (1 - p) sum_P r^e_P = p."""
    lo, hi = 0.0, 1.0
    for _ in range(100):
        r = 0.5 * (lo + hi)
        if (1.0 - p) * sum(r ** k for k in e) < p:
            lo = r
        else:
            hi = r
    return tuple((1.0 - p) * (0.5 * (lo + hi)) ** k for k in e)


def _mixed(seed, n, sizes, p):
    """n rows of code sizes drawn from `sizes`, concatenated, and the sizes."""
    rng = np.random.default_rng(int(seed) + 1)
    Ls = rng.choice(sizes, size=n).astype(np.int32)
    off = np.concatenate([[0], np.cumsum(2 * Ls.astype(np.int64) * (Ls - 1))])
    cat = torch.empty(int(off[-1]), dtype=torch.uint8, device=DEV)
    for L in sizes:
        idx = np.nonzero(Ls == L)[0]
        if len(idx) == 0:
            continue
        rows = _sample_planar(seed, len(idx), int(L), (p / 3,) * 3)
        at = torch.from_numpy(off[idx]).to(DEV)[:, None] + torch.arange(rows.shape[1], device=DEV)[None, :]
        cat[at.reshape(-1)] = rows.reshape(-1)
    return Ls, off, cat


def _params(seed):
    """Parameters of a network as training starts from them: He-scaled
    weights, small biases, the last layer's bias at -4 (flips unlikely)."""
    rng = np.random.default_rng(int(seed) + 7)
    parts = []
    for i in range(5):
        ci, co = CHANNELS[i], CHANNELS[i + 1]
        scale = math.sqrt(2.0 / (9 * ci)) * (0.15 if i == 4 else 1.0)
        parts.append(rng.normal(0, scale, size=co * 9 * ci))
        parts.append(np.full(co, -4.0) if i == 4 else rng.normal(0, 0.05, size=co))
    return np.concatenate(parts).astype(np.float32)


def _targets(seed, n):
    rng = np.random.default_rng(int(seed) + 9)
    return rng.dirichlet(np.ones(4) * 0.5, size=n).astype(np.float32)


_CTX = {}


def _ctx():
    """The program's one library context (grow-only scratch), as every
    benchmark here keeps it."""
    if "c" not in _CTX:
        _CTX["c"] = P.Context(0)
    return _CTX["c"]


def _opts(c, **kw):
    return P.Opts(chains_per_class=c["R"], n_sweeps=c["sweeps"], burn_in=c["burn"], anneal_stages=c["stages"],
                  anneal_beta0=c["a0"], **kw)


def prepare(case, seed):
    c = dict(case)
    s = {"case": c, "seed": int(seed) & 0x7FFFFFFF, "ctx": _ctx()}
    kind = c["kind"]
    dep = (c["p"] / 3,) * 3
    if kind == "decode":
        syn = _sample_planar(seed, c["n"], c["L"], dep)
        s["syn"] = syn.cpu().numpy() if c["host"] else syn
        s["opts"] = _opts(c)
    elif kind == "ti":
        s["syn"] = _sample_planar(seed, c["n"], c["L"], dep)
        s["opts"] = _opts(c)
    elif kind == "flips":
        s["syn"] = _sample_planar(seed, c["n"], c["L"], (c["p"],))
        s["opts"] = _opts(c, noise=1, beta_scale=0.85)
    elif kind == "general":
        s["syn"] = _sample_planar(seed, c["n"], c["L"], _general_probs(c["p"], PAULI_ENERGY))
        s["opts"] = _opts(c, noise=2, scan=1, pauli_energy=PAULI_ENERGY)
    elif kind == "toric":
        s["like"] = torch.zeros(1, device=DEV)
        s["opts"] = _opts(c, n_classes=16)
    elif kind == "serve":
        Ls, off, cat = _mixed(seed, c["n"], SERVE_LS, c["p"])
        cat = cat.cpu().numpy()
        s["rows"] = [(i, int(L), int(L) * int(L), cat[off[i]:off[i + 1]]) for i, L in enumerate(Ls)]
        s["server"] = P.Server(0, p=c["p"], opts=P.Opts(chains_per_class=c["R"], n_sweeps=100, burn_in=25,
                                                         anneal_stages=4, anneal_beta0=0.3), seed=s["seed"])
    elif kind == "plan":
        Ls, _, cat = _mixed(seed, c["n"], RAGGED_LS, c["p"])
        dLs = torch.from_numpy(Ls).to(DEV)
        sw = torch.from_numpy((Ls.astype(np.int64) ** 2).astype(np.uint32)).to(DEV)
        s["out"] = (torch.empty(c["n"], dtype=torch.int32, device=DEV),
                    torch.empty((c["n"], 4), dtype=torch.uint64, device=DEV),
                    torch.empty((c["n"], 4), dtype=torch.float64, device=DEV))
        s["plan"] = P.RaggedPlan(s["ctx"], dLs, c["p"], cat, *s["out"],
                                 opts=P.Opts(chains_per_class=c["R"], n_sweeps=max(RAGGED_LS) ** 2), n_sweeps=sw,
                                 seed=s["seed"])
    else:                       # early, forward, gradient: a network
        s["syn"] = _sample_planar(seed, c["n"], c["L"], dep)
        s["net"] = P.Network(s["ctx"], c["L"], max_batch=c["n"])
        s["net"].set_params(_params(seed if kind != "early" else 5))
        if kind == "gradient":
            s["q"] = torch.from_numpy(_targets(seed, c["n"])).to(DEV)
        if kind == "early":
            s["opts"] = _opts(c)
    return s


def run(s):
    c, ctx, kind = s["case"], s["ctx"], s["case"]["kind"]
    if kind in ("decode", "flips", "general"):
        return ctx.decode(s["syn"], c["L"], c["p"], s["opts"], seed=s["seed"])
    if kind == "toric":
        syn, true_class = ctx.gen_syndromes_toric(s["seed"], 0, c["n"], c["L"], c["p"], like=s["like"])
        return (true_class,) + ctx.decode(syn, c["L"], c["p"], s["opts"], seed=s["seed"])
    if kind == "ti":
        return ctx.decode_ti(s["syn"], c["L"], c["p"], s["opts"], n_beta=c["n_beta"], seed=s["seed"])
    if kind == "serve":
        return _serve(s)
    if kind == "plan":
        s["plan"].launch()
        return s["out"]
    if kind == "early":
        # tau = 0 stops a syndrome once the chains agree with the network's
        # best class (an untrained network's best class is clear of ties)
        return ctx.decode_early(s["net"], s["syn"], c["L"], c["p"], s["opts"], chunk_sweeps=c["chunk"], tau=0.0,
                                seed=s["seed"])
    if kind == "forward":
        return s["net"].forward(s["syn"])
    return s["net"].gradient(s["syn"], s["q"])


def _serve(s):
    """Submits every request, takes the results as they come, returns them in
    request order."""
    server, n = s["server"], len(s["rows"])
    for i, L, sweeps, row in s["rows"]:
        server.submit(i, L, sweeps, row)
    cls, sums, got = np.empty(n, np.int32), np.empty((n, 4), np.uint64), 0
    while got < n:
        ids, k, v, _ = server.poll(wait_us=1000)
        cls[ids], sums[ids] = k, v
        got += len(ids)
    return cls, sums


# ---------------------------------------------------------------------------
# Work
# ---------------------------------------------------------------------------
def work(case):
    """Bytes: syndromes in, results out.  flops: for the chains the integer
    operations of bench.py's count (4.25 per chain update in the bit-sliced
    form; a random-scan step is counted the same), for the network the
    multiply-adds of conv1..conv4 on the L x L maps (and, for the gradient,
    of their weight gradients and of the input gradients of conv2..conv4)."""
    c, kind = case, case["kind"]
    if kind in ("forward", "gradient"):
        L, n = c["L"], c["n"]
        fwd = [2 * 9 * a * b for a, b in zip(CHANNELS, CHANNELS[1:])][:4]
        per = sum(fwd) if kind == "forward" else 2 * sum(fwd) + sum(fwd[1:])
        io = n * 2 * L * (L - 1) + n * 16 + 4 * 113154 * (1 if kind == "forward" else 2)
        return {"bytes": io, "flops": per * n * L * L}
    if kind in ("serve", "plan"):
        sizes = SERVE_LS if kind == "serve" else RAGGED_LS
        upd = sum(4 * c["R"] * L * L * 2 * L * (L - 1) for L in sizes) * c["n"] / len(sizes)
        io = c["n"] * (sum(2 * L * (L - 1) for L in sizes) / len(sizes) + 4 + 32 + (32 if kind == "plan" else 0))
        return {"bytes": io, "flops": 4.25 * upd}
    upd = c["n"] * _chains(c) * c["sweeps"] * _n_stab(c) * (c["n_beta"] - 1 if kind == "ti" else 1)
    K = 16 if kind == "toric" else 4
    out = 4 + 8 * K * (c["n_beta"] + 1) if kind == "ti" else 8 + 32 if kind == "early" else 4 + 16 * K
    return {"bytes": c["n"] * (_n_stab(c) + out), "flops": 4.25 * upd}


# ---------------------------------------------------------------------------
# 64-bit values
# ---------------------------------------------------------------------------
def exact(case, seed):
    """The network in float64 (weights rounded to bfloat16 as the network is
    defined, activations not rounded).  The chains' results are whole numbers,
    compared as such; the float64 values beside them are simple functions of
    those sums, and a 64-bit value of the chains themselves would take a
    bit-level simulation of minutes: None."""
    if case["kind"] not in ("forward", "gradient"):
        return None
    L, n, grad = case["L"], case["n"], case["kind"] == "gradient"
    syn = _sample_planar(seed, n, L, (case["p"] / 3,) * 3)
    q = torch.from_numpy(_targets(seed, n)).to(DEV).double() if grad else None
    theta = torch.from_numpy(_params(seed)).to(DEV)
    w, b, off = [], [], 0
    for i in range(5):
        ci, co = CHANNELS[i], CHANNELS[i + 1]
        k = co * 9 * ci
        w.append(theta[off:off + k].bfloat16().double().reshape(co, 9, ci).requires_grad_(grad))
        b.append(theta[off + k:off + k + co].double().requires_grad_(grad))
        off += k + co
    step = max(1, 160000 // (L * L))
    out, loss = [], 0.0
    for a in range(0, n, step):
        with torch.set_grad_enabled(grad):
            lp = _network64(syn[a:a + step], L, w, b)
            if grad:
                part = -(q[a:a + step] * lp).sum() / n
                part.backward()
                loss += float(part.detach())
            else:
                out.append(lp)
    if not grad:
        return torch.cat(out)
    flat = torch.cat([t.grad.reshape(-1) for pair in zip(w, b) for t in pair])
    return loss, flat.cpu().numpy()


def _network64(syn, L, w, b):
    n = syn.shape[0]
    x = torch.zeros((n, L, L, 2), dtype=torch.float64, device=DEV)
    x[:, :L - 1, :, 0] = syn[:, :L * (L - 1)].reshape(n, L - 1, L).double()
    x[:, :, :L - 1, 1] = syn[:, L * (L - 1):].reshape(n, L, L - 1).double()
    for i in range(5):
        pad = torch.nn.functional.pad(x, (0, 0, 1, 1, 1, 1))
        cols = torch.cat([pad[:, t // 3:t // 3 + L, t % 3:t % 3 + L] for t in range(9)], dim=-1)
        x = cols @ w[i].reshape(w[i].shape[0], -1).T + b[i]
        if i < 4:
            x = x.relu()
    m = (L - 1) // 2
    s_maps = syn.long()
    # class code of the pure error: sigma_z defects joined left cross column
    # 0, sigma_x defects joined up cross row 0
    j = torch.arange(L - 1, device=DEV)
    near = (2 * (j + 1) <= L).long()
    b0 = (s_maps[:, :L * (L - 1)].reshape(n, L - 1, L).sum(2) * near).sum(1) % 2
    a0 = (s_maps[:, L * (L - 1):].reshape(n, L, L - 1).sum(1) * near).sum(1) % 2
    lim = 1.0 - 1e-6
    mx = torch.prod(-torch.tanh(0.5 * x[:, :, m, 0]), dim=1).clamp(-lim, lim)
    mz = torch.prod(-torch.tanh(0.5 * x[:, m, :, 1]), dim=1).clamp(-lim, lim)
    lx = torch.stack([torch.log1p(mx), torch.log1p(-mx)], 1) - math.log(2.0)
    lz = torch.stack([torch.log1p(mz), torch.log1p(-mz)], 1) - math.log(2.0)
    return torch.stack([lx.gather(1, ((k & 1) ^ a0)[:, None])[:, 0] + lz.gather(1, ((k >> 1) ^ b0)[:, None])[:, 0]
                        for k in range(4)], 1)
