"""The calls that stand for the library's use, for timing them on a GPU.

Each case is a dict of plain values; ``kind`` names the call sequence:

* ``batch``       one fire_simulate_batch on one landscape, device tensors or
                  host arrays, with or without burn-step maps, either update
                  rule
* ``generation``  one generation of the genetic algorithm: simulate, fitness,
                  replicate mean, breed (five genes, fixed ignition)
* ``generation7`` the same with the ignition as two more genes (cells snapped
                  to the target scar first)
* ``search``      one ignition_search over a lattice inside the target scar
* ``multi``       one uneven batch over several landscapes
* ``burnout``     one batch with per-fuel burn-out times
* ``train``       forward and backward of the surrogate network
* ``screen``      surrogate inputs, forward pass and predicted fitness of a
                  pool of candidates

All of them run with the launch shape the library picks by itself (no
fire_set_launch, no fire_autotune), as the calibration module's calls do.
"""
import math

import numpy as np
import torch

from paper_1701_03549_gb300 import fire, surrogate, synth

# Lane operations of one trial (a quarter Philox block, Eq. 1 in one
# direction, the logistic and the comparison).
_OPS_PER_TRIAL = 40.0
# Trials per simulation and grid cell by parameter distribution: the Table 1
# priors burn most of a map, the reference parameters a small part of it.
_TRIALS_PER_CELL = {"gauss": 1.2, "uniform": 1.15, "truth": 0.1, "near": 0.3}


# ---------------------------------------------------------------------------
# The cases.

def listed():
    return [
        # The smallest call: a handful of fires on a small ragged landscape
        # with their burn-step maps, as a program previews a parameter set.
        dict(name="preview_70x90", kind="batch", H=70, W=90, n=8,
             prior="truth", wind="field", steps=True, cell=False, host=False),
        # 64 replicates of one fire on 128 x 128 with burn-step maps.
        dict(name="replicates_128", kind="batch", H=128, W=128, n=64,
             prior="truth", wind="constant", steps=True, cell=False,
             host=False),
        # A batch through host arrays on a ragged landscape: the README's
        # call (numpy in, results and fitness out).
        dict(name="host_333x517", kind="batch", H=333, W=517, n=512,
             prior="gauss", wind="field", steps=False, cell=False, host=True),
        # Brute-force Monte Carlo on the paper's 801 x 801 map with the
        # paper's own update (one uniform per cell and step).
        dict(name="monte_carlo_801_cell", kind="batch", H=801, W=801, n=1024,
             prior="uniform", wind="constant", steps=False, cell=True,
             host=False),
        # One generation of the genetic algorithm on 512 x 512.
        dict(name="ga_512", kind="generation", H=512, W=512, pop=256, reps=16,
             prior="gauss", wind="constant"),
        # One generation of the variable-ignition algorithm on 1024 x 1024,
        # wind varying in space, midway through a run.
        dict(name="ga_ignition_1024", kind="generation7", H=1024, W=1024,
             pop=256, reps=16, prior="near", wind="field"),
        # The ignition-point search on 1024 x 1024: many short fires.
        dict(name="search_1024", kind="search", H=1024, W=1024, lattice=32,
             reps=16, wind="field"),
        # The nine-fire uneven batch, 200 x 300 ... 2000 x 1500.
        dict(name="uneven_9", kind="multi", maps=9, h0=200, w0=300, dh=225,
             dw=150, n=18000, prior="uniform", wind="constant"),
        # Per-fuel burn-out times on the 512 x 512 generation's landscape.
        dict(name="burnout_512", kind="burnout", H=512, W=512, n=1024,
             prior="gauss", wind="constant"),
        # A training step's gradient of the surrogate at its full size, and
        # at the small size that launches dominate.
        dict(name="train_256", kind="train", S=256, n=8),
        dict(name="train_32", kind="train", S=32, n=32),
        # Screening a pool of candidates before they are simulated.
        dict(name="screen_256", kind="screen", S=256, n=16, batch=8, H=1024,
             W=1024),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["batch", "batch", "generation", "generation7",
                       "search", "multi", "burnout", "train", "screen"])
    if kind in ("train", "screen"):
        S = rng.choice([16, 32, 64, 128, 256])
        most = 8 * 256 * 256 // (S * S)
        n = _log_int(rng, 1, min(most, 256))
        if kind == "train":
            return dict(kind=kind, S=S, n=n)
        return dict(kind=kind, S=S, n=n, batch=max(1, n // rng.choice([1, 2])),
                    H=S * rng.choice([1, 2, 4]), W=S * rng.choice([1, 2, 4]))
    wind = rng.choice(["constant", "field"])
    if kind == "multi":
        k = rng.randint(2, 9)
        h0, w0 = _log_int(rng, 60, 300), _log_int(rng, 60, 300)
        return dict(kind=kind, maps=k, h0=h0, w0=w0, dh=rng.randint(0, 150),
                    dw=rng.randint(0, 150), n=_log_int(rng, 64, 8192),
                    prior=rng.choice(["gauss", "uniform", "near"]), wind=wind)
    H, W = _log_int(rng, 64, 1024), _log_int(rng, 64, 1024)
    if kind == "batch":
        steps = rng.random() < 0.4
        most = min(4096, max(1, (32 << 20) // (H * W))) if steps else 4096
        return dict(kind=kind, H=H, W=W, n=_log_int(rng, 1, most),
                    prior=rng.choice(["gauss", "uniform", "truth", "near"]),
                    wind=wind, steps=steps, cell=rng.random() < 0.3,
                    host=rng.random() < 0.3)
    if kind == "search":
        return dict(kind=kind, H=max(H, 128), W=max(W, 128),
                    lattice=rng.randint(3, 32), reps=rng.randint(1, 16),
                    wind=wind)
    if kind == "burnout":
        return dict(kind=kind, H=H, W=W, n=_log_int(rng, 16, 1024),
                    prior=rng.choice(["gauss", "near"]), wind=wind)
    return dict(kind=kind, H=max(H, 96), W=max(W, 96),
                pop=_log_int(rng, 8, 256), reps=rng.randint(1, 16),
                prior=rng.choice(["gauss", "uniform", "near"]), wind=wind)


# ---------------------------------------------------------------------------
# Inputs.

def _landscape(H, W, wind, seed):
    return synth.landscape(H, W, seed,
                           wind_seed=seed if wind == "field" else None)


def _population(prior, n, seed):
    """(n, 5) parameter vectors: a Table 1 prior, the reference parameters,
    or the spread of a population midway through a calibration."""
    if prior == "gauss":
        return np.clip(synth.gauss_population(n, seed), -30.0, 30.0)
    if prior == "uniform":
        return synth.uniform_population(n, seed)
    p = np.tile(np.asarray(synth.TRUTH_BETA, np.float64), (n, 1))
    if prior == "near":
        p += np.random.default_rng([seed, 17]).normal(0.0, 2.0, (n, 5))
    return p


def _target(m, ign, burnable):
    """A reference scar: the first of 64 fires of the reference parameters
    that burns a hundredth of the burnable cells (else the largest)."""
    n = 64
    p = _population("truth", n, 0)
    g = np.tile(np.asarray(ign, np.int32), (n, 1))
    s = synth.replicate_seeds(n, synth.TARGET_SEED)
    res, _ = m.simulate_batch(p, g, s)
    big = np.flatnonzero(res["burnt"] >= 0.01 * burnable.sum())
    k = int(big[0]) if big.size else int(np.argmax(res["burnt"]))
    _, bs = m.simulate_batch(p[k:k + 1], g[k:k + 1], s[k:k + 1],
                             want_steps=True)
    return bs[0] >= 0


class _State:
    pass


def _device_inputs(st, p, g, s, n):
    st.p = torch.tensor(p, dtype=torch.float64, device="cuda")
    st.g = torch.tensor(g, dtype=torch.int32, device="cuda")
    st.s = torch.tensor(s.view(np.int64), device="cuda")
    st.out = torch.zeros((n, 6), dtype=torch.int32, device="cuda")


def prepare(case, seed):
    st = _State()
    st.case, st.kind = case, case["kind"]
    st.ctx = fire.Context(0, torch.cuda.current_stream())
    if st.kind in ("train", "screen"):
        _prepare_net(st, case, seed)
    elif st.kind == "multi":
        _prepare_multi(st, case, seed)
    else:
        _prepare_map(st, case, seed)
    return st


def _prepare_map(st, case, seed):
    H, W = case["H"], case["W"]
    land = _landscape(H, W, case["wind"], 100 + seed)
    st.m = st.ctx.landscape_upload(land)
    ign = synth.centre_ignition(land.veg)
    burnable = land.veg != 0
    target = _target(st.m, ign, burnable)
    st.m.target_upload(target)
    first = 1 + 1000003 * seed
    if st.kind == "search":
        st.seed = first
        return
    if st.kind in ("batch", "burnout"):
        n = case["n"]
        p = _population(case["prior"], n, seed)
        g = np.tile(np.asarray(ign, np.int32), (n, 1))
        s = synth.replicate_seeds(n, first)
        if case.get("host"):
            st.host = (p, g, s)
            return
        _device_inputs(st, p, g, s, n)
        st.bs = (torch.empty((n, H, W), dtype=torch.int32, device="cuda")
                 if case.get("steps") else None)
        if st.kind == "burnout":
            times = np.asarray((1, 3, 1, 2, 4), np.uint8)[
                np.minimum(land.veg, 4)]
            st.times = torch.tensor(times, device="cuda")
        return
    # a generation: pop individuals, reps replicates each
    pop, reps = case["pop"], case["reps"]
    n = pop * reps
    genes = _population(case["prior"], pop, seed)
    if st.kind == "generation7":
        xy = synth.burnt_area_points(target & burnable, pop, seed)
        genes = np.concatenate([genes, xy], axis=1)
        lo, hi = [-30.0] * 5 + [0.0, 0.0], [30.0] * 5 + [W - 1.0, H - 1.0]
    else:
        lo, hi = [-30.0] * 5, [30.0] * 5
    _device_inputs(st, np.repeat(genes[:, :5], reps, axis=0),
                   np.tile(np.asarray(ign, np.int32), (n, 1)),
                   synth.replicate_seeds(n, first), n)
    f64 = dict(dtype=torch.float64, device="cuda")
    st.genes = torch.tensor(genes, **f64)
    st.next = torch.empty_like(st.genes)
    st.lo, st.hi = torch.tensor(lo, **f64), torch.tensor(hi, **f64)
    st.fit, st.mean = torch.empty(n, **f64), torch.empty(pop, **f64)
    st.ga_seed = first


def _prepare_multi(st, case, seed):
    k, n = case["maps"], case["n"]
    st.maps, ign = [], []
    for i in range(k):
        H, W = case["h0"] + case["dh"] * i, case["w0"] + case["dw"] * i
        land = _landscape(H, W, case["wind"], 100 + 16 * seed + i)
        m = st.ctx.landscape_upload(land)
        ign.append(synth.centre_ignition(land.veg))
        m.target_upload(_target(m, ign[-1], land.veg != 0))
        st.maps.append(m)
    counts = [n // k + (1 if i < n % k else 0) for i in range(k)]
    mos = np.repeat(np.arange(k, dtype=np.int32), counts)
    _device_inputs(st, _population(case["prior"], n, seed),
                   np.asarray(ign, np.int32)[mos],
                   synth.replicate_seeds(n, 1 + 1000003 * seed), n)
    st.mos = torch.tensor(mos, device="cuda")


def _prepare_net(st, case, seed):
    S, n = case["S"], case["n"]
    theta = surrogate.init_params(seed)
    st.net = fire.Net(st.ctx, S, case.get("batch", n))
    st.net.set_params(theta)
    x, target = _net_inputs(case, seed)
    if st.kind == "train":
        st.x, st.t = x, target
        st.loss = torch.zeros(1, dtype=torch.float64, device="cuda")
        st.grad = torch.empty(theta.size, dtype=torch.float32, device="cuda")
        return
    st.planes, st.p, st.g = x
    st.frac = target
    st.x = torch.empty((n, S, S, fire.NET_CIN), dtype=torch.bfloat16,
                       device="cuda")
    st.prob = torch.empty((n, S, S), dtype=torch.float32, device="cuda")
    st.pred = torch.empty(n, dtype=torch.float64, device="cuda")


def _smooth(shape, rng, step=8):
    """Smooth fields in [0, 1], shape (n, S, S)."""
    n, S, _ = shape
    k = max(2, S // step)
    c = torch.tensor(rng.uniform(0.0, 1.0, (n, 1, k, k)), dtype=torch.float32,
                     device="cuda")
    return torch.nn.functional.interpolate(
        c, size=(S, S), mode="bilinear", align_corners=True)[:, 0]


def _net_inputs(case, seed):
    """Network inputs shaped like the automaton's: fuel fractions, slope and
    bearings that vary smoothly, parameters of the GA's prior, burn fractions
    as labels."""
    S, n = case["S"], case["n"]
    rng = np.random.default_rng([seed, 29])
    planes = torch.stack(list(_smooth((10, S, S), rng)), dim=-1).contiguous()
    planes[..., 6:] = planes[..., 6:] * 2 - 1
    params = _population("gauss", n, seed)
    burnt = (_smooth((n, S, S), rng) * 3 - 1).clamp(0, 1).contiguous()
    if case["kind"] == "screen":
        H, W = case["H"], case["W"]
        ign = np.stack([rng.integers(0, H, n), rng.integers(0, W, n)], 1)
        return ((planes, torch.tensor(params, device="cuda"),
                 torch.tensor(ign, dtype=torch.int32, device="cuda")),
                burnt[0].contiguous())
    x = torch.zeros((n, S, S, fire.NET_CIN), dtype=torch.float32,
                    device="cuda")
    x[..., :10] = planes
    x[:, S // 2, S // 2, 10] = 1.0
    x[..., 11:] = torch.tensor(params / 10.0, dtype=torch.float32,
                               device="cuda")[:, None, None, :]
    return x.to(torch.bfloat16), burnt


# ---------------------------------------------------------------------------
# One pass.

def run(st):
    return _RUN[st.kind](st)


def _run_batch(st):
    case = st.case
    if case["host"]:
        res, bs = st.m.simulate_batch(*st.host, want_steps=case["steps"],
                                      cell_uniform=case["cell"])
        fit = fire.fire_fitness(st.ctx, res)
        raw = res.view(np.int32).reshape(-1, 6)
        return (raw, fit, bs) if case["steps"] else (raw, fit)
    st.m.simulate_batch(st.p, st.g, st.s, want_steps=case["steps"],
                        cell_uniform=case["cell"], device=True, out=st.out,
                        burn_step=st.bs)
    return (st.out, st.bs) if case["steps"] else st.out


def _run_generation(st):
    case = st.case
    if st.kind == "generation7":
        fire.fire_snap_ignitions(st.ctx, st.m, st.genes, 5, 6, case["reps"],
                                 device=True, out=st.g)
    st.m.simulate_batch(st.p, st.g, st.s, device=True, out=st.out,
                        longest_first=True)
    fire.fire_fitness(st.ctx, st.out, fire.FITNESS_JACCARD, device=True,
                      out=st.fit)
    fire.fire_group_mean(st.ctx, st.fit, case["reps"], device=True,
                         out=st.mean)
    fire.ga_step(st.ctx, st.genes, st.mean, 10, 50, st.ga_seed, st.lo, st.hi,
                 device=True, out=st.next)
    return st.out, st.g, st.fit, st.mean, st.next


def _run_search(st):
    k = st.case["lattice"]
    return fire.ignition_search(st.ctx, st.m, synth.TRUTH_BETA, k, k,
                                st.case["reps"], st.seed)


def _run_multi(st):
    return fire.fire_simulate_multi(st.ctx, st.maps, st.mos, st.p, st.g, st.s,
                                    device=True, out=st.out)


def _run_burnout(st):
    st.m.simulate_burnout(st.p, st.g, st.s, st.times, device=True, out=st.out)
    return st.out


def _run_train(st):
    st.net.backward(st.x, st.t, st.loss)
    # the gradient stays on the device (fire_net_get with device pointers)
    st.ctx.check(st.ctx.lib.fire_net_get(
        st.ctx.h, st.net.h, fire.NET_GRAD, fire.FIRE_DEVICE_PTRS,
        st.grad.data_ptr()))
    return st.loss, st.grad


def _run_screen(st):
    case = st.case
    S, H, W = case["S"], case["H"], case["W"]
    fire.fire_net_inputs(st.ctx, S, H, W, st.planes, st.p, st.g, st.x)
    st.net.forward(st.x, st.prob)
    fire.fire_net_screen(st.ctx, S, st.prob, st.frac,
                         float(H * W) / (S * S), fire.FITNESS_JACCARD, 0,
                         st.pred)
    return st.prob, st.pred


_RUN = {"batch": _run_batch, "generation": _run_generation,
        "generation7": _run_generation, "search": _run_search,
        "multi": _run_multi, "burnout": _run_burnout, "train": _run_train,
        "screen": _run_screen}


# ---------------------------------------------------------------------------
# What a pass cannot do without.

def _map_bytes(H, W, wind):
    """Covariates and flags of every cell, and the fuel and target planes."""
    return H * W * ((10 if wind == "constant" else 26) + 0.25)


def work(case):
    kind = case["kind"]
    if kind in ("train", "screen"):
        pix = case["n"] * case["S"] ** 2
        weights = 9 * 16 * 128 + 7 * 9 * 128 * 128
        fwd = 2.0 * pix * (weights + 128)
        if kind == "screen":
            return {"bytes": pix * (32 + 4) + 2 * weights, "flops": fwd}
        # input gradients of layers 2..8, weight gradients of all
        back = 2.0 * pix * (7 * 9 * 128 * 128 + weights + 256)
        return {"bytes": pix * 36 + 10 * weights, "flops": fwd + back}
    if kind == "search":
        n, prior = case["lattice"] ** 2 * case["reps"], "truth"
    elif kind.startswith("generation"):
        n, prior = case["pop"] * case["reps"], case["prior"]
    else:
        n, prior = case["n"], case["prior"]
    per_sim = 40 + 8 + 8 + 24
    if kind == "multi":
        shapes = [(case["h0"] + case["dh"] * i, case["w0"] + case["dw"] * i)
                  for i in range(case["maps"])]
    else:
        shapes = [(case["H"], case["W"])]
    cells = sum(h * w for h, w in shapes) / len(shapes)
    nbytes = n * per_sim + sum(_map_bytes(h, w, case["wind"])
                               for h, w in shapes)
    if case.get("steps"):
        nbytes += 4.0 * n * cells
    if kind == "burnout":
        nbytes += cells
    trials = n * cells * _TRIALS_PER_CELL[prior]
    return {"bytes": float(nbytes), "flops": trials * _OPS_PER_TRIAL}


# ---------------------------------------------------------------------------
# The same outputs in 64 bits, without the library.

_DILATION = (1, 1, 2, 4, 8, 16, 32, 64)


def _net64(theta, x):
    """Logits of the network on x (1, S, S, 16), all float64."""
    off, h, S = 0, x, x.shape[1]
    for d in _DILATION:
        ci = h.shape[-1]
        w = theta[off:off + 128 * 9 * ci].view(128, 9, ci)
        off += 128 * 9 * ci
        z = theta[off:off + 128]
        off += 128
        hp = torch.nn.functional.pad(h, (0, 0, d, d, d, d))
        for t in range(9):
            r, c = (t // 3) * d, (t % 3) * d
            z = z + hp[:, r:r + S, c:c + S, :] @ w[:, t, :].T
        h = torch.relu(z)
    return h @ theta[off:off + 128] + theta[off + 128]


def exact(case, seed):
    if case["kind"] not in ("train", "screen"):
        return None     # whole numbers, and ratios and means of them
    S, n = case["S"], case["n"]
    theta = torch.tensor(surrogate.init_params(seed).astype(np.float64),
                         device="cuda")
    x, t = _net_inputs(case, seed)
    if case["kind"] == "screen":
        planes, p, g = x
        prob = torch.empty((n, S, S), dtype=torch.float64, device="cuda")
        fr, fc = case["H"] // S, case["W"] // S
        for i in range(n):
            xi = torch.zeros((1, S, S, 16), dtype=torch.float64,
                             device="cuda")
            xi[0, ..., :10] = planes.double()
            xi[0, int(g[i, 0]) // fr, int(g[i, 1]) // fc, 10] = 1.0
            xi[0, ..., 11:] = p[i] / 10.0
            prob[i] = torch.sigmoid(_net64(theta, xi))[0]
        td = t.double()
        inter = (prob * td).sum((1, 2))
        both = prob.sum((1, 2)) + td.sum()
        return prob, (both - 2 * inter) / (both - inter)
    theta.requires_grad_(True)
    loss = torch.zeros(1, dtype=torch.float64, device="cuda")
    for i in range(n):
        z = _net64(theta, x[i:i + 1].double())
        part = torch.nn.functional.binary_cross_entropy_with_logits(
            z, t[i:i + 1].double(), reduction="sum") / (n * S * S)
        part.backward()
        loss += part.detach()
    return loss, theta.grad
