"""The work that users of this framework have it do, as measurable cases.

Every case continues one seeded Markov chain (or takes one training gradient)
through the package's public entry points and returns what a program reads
back: the configuration and the recorded series, or the loss and the gradients.

Kinds of case:
  sweep  checkerboard Metropolis sweeps of one Ising lattice (int8 or packed),
         with the default kernel choice, as a program that does not tune has it
  batch  uneven replicas with parallel tempering in one persistent launch
  sw     Swendsen-Wang cluster steps
  xy     the XY model (64: the paper's precision, 32: single precision)
  quad   the four-sublattice lattices (square-octagon, square NN + NNN)
  train  loss and gradients of the learned block proposal's network
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2402_06415_gb300 as ising
from paper_2402_06415_gb300 import learned, workloads

BETA_C = 0.4406868
LARGEST = 16384 * 16384 * 10  # site updates of the largest listed pass


def listed():
    return [
        # the study lattice of the exact checks: E and M after every sweep, bytes per spin
        {"name": "sweep_int8_64", "kind": "sweep", "layout": "int8", "L": 64, "beta": BETA_C, "sweeps": 100,
         "every": 1},
        # the plain chain that every speed-up at beta_c is quoted against (tau_int at L = 256)
        {"name": "sweep_256", "kind": "sweep", "layout": "bits", "L": 256, "beta": BETA_C, "sweeps": 100, "every": 1},
        # a size that is no multiple of a word or tile, as finite-size scans have
        {"name": "sweep_1000", "kind": "sweep", "layout": "bits", "L": 1000, "beta": 0.40, "sweeps": 40, "every": 10},
        # a middle size of the same scans
        {"name": "sweep_2048", "kind": "sweep", "layout": "bits", "L": 2048, "beta": 0.50, "sweeps": 40, "every": 10},
        # the headline lattice
        {"name": "sweep_16384", "kind": "sweep", "layout": "bits", "L": 16384, "beta": BETA_C, "sweeps": 10,
         "every": 10},
        # 4096 replicas, 64 ladders of 64 temperatures, exchanges every 10 sweeps
        {"name": "batch_4096", "kind": "batch", "ladders": 64, "betas": 64, "sizes": 6, "sweeps": 20},
        # cluster chain of a tau_int measurement
        {"name": "sw_256", "kind": "sw", "L": 256, "beta": BETA_C, "steps": 20, "every": 1},
        # cluster steps of a large lattice
        {"name": "sw_4096", "kind": "sw", "L": 4096, "beta": BETA_C, "steps": 2, "every": 1},
        # the paper's own benchmark: L = 32, T = 0.85, double precision
        {"name": "xy64_32", "kind": "xy", "precision": 64, "L": 32, "T": 0.85, "sweeps": 100, "every": 1},
        # a production XY lattice in single precision
        {"name": "xy32_512", "kind": "xy", "precision": 32, "L": 512, "T": 0.85, "sweeps": 100, "every": 10},
        # the square-octagon lattice of the paper's partition study
        {"name": "quad_oct_1024", "kind": "quad", "lattice": "sqoct", "Lc": 1024, "J2": 1.0, "beta": BETA_C,
         "sweeps": 100, "every": 10},
        # one minibatch of the proposal's training: 512 windows, 8 network stages each
        {"name": "train_512", "kind": "train", "block": 16, "windows": 512},
    ]


def _even(v, lo):
    return max(lo, 2 * int(round(v / 2)))


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["sweep", "sweep", "sweep", "int8", "batch", "sw", "xy", "quad", "train"])
    beta = rng.choice([0.40, BETA_C, 0.50, round(rng.uniform(0.3, 0.6), 4)])
    if kind == "int8":
        return {"kind": "sweep", "layout": "int8", "L": _even(_log(rng, 8, 160), 8), "beta": beta,
                "sweeps": rng.randint(20, 150), "every": rng.choice([0, 1, 10])}
    if kind == "sweep":
        L = _even(_log(rng, 16, 16384), 16)
        if L >= 256 and rng.random() < 0.4:
            L = min(16384, 256 * max(1, round(L / 256)))
        most = max(1, min(200, LARGEST // (L * L)))
        return {"kind": "sweep", "layout": "bits", "L": L, "beta": beta, "sweeps": rng.randint(max(1, most // 4), most),
                "every": rng.choice([0, 1, 5, 10])}
    if kind == "batch":
        return {"kind": "batch", "ladders": rng.randint(4, 64), "betas": rng.randint(8, 64), "sizes": rng.randint(0, 99),
                "sweeps": rng.randint(5, 25)}
    if kind == "sw":
        L = _even(_log(rng, 16, 4096), 16)
        if L >= 1024 and rng.random() < 0.5:
            L = 128 * max(1, round(L / 128))
        return {"kind": "sw", "L": L, "beta": beta, "steps": rng.randint(2, 20) if L < 1024 else rng.randint(1, 2),
                "every": rng.choice([0, 1])}
    if kind == "xy":
        p = rng.choice([32, 64])
        return {"kind": "xy", "precision": p, "L": _even(_log(rng, 8, 1024 if p == 32 else 256), 8),
                "T": round(rng.uniform(0.6, 1.1), 3), "sweeps": rng.randint(20, 100), "every": rng.choice([1, 10])}
    if kind == "quad":
        return {"kind": "quad", "lattice": rng.choice(["sqoct", "square"]), "Lc": int(round(_log(rng, 8, 1024))),
                "J2": rng.choice([0.0, 0.5, 1.0]), "beta": beta, "sweeps": rng.randint(20, 100), "every": rng.choice([1, 10])}
    return {"kind": "train", "block": rng.choice([8, 16]), "windows": rng.randint(32, 512)}


# ---- inputs ----

def _gauss_field(rng, L, spectrum):
    """A real periodic Gaussian field with the given power spectrum of the wave numbers."""
    k = 2 * np.pi * np.fft.fftfreq(L)
    lap = 4 * np.sin(k[:, None] / 2) ** 2 + 4 * np.sin(k[None, :] / 2) ** 2
    lap[0, 0] = 1.0
    amp = np.sqrt(spectrum(lap))
    amp[0, 0] = 0.0
    return np.fft.ifft2(np.fft.fft2(rng.standard_normal((L, L))) * amp).real


def _xy_spins(case, seed):
    """Spin-wave angles of the temperature: the state a thermalised XY lattice is near."""
    rng = np.random.default_rng([seed, case["L"]])
    th = _gauss_field(rng, case["L"], lambda q: case["T"] / q) + rng.uniform(0, 2 * np.pi)
    return np.stack([np.cos(th), np.sin(th)], axis=-1)


def _windows(case, seed):
    """(block + 2)^2 windows of spins with critical correlations, S(k) ~ k^(-7/4)."""
    rng = np.random.default_rng([seed, case["windows"], case["block"]])
    f = _gauss_field(rng, 512, lambda q: q ** -0.875)
    return learned.extract_windows(np.where(f > 0, 1, -1).astype(np.int8), case["windows"], case["block"], rng)


def prepare(case, seed):
    kind, seed = case["kind"], int(seed)
    stream = torch.cuda.current_stream()
    if kind == "sweep":
        L, i8 = case["L"], case["layout"] == "int8"
        lat = ising.Lattice(L, case["beta"], ising.ISING_LAYOUT_I8 if i8 else ising.ISING_LAYOUT_BITS, stream=stream,
                            seed=seed)
        lat.sweep(20, 0)  # past the random start: domains have formed
        out = (torch.empty((L, L), dtype=torch.int8, device="cuda") if i8 else
               torch.empty((2, L, ising.ising_words_per_row(L)), dtype=torch.int32, device="cuda"))
        return {"case": case, "lat": lat, "out": out, "records": _records(20, case["sweeps"], case["every"])}
    if kind == "sw":
        L = case["L"]
        lat = ising.Lattice(L, case["beta"], ising.ISING_LAYOUT_BITS, stream=stream, seed=seed)
        lat.sw_step(4, 0)
        out = torch.empty((2, L, ising.ising_words_per_row(L)), dtype=torch.int32, device="cuda")
        return {"case": case, "lat": lat, "out": out, "records": case["steps"] if case["every"] else 0}
    if kind == "batch":
        Ls = workloads.batch_ladder_sizes(case["ladders"], case["sizes"])
        b = ising.Batch(Ls, workloads.batch_betas(case["betas"]), workloads.BATCH_PT_EVERY, stream=stream, seed=seed)
        b.run(20)
        return {"case": case, "batch": b}
    if kind == "xy":
        xy = ising.XY(case["L"], 1.0 / case["T"], case["precision"], stream=stream, seed=seed)
        xy.set_spins(_xy_spins(case, seed))
        return {"case": case, "xy": xy, "records": _records(0, case["sweeps"], case["every"])}
    if kind == "quad":
        q = ising.Quad(ising.ISING_QUAD_SQOCT if case["lattice"] == "sqoct" else ising.ISING_QUAD_SQUARE, case["Lc"],
                       case["beta"], 1.0, case["J2"], stream=stream, seed=seed)
        q.sweep(20, 0)
        return {"case": case, "quad": q, "records": _records(20, case["sweeps"], case["every"])}
    tr = learned.Trainer(case["block"], seed=seed & 0xffff, stream=stream, proposal=ising.ISING_PROPOSAL_STAGED,
                         precision=ising.ISING_NN_TRAIN_BF16_TC)
    return {"case": case, "trainer": tr, "windows": torch.from_numpy(_windows(case, seed)).cuda()}


def _records(t0, n, every):
    """Records made by sweeps t0 .. t0 + n - 1 (later passes make as many or one more)."""
    return (t0 + n) // every - t0 // every if every else 0


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind in ("sweep", "sw"):
        lat = state["lat"]
        if kind == "sw":
            lat.sw_step(case["steps"], case["every"])
        else:
            lat.sweep(case["sweeps"], case["every"])
        if case.get("layout") == "int8":
            ising.ising_get_spins_device(lat.ctx, state["out"])
        else:
            ising.ising_get_bits_device(lat.ctx, state["out"])
        if not state["records"]:
            return {"spins": state["out"]}
        E, M = lat.series(state["records"])
        return {"spins": state["out"], "E": E, "M": M}
    if kind == "batch":
        b = state["batch"]
        b.run(case["sweeps"])
        perm, E, M = b.state()
        acc, att = b.swap_counts()
        last = len(b.Ls) - 1
        return {"perm": perm, "E": E, "M": M, "accepted": acc, "attempted": att, "first": b.spins(0, 0),
                "last": b.spins(last, b.n_beta - 1)}
    if kind == "xy":
        xy = state["xy"]
        xy.sweep(case["sweeps"], case["every"])
        out = {"spins": xy.spins()}
        if state["records"]:
            out["E"], out["Mx"], out["My"] = xy.series(state["records"])
        return out
    if kind == "quad":
        q = state["quad"]
        q.sweep(case["sweeps"], case["every"])
        out = {"spins": q.spins()}
        if state["records"]:
            out["B1"], out["B2"], out["M"] = q.series(state["records"])
        return out
    loss, grads = ising.ising_nn_loss_grad(state["trainer"].h, state["windows"], case["windows"])
    return {"loss": np.array([loss], dtype=np.float32), **ising.nn_unflatten(grads)}


# ---- work a pass cannot do without ----
# A 32-site word of a Metropolis half sweep needs about 112 integer operations:
# 1.95 Philox4x32-10 blocks at 40, their bit planes, the neighbour classes and
# the update; an XY trial about 70 (half a block, sin, cos, dE).

def work(case):
    kind = case["kind"]
    if kind == "sweep":
        L, n = case["L"], case["sweeps"]
        state = L * L if case["layout"] == "int8" else L * L / 8
        return {"bytes": 2 * state + 16 * _records(20, n, case["every"]), "flops": 3.5 * L * L * n}
    if kind == "batch":
        Ls = workloads.batch_ladder_sizes(case["ladders"], case["sizes"])
        sites = case["betas"] * sum(L * L for L in Ls)
        words = case["betas"] * sum(2 * L * ((L // 2 + 31) // 32) for L in Ls)
        return {"bytes": 8 * words, "flops": 3.5 * sites * case["sweeps"]}
    if kind == "sw":  # per site: half a block for its two bonds, their tests, a union or two
        L, n = case["L"], case["steps"]
        return {"bytes": 2 * L * L / 8 + 16 * n, "flops": 35.0 * L * L * n}
    if kind == "xy":
        L, n = case["L"], case["sweeps"]
        return {"bytes": 2 * L * L * (case["precision"] // 4), "flops": 70.0 * L * L * n}
    if kind == "quad":
        N = 4 * case["Lc"] ** 2
        return {"bytes": 2 * N / 8, "flops": (3.5 if case["lattice"] == "sqoct" else 5.0) * N * case["sweeps"]}
    n1, n2, n3, _ = _stage_positions(case["block"])
    per = 2 * 2 * 18 * 32 * n1 + 3 * 2 * 288 * 32 * n2 + 3 * 2 * 288 * n3
    return {"bytes": case["windows"] * (case["block"] + 2) ** 2 + 8 * 10145, "flops": float(per) * case["windows"]}


def _grow(m):
    p = np.pad(m, 1)
    F = m.shape[0]
    return np.any([p[a:a + F, b:b + F] for a in range(3) for b in range(3)], axis=0)


def _stage_positions(block):
    """Positions of layers 1, 2 and 3 that the loss terms depend on, over all network stages, and per
    stage (known mask of the frame, mask of the interior's loss terms)."""
    so, ex = ising.ising_proposal_schedule(block, ising.ISING_PROPOSAL_STAGED)
    F = block + 2
    n1 = n2 = n3 = 0
    stages = []
    for k in np.flatnonzero(ex == 0):
        sites = np.zeros((F, F), dtype=bool)
        sites[1:-1, 1:-1] = so == k
        known = np.ones((F, F), dtype=bool)
        known[1:-1, 1:-1] = so < k
        known[[0, 0, -1, -1], [0, -1, 0, -1]] = False
        l2 = _grow(sites)
        n1, n2, n3 = n1 + int(_grow(l2).sum()), n2 + int(l2.sum()), n3 + int(sites.sum())
        stages.append((known, so == k))
    return n1, n2, n3, stages


# ---- the same in 64 bits ----

def exact(case, seed):
    """Double-precision results.  The integer chains need none; a single-precision XY chain has none (a rounding
    that tips one trial changes every later one)."""
    if case["kind"] == "xy" and case["precision"] == 64 and case["L"] <= 256:
        return _xy_exact(case, int(seed))
    if case["kind"] == "train":
        return _train_exact(case, int(seed))
    return None


def _philox(c0, c1, c2, c3, seed):
    """Philox4x32-10 (Salmon et al., SC'11) of arrays of counters."""
    m32 = np.uint64(0xffffffff)
    c = [np.broadcast_to(np.asarray(v, dtype=np.uint64), c0.shape) for v in (c0, c1, c2, c3)]
    k0, k1 = seed & 0xffffffff, (seed >> 32) & 0xffffffff
    for _ in range(10):
        p0, p1 = c[0] * np.uint64(0xD2511F53), c[2] * np.uint64(0xCD9E8D57)
        c = [(p1 >> np.uint64(32)) ^ c[1] ^ np.uint64(k0), p1 & m32, (p0 >> np.uint64(32)) ^ c[3] ^ np.uint64(k1),
             p0 & m32]
        k0, k1 = (k0 + 0x9E3779B9) & 0xffffffff, (k1 + 0xBB67AE85) & 0xffffffff
    return c


def _xy_exact(case, seed):
    L, beta = case["L"], 1.0 / case["T"]
    half = L // 2
    u = _xy_spins(case, seed)
    y, j = np.divmod(np.arange(L * half), half)
    E, Mx, My = [], [], []
    block = np.arange((L * half + 1) // 2, dtype=np.uint64)
    for t in range(case["sweeps"]):
        for c in range(2):
            r = np.stack(_philox(block, t, 0, 9 << 16 | c << 8, seed), axis=1).reshape(-1, 2)[:L * half]
            w = (r >> np.uint64(8)).astype(np.float64) / 16777216.0
            x = 2 * j + ((y + c) & 1)
            th = 2 * np.pi * w[:, 0]
            h = u[y, (x + 1) % L] + u[y, (x - 1) % L] + u[(y + 1) % L, x] + u[(y - 1) % L, x]
            new = np.stack([np.cos(th), np.sin(th)], axis=1)
            dE = -((new - u[y, x]) * h).sum(1)
            ok = (dE <= 0) | (w[:, 1] < np.exp(-beta * np.maximum(dE, 0)))
            u[y[ok], x[ok]] = new[ok]
        if case["every"] and (t + 1) % case["every"] == 0:
            E.append(-(u * (np.roll(u, -1, 0) + np.roll(u, -1, 1))).sum())
            Mx.append(u[..., 0].sum())
            My.append(u[..., 1].sum())
    out = {"spins": u}
    if E:
        out.update(E=np.array(E), Mx=np.array(Mx), My=np.array(My))
    return out


def _train_exact(case, seed):
    """Loss and gradients of the training objective by torch's autograd in double precision."""
    B, n = case["block"], case["windows"]
    p = {k: torch.from_numpy(v.astype(np.float64)).cuda().requires_grad_()
         for k, v in learned.init_params(seed & 0xffff).items()}
    win = torch.from_numpy(_windows(case, seed)).cuda().double()

    def conv(x, W, b):
        cols = torch.nn.functional.unfold(x, 3, padding=1)
        return (W.reshape(W.shape[0], -1) @ cols).reshape(x.shape[0], W.shape[0], B + 2, B + 2) + b[:, None, None]

    total = 0.0
    for known, sites in _stage_positions(B)[3]:
        k = torch.from_numpy(known).cuda().double()
        m = torch.from_numpy(sites).cuda().double()
        for s in range(0, n, 128):
            w = win[s:s + 128]
            x = torch.stack([w * k, k.expand_as(w)], dim=1)
            z = conv(conv(conv(x, p["W1"], p["b1"]).relu(), p["W2"], p["b2"]).relu(), p["W3"], p["b3"])[:, 0, 1:-1, 1:-1]
            y = (w[:, 1:-1, 1:-1] + 1) / 2
            loss = (torch.nn.functional.binary_cross_entropy_with_logits(z, y, reduction="none") * m).sum() / n
            loss.backward()
            total += float(loss)
    return {"loss": np.array([total]), **{k: v.grad.cpu().numpy() for k, v in p.items()}}
