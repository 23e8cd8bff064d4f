"""What a user of the framework has it do, as cases that can be timed.

A case is a dict of plain values; ``prepare`` makes what the user's program
has in hand before the call, ``run`` makes the call through the public entry
points (``Lattice``, ``Batch``, ``Mlp``, ``lbm_field_pressure_jump_static``)
and returns its results, ``exact`` gives the same results in 64 bits from
plain torch (no code of this repository), ``work`` what one call cannot do
without.  The kinds:

- ``run``: a single lattice that is already running goes on for some steps
  and its density is read (the oscillation experiment, a droplet relaxing).
- ``whole``: host fields in, some steps, host fields out (the benchmark's
  end-to-end call).
- ``slabs``: a small FP64 batch of flat interfaces (coexistence densities).
- ``window``: one interval of the Laplace sampling window: equal droplets
  stepped together, then every droplet sampled twice (discs that follow it).
- ``sweep``: uneven droplets stepped together, then each one's status,
  Laplace sample and peak velocity, as a sweep harvests them.
- ``probe``: macroscopic fields, run statistics and a Laplace sample of a
  lattice with a flow.
- ``train`` / ``pick``: the surrogate's training, and its predictions and
  kappa picks.
- ``static``: Laplace sums over a density field in device memory.
"""
import math

import numpy as np
import torch

S_CFG = (1.0, 1.1, 1.1, 1.0, 1.1, 1.0, 1.1, 1.0, 1.0)   # relaxation rates of the droplet workloads
S_ONE = (1.0,) * 9                                       # and of the paper's van der Waals and Peng-Robinson runs
TC_CS = 0.0943287                                        # critical temperature, Carnahan-Starling a = 1, b = 4
TC_VDW = 8.0 / 27.0 * (9.0 / 49.0) / (2.0 / 21.0)        # van der Waals a = 9/49, b = 2/21
PR_A, PR_B, PR_OMEGA = 0.0703, 2.0 / 21.0, 0.344
TC_PR = 0.0778 * PR_A / (0.45724 * PR_B)


def listed():
    return [
        # the plain-method workload: one small droplet, 10^4 steps in all, looked at every 200
        dict(name="drop_64_f32", kind="run", law="cs", nx=64, ny=64, prec="f32", steps=200, visc=False),
        # the oscillation experiment: a Peng-Robinson ellipse with density-dependent viscosity, its density
        # read every 10 steps (the smallest call)
        dict(name="oscillation_120_f32", kind="run", law="pr", nx=120, ny=120, prec="f32", steps=10, visc=True),
        # flat interfaces at six values of A: the coexistence runs of Figs. 1-2
        dict(name="slabs_6x128x4_f64", kind="slabs", n=6, nx=128, ny=4, steps=400),
        # the Laplace sweep's 60 droplets, one of its 101 sampling intervals
        dict(name="window_60x256_f32", kind="window", n=60, L=256, steps=20),
        # the batched uneven sweep: 64 droplets of 128^2 to 1024^2, and its harvest
        dict(name="sweep_64_uneven_f32", kind="sweep", n=64, sizes_seed=7228, lo=128, hi=1024, steps=40),
        # the benchmark's end-to-end call: spinodal decomposition, FP32 fields in and out
        dict(name="spinodal_4096_f32", kind="whole", nx=4096, ny=4096, prec="f32", steps=20, flow=False),
        # the same method in FP64 (the precision of the parity and sigma checks)
        dict(name="spinodal_1024_f64", kind="whole", nx=1024, ny=1024, prec="f64", steps=20, flow=False),
        # a ragged lattice (no tile shape divides it) with an initial flow, every field read
        dict(name="flow_1531x1117_f32", kind="whole", nx=1531, ny=1117, prec="f32", steps=24, flow=True),
        # what is read at the end of an FP64 run
        dict(name="probe_512_f64", kind="probe", nx=512, ny=512, prec="f64"),
        # the surrogate: 2000 samples, minibatches of 128 (four of its 600 epochs)
        dict(name="train_2000", kind="train", n=2000, batch=128, epochs=4),
        # its use: the predictions of the whole data set and 16 kappa picks
        dict(name="pick_2000_16", kind="pick", n=2000, m=16),
        # Laplace sums of a caller's field, the largest the entry point takes
        dict(name="static_4096", kind="static", nx=4096, ny=4096),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("run", "run", "whole", "whole", "slabs", "window", "sweep", "probe", "train", "pick", "static"))
    if kind == "run":
        law = rng.choice(("cs", "cs", "pr"))
        prec = rng.choice(("f32", "f32", "f64"))
        lo, hi = (100, 160) if law == "pr" else (32, 512 if prec == "f32" else 160)
        return dict(kind=kind, law=law, nx=_log(rng, lo, hi), ny=_log(rng, lo, hi), prec=prec,
                    steps=_log(rng, 10, 200 if prec == "f32" else 60), visc=law == "pr" and rng.random() < 0.5)
    if kind == "whole":
        prec = rng.choice(("f32", "f32", "f64"))
        hi = 4096 if prec == "f32" else 1400
        return dict(kind=kind, nx=_log(rng, 256, hi), ny=_log(rng, 256, hi), prec=prec, steps=rng.randint(8, 20),
                    flow=rng.random() < 0.4)
    if kind == "slabs":
        return dict(kind=kind, n=rng.randint(1, 12), nx=_log(rng, 64, 256), ny=rng.choice((4, 5, 8, 16)),
                    steps=_log(rng, 100, 400))
    if kind == "window":
        return dict(kind=kind, n=rng.randint(8, 60), L=_log(rng, 192, 300), steps=20)
    if kind == "sweep":
        return dict(kind=kind, n=rng.randint(8, 60), sizes_seed=rng.randint(0, 10 ** 6), lo=100,
                    hi=rng.choice((512, 800, 1000)), steps=rng.randint(10, 40))
    if kind == "probe":
        return dict(kind=kind, nx=_log(rng, 128, 1600), ny=_log(rng, 128, 1600), prec=rng.choice(("f32", "f64")))
    if kind == "train":
        return dict(kind=kind, n=_log(rng, 300, 4000), batch=rng.choice((32, 64, 100, 128, 256)),
                    epochs=rng.randint(1, 4))
    if kind == "pick":
        return dict(kind=kind, n=_log(rng, 16, 8192), m=_log(rng, 1, 256))
    return dict(kind=kind, nx=_log(rng, 64, 4096), ny=_log(rng, 64, 4096))


# ---- inputs ----------------------------------------------------------------
def _pressure(law, p, rho):
    if law == "cs":
        n = p["b"] * rho / 4.0
        return p["K"] * (rho * p["T"] * (1.0 + n + n * n - n * n * n) / (1.0 - n) ** 3 - p["a"] * rho * rho)
    if law == "vdw":
        return p["K"] * (rho * p["T"] / (1.0 - p["b"] * rho) - p["a"] * rho * rho)
    br = p["b"] * rho
    m = 0.37464 + 1.54226 * PR_OMEGA - 0.26992 * PR_OMEGA ** 2
    alpha = (1.0 + m * (1.0 - math.sqrt(p["T"] / TC_PR))) ** 2
    return p["K"] * (rho * p["T"] / (1.0 - br) - p["a"] * alpha * rho * rho / (1.0 + 2.0 * br - br * br))


def _law(law, t):
    """Constants of a law at t times its critical temperature."""
    if law == "cs":
        return dict(law=law, a=1.0, b=4.0, K=1.0, T=t * TC_CS)
    if law == "vdw":
        return dict(law=law, a=9.0 / 49.0, b=2.0 / 21.0, K=0.3, T=t * TC_VDW)
    return dict(law=law, a=PR_A, b=PR_B, K=0.5, T=t * TC_PR)


def _cs_coexistence(t):
    """Gas and liquid densities of equal pressure and chemical potential."""
    p = _law("cs", t)
    pr = lambda r: _pressure("cs", p, r)
    mu = lambda r: p["T"] * (math.log(r) + (8 * r - 9 * r * r + 3 * r ** 3) / (1 - r) ** 3) - 2.0 * r
    grid = np.geomspace(1e-7, 0.95, 20001)
    pg = pr(grid)
    d = np.diff(pg)
    i1 = int(np.argmax(d < 0))
    i2 = i1 + int(np.argmax(d[i1:] > 0))

    def root(p0, lo, hi):
        for _ in range(80):
            mid = 0.5 * (lo + hi)
            if pr(mid) < p0:
                lo = mid
            else:
                hi = mid
        return 0.5 * (lo + hi)

    a, b = max(float(pg[i2]), 1e-12), float(pg[i1])
    for _ in range(80):
        p0 = 0.5 * (a + b)
        rg, rl = root(p0, 1e-9, float(grid[i1])), root(p0, float(grid[i2]), 0.95)
        if mu(rl) > mu(rg):
            a = p0
        else:
            b = p0
    return rg, rl


def _distance(nx, ny, cx, cy, ax=1.0, ay=1.0):
    dx = np.arange(nx, dtype=np.float64)[None, :] - cx
    dy = np.arange(ny, dtype=np.float64)[:, None] - cy
    dx -= nx * np.round(dx / nx)
    dy -= ny * np.round(dy / ny)
    return np.sqrt((dx / ax) ** 2 + (dy / ay) ** 2)


def _drop(nx, ny, R, rg, rl, width, rng, ellipse=1.0):
    """A drop near the centre; radius and centre vary with the seed."""
    cx, cy = nx / 2.0 + rng.uniform(-0.5, 0.5), ny / 2.0 + rng.uniform(-0.5, 0.5)
    R = R * rng.uniform(0.97, 1.03)
    r = _distance(nx, ny, cx, cy, math.sqrt(ellipse), 1.0 / math.sqrt(ellipse))
    return rg + 0.5 * (rl - rg) * (1.0 - np.tanh(2.0 * (r - R) / width))


def _lattices(case, seed):
    """The lattices of a case: per lattice its size, law, A, kappa, rates,
    reference density, initial fields and viscosity law."""
    rng = np.random.default_rng([int(seed), 7228])
    kind = case["kind"]
    out = []
    if kind == "run" and case["law"] == "pr":
        nx, ny = case["nx"], case["ny"]
        rho = _drop(nx, ny, 0.24 * min(nx, ny), 0.0167, 7.17, 4.0, rng, ellipse=30.0 / 27.0)
        visc = (0.2, 0.05, 0.0167, 7.17) if case["visc"] else None
        out.append(dict(nx=nx, ny=ny, p=_law("pr", 0.8), A=-0.3, kappa=float(rng.uniform(-0.2, 0.5)), s=S_ONE, ref=0.0167,
                        rho=rho, visc=visc))
    elif kind == "run":
        rg, rl = _cs_coexistence(0.7)
        nx, ny = case["nx"], case["ny"]
        out.append(dict(nx=nx, ny=ny, p=_law("cs", 0.7), A=-0.85, kappa=0.0, s=S_CFG, ref=rg,
                        rho=_drop(nx, ny, 15.0 / 64.0 * min(nx, ny), rg, rl, 2.0, rng)))
    elif kind in ("whole", "probe"):
        nx, ny = case["nx"], case["ny"]
        rho = rng.random((ny, nx), dtype=np.float32)
        if case["prec"] == "f64":
            rho = rho.astype(np.float64)
        rho *= 0.005
        rho += 0.2475
        d = dict(nx=nx, ny=ny, p=_law("cs", 0.7), A=-0.85, kappa=0.3, s=S_CFG, ref=0.25, rho=rho)
        if kind == "probe":
            rg, rl = _cs_coexistence(0.7)
            d.update(ref=rg, rho=_drop(nx, ny, 0.2 * min(nx, ny), rg, rl, 4.0, rng))
        if kind == "probe" or case["flow"]:
            a, b = rng.uniform(0, 2 * math.pi, 2)
            y, x = np.arange(ny)[:, None] * (2 * math.pi / ny), np.arange(nx)[None, :] * (2 * math.pi / nx)
            d.update(ux=0.02 + 0.02 * np.sin(y + a) + 0.0 * x, uy=0.01 + 0.02 * np.sin(2 * x + b) + 0.0 * y)
        if case["prec"] == "f32":
            for k in ("rho", "ux", "uy"):
                if k in d:
                    d[k] = d[k].astype(np.float32)
        out.append(d)
    elif kind == "slabs":
        nx, ny = case["nx"], case["ny"]
        x = np.arange(nx, dtype=np.float64)
        for A in np.linspace(-0.9, 0.5, case["n"]) + rng.uniform(0, 0.02, case["n"]):
            rl, rg = 5.8 * rng.uniform(0.99, 1.01), 1.47
            prof = rg + 0.5 * (rl - rg) * (np.tanh(0.5 * (x - nx / 4.0)) - np.tanh(0.5 * (x - 0.75 * nx)))
            out.append(dict(nx=nx, ny=ny, p=_law("vdw", 0.9), A=float(A), kappa=0.0, s=S_ONE, ref=rg,
                            rho=np.broadcast_to(prof[None, :], (ny, nx)).copy()))
    elif kind == "window":
        L = case["L"]
        combos = [(t, k, R) for t in (0.6, 0.7, 0.8) for k in (0.0, 0.1, 0.3, 0.5) for R in (20, 30, 40, 50, 60)]
        for i in range(case["n"]):
            t, k, R = combos[i % len(combos)]
            rg, rl = _cs_coexistence(t)
            R = R * L / 256.0
            out.append(dict(nx=L, ny=L, p=_law("cs", t), A=-0.85, kappa=k, s=S_CFG, ref=rg, R=R,
                            rho=_drop(L, L, R, rg, rl, 2.0, rng)))
    elif kind == "sweep":
        size = np.random.default_rng(case["sizes_seed"])   # the sizes belong to the case, not to the seed
        sizes = [L for L in (128, 256, 512, 1024) if case["lo"] <= L <= case["hi"]]
        for i in range(case["n"]):
            L = int(size.choice(sizes)) if case["lo"] == 128 else int(round(case["lo"] * (case["hi"] / case["lo"]) ** size.random()))
            t, A, k = round(float(rng.uniform(0.6, 0.85)), 2), float(rng.uniform(-0.9, -0.8)), float(rng.uniform(0, 0.6))
            rg, rl = _cs_coexistence(t)
            out.append(dict(nx=L, ny=L, p=_law("cs", t), A=A, kappa=k, s=S_CFG, ref=rg, R=0.2 * L,
                            rho=_drop(L, L, 0.2 * L, rg, rl, 2.0, rng)))
    return out


def _samples(case, seed):
    """The surrogate's data: (T/Tc, A, kappa) -> (log sigma, rho_l, rho_g,
    log u_max), smooth laws of the size the simulations give, with noise."""
    rng = np.random.default_rng([int(seed), 1])
    n = case["n"]
    X = np.stack([rng.uniform(0.6, 0.85, n), rng.uniform(-0.9, -0.8, n), rng.uniform(0, 0.6, n)], 1)
    t, A, k = X.T
    Y = np.stack([np.log((1.02 - k) * (0.95 - t) ** 1.3 * 0.06 * (1 + 0.3 * (A + 0.85))), 0.28 + 0.45 * (0.85 - t),
                  0.03 * t ** 4 * (1 + A / 10), np.log(2e-3 * (1.0 - t) * (1.1 - k))], 1)
    Y += rng.normal(0, 1e-3, Y.shape) * np.abs(Y)
    W = [(rng.random((r, c)) * 2 - 1) * math.sqrt(6.0 / (r + c)) for r, c in ((64, 3), (64, 64), (4, 64))]
    return X.astype(np.float32), Y.astype(np.float32), W


def _flat(W1, b1, W2, b2, W3, b3):
    return np.concatenate([np.asarray(v, dtype=np.float64).ravel() for v in (W1, b1, W2, b2, W3, b3)]).astype(np.float32)


def _norm(X, Y):
    X, Y = X.astype(np.float64), Y.astype(np.float64)
    return [v.astype(np.float32) for v in (X.mean(0), X.std(0) + 1e-12, Y.mean(0), Y.std(0) + 1e-12)]


def _gelu(z):
    return 0.5 * z * (1.0 + torch.erf(z / math.sqrt(2.0)))


def _fitted(case, seed):
    """A surrogate that follows its data: random hidden layers, the last one
    by least squares (on 512 samples of its own)."""
    X, Y, W = _samples(dict(n=512), seed)
    norm = _norm(X, Y)
    x = torch.from_numpy((X.astype(np.float64) - norm[0]) / norm[1])
    y = (Y.astype(np.float64) - norm[2]) / norm[3]
    h = _gelu(_gelu(x @ torch.from_numpy(W[0]).T) @ torch.from_numpy(W[1]).T).numpy()
    h = np.concatenate([h, np.ones((len(h), 1))], 1)
    c = np.linalg.solve(h.T @ h + 1e-3 * np.eye(65), h.T @ y)
    return norm, _flat(W[0], np.zeros(64), W[1], np.zeros(64), c[:64].T, c[64])


def _picks(case, seed):
    rng = np.random.default_rng([int(seed), 2])
    X = np.stack([rng.uniform(0.6, 0.85, case["n"]), rng.uniform(-0.9, -0.8, case["n"]),
                  rng.uniform(0, 0.6, case["n"])], 1).astype(np.float32)
    m = case["m"]
    t, A, k = rng.uniform(0.65, 0.8, m), rng.uniform(-0.88, -0.82, m), rng.uniform(0.08, 0.5, m)
    sig = np.log((1.02 - k) * (0.95 - t) ** 1.3 * 0.06 * (1 + 0.3 * (A + 0.85)))
    return X, t.astype(np.float32), A.astype(np.float32), sig.astype(np.float32)


def _field(case, seed):
    """A droplet density with noise, on the device, and its discs."""
    nx, ny = case["nx"], case["ny"]
    rng = np.random.default_rng([int(seed), 3])
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    R, c = 0.25 * min(nx, ny) * rng.uniform(0.9, 1.1), rng.uniform(0.3, 0.7, 2)
    cx, cy = c[0] * nx, c[1] * ny
    dx = torch.arange(nx, dtype=torch.float64, device=dev)[None, :] - cx
    dy = torch.arange(ny, dtype=torch.float64, device=dev)[:, None] - cy
    dx, dy = dx - nx * torch.round(dx / nx), dy - ny * torch.round(dy / ny)
    g = torch.Generator(device=dev).manual_seed(int(seed))
    rho = 0.0093 + 0.1744 * (1.0 - torch.tanh(torch.sqrt(dx * dx + dy * dy) - R))
    rho = (rho * (1.0 + 0.01 * torch.rand((ny, nx), dtype=torch.float64, device=dev, generator=g))).contiguous()
    return rho, cx, cy, R / 2.0, R + 10.0


# ---- the user's program ----------------------------------------------------
def _eos(P, p):
    kind = {"cs": P.LBM_EOS_CS, "vdw": P.LBM_EOS_VDW, "pr": P.LBM_EOS_PR}[p["law"]]
    more = dict(omega=PR_OMEGA, Tc=TC_PR) if p["law"] == "pr" else {}
    return P.Eos(kind=kind, a=p["a"], b=p["b"], R=1.0, K=p["K"], T=p["T"], **more)


def _pinned(shape, dtype):
    t = torch.empty(shape, dtype=dtype)
    return (t.pin_memory() if torch.cuda.is_available() else t).numpy()


def prepare(case, seed):
    import paper_1412_7228_gb300 as P
    from paper_1412_7228_gb300 import lbm as B
    P.lib()
    kind = case["kind"]
    s = dict(case=case)
    if kind == "static":
        rho, cx, cy, r_in, r_out = _field(case, seed)
        s.update(call=B.lbm_field_pressure_jump_static, rho=rho, eos=_eos(P, _law("cs", 0.7)), at=(cx, cy, r_in, r_out))
        return s
    if kind == "train":
        X, Y, W = _samples(case, seed)
        s.update(mlp=B.Mlp(max_samples=max(case["n"], 64), seed=0), X=X, Y=Y,
                 p0=_flat(W[0], np.zeros(64), W[1], np.zeros(64), W[2], np.zeros(4)))
        s["mlp"].set_normalization(*_norm(X, Y))
        return s
    if kind == "pick":
        norm, p = _fitted(case, seed)
        X, t, A, sig = _picks(case, seed)
        s.update(mlp=B.Mlp(max_samples=max(case["n"], case["m"], 64), seed=0), X=X, t=t, A=A, sig=sig)
        s["mlp"].set_normalization(*norm)
        s["mlp"].set_params(p)
        return s

    lats = _lattices(case, seed)
    prec = P.LBM_FP64 if case.get("prec", "f64" if kind == "slabs" else "f32") == "f64" else P.LBM_FP32
    b = P.Batch([d["nx"] for d in lats], [d["ny"] for d in lats], prec)
    for i, d in enumerate(lats):
        b.set_params(i, _eos(P, d["p"]), d["A"], d["kappa"], G=-1.0, s=d["s"], rho_ref=d["ref"])
        if d.get("visc"):
            b.set_viscosity(i, *d["visc"])
        b.init_density(i, d["rho"], d.get("ux"), d.get("uy"))
    b.use_graphs(True)
    if kind == "whole":
        b.capture_graphs()
    elif kind != "probe":
        b.autotune(40)
    f32 = prec == P.LBM_FP32
    dtype = np.float32 if f32 else np.float64
    names = ("rho", "ux", "uy", "psi") if kind == "probe" or case.get("flow") else ("rho",)
    if kind in ("whole", "probe", "window", "sweep"):
        # results go to pinned memory, one array for all lattices
        total = sum(d["nx"] * d["ny"] for d in lats)
        s["out"] = {k: _pinned(total, torch.float32 if f32 else torch.float64) for k in names}
        s["views"], at = [], 0
        for d in lats:
            n = d["nx"] * d["ny"]
            s["views"].append({k: s["out"][k][at:at + n].reshape(d["ny"], d["nx"]) for k in names})
            at += n
    if kind == "whole":
        for k in ("rho", "ux", "uy"):
            if k in lats[0]:
                s[k] = _pinned((case["ny"], case["nx"]), torch.float32 if f32 else torch.float64)
                s[k][:] = lats[0][k]
    s.update(batch=b, names=names, dtype=dtype, size=[(d["nx"], d["ny"], d.get("R")) for d in lats])
    return s


KEYS = ("p_in", "p_out", "rho_in", "rho_out", "R_eq", "mass", "n_in", "n_out")


def _sample(b, i, L, R):
    """A droplet's Laplace sample with discs that follow its size."""
    m = b.measure(i, L / 2.0, L / 2.0, R / 2.0, R + 10.0)
    R = m["R_eq"]
    if not (R > 0 and math.isfinite(R)):   # it has evaporated
        return m
    return b.measure(i, L / 2.0, L / 2.0, R / 2.0, R + 10.0)


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "static":
        rho = s["rho"]
        return s["call"](rho.data_ptr(), case["nx"], case["ny"], s["eos"], *s["at"],
                         stream_ptr=torch.cuda.current_stream().cuda_stream)
    if kind == "train":
        m = s["mlp"]
        m.set_params(s["p0"])
        losses = m.train(s["X"], s["Y"], epochs=case["epochs"], batch=case["batch"], lr=3e-3, seed=1)
        return {"losses": losses, "params": m.get_params()}
    if kind == "pick":
        m = s["mlp"]
        return {"predicted": m.predict(s["X"]), "kappa": m.invert_kappa(s["t"], s["A"], s["sig"], 0.0, 0.6)}
    b = s["batch"]
    if kind == "run":
        b.step(case["steps"])
        return b.read_fields(which=("rho",), dtype=s["dtype"])
    if kind == "slabs":
        b.step(case["steps"])
        return [b.read_fields(i, which=("rho",))["rho"] for i in range(case["n"])]
    if kind == "whole":
        b.init_density(0, s["rho"], s.get("ux"), s.get("uy"))
        b.step(case["steps"])
        return b.read_fields(which=s["names"], out=s["views"][0], dtype=s["dtype"])
    if kind == "probe":
        out = dict(b.read_fields(which=s["names"], out=s["views"][0], dtype=s["dtype"]))
        nx, ny = case["nx"], case["ny"]
        m = b.measure(0, nx / 2.0, ny / 2.0, 0.1 * min(nx, ny), 0.2 * min(nx, ny) + 10.0)
        out.update({k: m[k] for k in KEYS})
        out.update({"stats_" + k: v for k, v in b.stats(0).items()})
        return out
    b.step(case["steps"])
    if kind == "window":
        got = [_sample(b, i, L, R) for i, (L, _, R) in enumerate(s["size"])]
    else:
        got = []
        for i, (L, _, R) in enumerate(s["size"]):
            status = b.status(i)
            got.append(dict(_sample(b, i, L, R), status=status, umax=b.stats(i)["umax"]))
    for i, view in enumerate(s["views"]):
        b.read_fields(i, which=("rho",), out=view, dtype=s["dtype"])
    out = {k: np.array([m[k] for m in got]) for k in got[0] if k in KEYS + ("umax", "status")}
    out["rho"] = s["out"]["rho"]
    return out


# ---- what one pass cannot do without ----------------------------------------
FLOPS = {"cs": 302.0, "vdw": 293.0, "pr": 298.0}   # of one lattice update (the FP64 oracle's operations)
L2_BYTES = 129e6


def work(case):
    kind = case["kind"]
    if kind == "static":
        n = case["nx"] * case["ny"]
        return {"bytes": 8.0 * n + 64, "flops": 25.0 * n}
    if kind == "train":
        n = case["n"]
        return {"bytes": 4.0 * (7 * n + 2 * 4676), "flops": 6.0 * 4676 * n * case["epochs"]}
    if kind == "pick":
        return {"bytes": 4.0 * (7 * case["n"] + 4 * case["m"] + 4676), "flops": 2.0 * 4676 * (case["n"] + 25 * case["m"])}
    if kind in ("window", "sweep"):
        sizes = [case["L"] ** 2] * case["n"] if kind == "window" else [d["nx"] * d["ny"] for d in _sizes(case)]
        law, e, fields, steps = "cs", 4, 1, case["steps"]
    else:
        sizes = [case["nx"] * case["ny"]] * case.get("n", 1)
        law = "vdw" if kind == "slabs" else case.get("law", "cs")
        e = 4 if case.get("prec", "f64") == "f32" else 8
        fields = 4 if kind == "probe" or case.get("flow") else 1
        steps = case.get("steps", 0)
    n = float(sum(sizes))
    # populations too large for L2 are read and written every step; smaller ones once a pass
    moves = steps if 9 * e * n > L2_BYTES else min(steps, 1)
    into = 0 if kind != "whole" else (3 if case["flow"] else 1)
    flops = FLOPS[law] * steps * n + (9 * n if kind != "probe" else 150 * n)
    return {"bytes": n * e * (18 * moves + (9 if not moves else 0) + fields + into), "flops": flops}


def _sizes(case):
    size = np.random.default_rng(case["sizes_seed"])
    sizes = [L for L in (128, 256, 512, 1024) if case["lo"] <= L <= case["hi"]]
    out = []
    for _ in range(case["n"]):
        L = int(size.choice(sizes)) if case["lo"] == 128 else int(round(case["lo"] * (case["hi"] / case["lo"]) ** size.random()))
        out.append(dict(nx=L, ny=L))
    return out


# ---- the same results in 64 bits, in plain torch ----------------------------
EX, EY = (0, 1, 0, -1, 0, 1, -1, -1, 1), (0, 0, 1, 0, -1, 1, 1, -1, -1)
M = np.array([[1, 1, 1, 1, 1, 1, 1, 1, 1], [-4, -1, -1, -1, -1, 2, 2, 2, 2], [4, -2, -2, -2, -2, 1, 1, 1, 1],
              [0, 1, 0, -1, 0, 1, -1, -1, 1], [0, -2, 0, 2, 0, 1, -1, -1, 1], [0, 0, 1, 0, -1, 1, 1, -1, -1],
              [0, 0, -2, 0, 2, 1, 1, -1, -1], [0, 1, -1, 1, -1, 0, 0, 0, 0], [0, 0, 0, 0, 0, 1, -1, 1, -1]], dtype=np.float64)
MINV = M.T / (M * M).sum(1)[None, :]


def _at(v, dx, dy):
    """v(x + d) at every x, periodic."""
    return torch.roll(v, shifts=(-dy, -dx), dims=(-2, -1)) if dx or dy else v


def _lin(c, f):
    out = None
    for k, v in zip(c, f):
        if k:
            t = v if k == 1 else -v if k == -1 else float(k) * v
            out = t if out is None else out + t
    return out


def _psi(d, rho):
    return torch.sqrt(2.0 / -1.0 * (_pressure(d["p"]["law"], d["p"], rho) - rho / 3.0))


def _force(d, psi):
    w = [0.0] + [1.0 / 3.0] * 4 + [1.0 / 12.0] * 4
    n = [_at(psi, EX[a], EY[a]) for a in range(9)]
    g = [sum(w[a] * e[a] * n[a] for a in range(1, 9) if e[a]) for e in (EX, EY)]
    h = [sum(w[a] * e[a] * n[a] * n[a] for a in range(1, 9) if e[a]) for e in (EX, EY)]
    return n, w, [0.5 * d["A"] * h[k] + (1.0 - d["A"]) * psi * g[k] for k in (0, 1)]   # G = -1


def _step(d, f):
    rho = sum(f)
    psi = _psi(d, rho)
    n, w, (Fx, Fy) = _force(d, psi)
    Q = []
    for e in ([x * x for x in EX], [y * y for y in EY], [x * y for x, y in zip(EX, EY)]):
        q1 = sum(w[a] * e[a] * (n[a] - psi) for a in range(1, 9) if e[a])
        q2 = sum(w[a] * e[a] * (n[a] * n[a] - psi * psi) for a in range(1, 9) if e[a])
        Q.append(-0.5 * d["kappa"] * ((1.0 - d["A"]) * psi * q1 + 0.5 * d["A"] * q2))
    m = [_lin(M[k], f) for k in range(9)]
    ux, uy = (m[3] + 0.5 * Fx) / rho, (m[5] + 0.5 * Fy) / rho
    u2, vF = ux * ux + uy * uy, ux * Fx + uy * Fy
    eq = [rho, rho * (3 * u2 - 2), rho * (1 - 3 * u2), rho * ux, -rho * ux, rho * uy, -rho * uy, rho * (ux * ux - uy * uy),
          rho * ux * uy]
    S = [0.0, 6 * vF, -6 * vF, Fx, -Fx, Fy, -Fy, 2 * (ux * Fx - uy * Fy), ux * Fy + uy * Fx]
    s = list(d["s"])
    if d.get("visc"):
        ng, nl, rg, rl = d["visc"]
        s[7] = s[8] = 1.0 / (3.0 * (ng + (nl - ng) * torch.clamp((rho - rg) / (rl - rg), 0.0, 1.0)) + 0.5)
    C = [0.0, 1.5 * s[1] * (Q[0] + Q[1]), 0.0, 0.0, 0.0, 0.0, 0.0, -s[7] * (Q[0] - Q[1]), -s[8] * Q[2]]
    m = [m[k] - s[k] * (m[k] - eq[k]) + (1.0 - 0.5 * s[k]) * S[k] + C[k] for k in range(9)]
    return [_at(_lin(MINV[a], m), -EX[a], -EY[a]) for a in range(9)]


def _start(d, dev):
    t = [4.0 / 9.0] + [1.0 / 9.0] * 4 + [1.0 / 36.0] * 4
    rho = torch.from_numpy(d["rho"]).to(dev).double()
    if "ux" not in d:
        return [t[a] * rho for a in range(9)]
    ux, uy = (torch.from_numpy(d[k]).to(dev).double() for k in ("ux", "uy"))
    u2 = ux * ux + uy * uy
    eu = [EX[a] * ux + EY[a] * uy for a in range(9)]
    return [t[a] * rho * (1 + 3 * eu[a] + 4.5 * eu[a] ** 2 - 1.5 * u2) for a in range(9)]


def _fields(d, f):
    rho = sum(f)
    psi = _psi(d, rho)
    _, _, (Fx, Fy) = _force(d, psi)
    return {"rho": rho, "ux": (_lin(M[3], f) + 0.5 * Fx) / rho, "uy": (_lin(M[5], f) + 0.5 * Fy) / rho, "psi": psi}


def _laplace(p, rho, cx, cy, r_in, r_out):
    ny, nx = rho.shape
    dx = torch.arange(nx, dtype=torch.float64, device=rho.device)[None, :] - cx
    dy = torch.arange(ny, dtype=torch.float64, device=rho.device)[:, None] - cy
    dx, dy = dx - nx * torch.round(dx / nx), dy - ny * torch.round(dy / ny)
    r = torch.sqrt(dx * dx + dy * dy)
    pr = _pressure(p["law"], p, rho)
    i, o = r <= r_in, r >= r_out
    zero = torch.zeros((), dtype=torch.float64, device=rho.device)
    mean = lambda v, k: float(torch.where(k, v, zero).sum() / k.sum())
    got = {"p_in": mean(pr, i), "p_out": mean(pr, o), "rho_in": mean(rho, i), "rho_out": mean(rho, o),
           "mass": float(rho.sum()), "n_in": float(i.sum()), "n_out": float(o.sum())}
    ex = got["mass"] - got["rho_out"] * nx * ny
    got["R_eq"] = math.sqrt(max(ex, 0.0) / (math.pi * (got["rho_in"] - got["rho_out"])))
    return got


def exact(case, seed):
    kind = case["kind"]
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    if kind == "static":
        rho, *at = _field(case, seed)
        return _laplace(_law("cs", 0.7), rho, *at)
    if kind == "train":
        return _exact_train(case, seed)
    if kind == "pick":
        return _exact_pick(case, seed)
    out = []
    for d in _lattices(case, seed):
        f = _start(d, dev)
        for _ in range(case.get("steps", 0)):
            f = _step(d, f)
        out.append((d, f))
    host = lambda v: v.cpu().numpy()
    if kind == "slabs":
        return [host(sum(f)) for _, f in out]
    d, f = out[0]
    if kind == "run":
        return {"rho": host(sum(f))}
    if kind in ("whole", "probe"):
        v = _fields(d, f)
        got = {k: host(x) for k, x in v.items() if k == "rho" or kind == "probe" or case["flow"]}
        if kind == "probe":
            nx, ny = case["nx"], case["ny"]
            got.update(_laplace(d["p"], v["rho"], nx / 2.0, ny / 2.0, 0.1 * min(nx, ny), 0.2 * min(nx, ny) + 10.0))
            sp2 = v["ux"] ** 2 + v["uy"] ** 2
            got.update(stats_mass=float(v["rho"].sum()), stats_mom_x=float((v["rho"] * v["ux"]).sum()),
                       stats_mom_y=float((v["rho"] * v["uy"]).sum()), stats_ke=float((0.5 * v["rho"] * sp2).sum()),
                       stats_umax=float(sp2.max().sqrt()))
        return got
    res = []
    for d, f in out:
        L, rho = d["nx"], sum(f)
        m = _laplace(d["p"], rho, L / 2.0, L / 2.0, d["R"] / 2.0, d["R"] + 10.0)
        m = _laplace(d["p"], rho, L / 2.0, L / 2.0, m["R_eq"] / 2.0, m["R_eq"] + 10.0)
        if kind == "sweep":
            v = _fields(d, f)
            m.update(status=0, umax=float((v["ux"] ** 2 + v["uy"] ** 2).max().sqrt()))
        res.append(m)
    got = {k: np.array([m[k] for m in res]) for k in res[0]}
    got["rho"] = torch.cat([sum(f).reshape(-1) for _, f in out]).cpu().numpy()
    return got


def _unpack(p):
    p = torch.from_numpy(p.astype(np.float64))
    o = np.cumsum([0, 192, 64, 4096, 64, 256, 4])
    return [p[a:b].reshape(s).clone() for a, b, s in zip(o[:-1], o[1:], ((64, 3), (64,), (64, 64), (64,), (4, 64), (4,)))]


def _net(w, x):
    return _gelu(_gelu(x @ w[0].T + w[1]) @ w[2].T + w[3]) @ w[4].T + w[5]


def _exact_train(case, seed):
    X, Y, W = _samples(case, seed)
    im, sd, om, os_ = (torch.from_numpy(v).double() for v in _norm(X, Y))
    x, y = (torch.from_numpy(X).double() - im) / sd, (torch.from_numpy(Y).double() - om) / os_
    w = [v.requires_grad_() for v in _unpack(_flat(W[0], np.zeros(64), W[1], np.zeros(64), W[2], np.zeros(4)))]
    mom, var = [torch.zeros_like(v) for v in w], [torch.zeros_like(v) for v in w]
    n, batch = case["n"], case["batch"]
    order, state, mask, t, losses = list(range(n)), 1, (1 << 64) - 1, 0, []
    b1, b2, lr, eps = 0.9, 0.999, 3e-3, 1e-8
    for _ in range(case["epochs"]):
        for i in range(n - 1, 0, -1):   # Fisher-Yates from a splitmix64 stream
            state = (state + 0x9E3779B97F4A7C15) & mask
            z = ((state ^ (state >> 30)) * 0xBF58476D1CE4E5B9) & mask
            z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & mask
            j = (z ^ (z >> 31)) % (i + 1)
            order[i], order[j] = order[j], order[i]
        got = []
        for first in range(0, n, batch):
            idx = torch.tensor(order[first:first + batch])
            loss = ((_net(w, x[idx]) - y[idx]) ** 2).mean()
            grads = torch.autograd.grad(loss, w)
            t += 1
            with torch.no_grad():
                for v, g, a, c in zip(w, grads, mom, var):
                    a.mul_(b1).add_(g, alpha=1 - b1)
                    c.mul_(b2).addcmul_(g, g, value=1 - b2)
                    v.sub_(lr * (a / (1 - b1 ** t)) / ((c / (1 - b2 ** t)).sqrt() + eps))
            got.append(float(loss.detach()))
        losses.append(sum(got) / len(got))
    return {"losses": np.array(losses), "params": torch.cat([v.detach().reshape(-1) for v in w]).numpy()}


def _exact_pick(case, seed):
    norm, p = _fitted(case, seed)
    im, sd, om, os_ = (torch.from_numpy(v).double() for v in norm)
    w = _unpack(p)
    X, t, A, sig = (torch.from_numpy(v).double() for v in _picks(case, seed))
    out = lambda x: _net(w, (x - im) / sd) * os_ + om
    lo, hi = torch.zeros_like(t), torch.full_like(t, float(np.float32(0.6)))
    f = lambda k: out(torch.stack([t, A, k], 1))[:, 0] - sig
    inside = (f(lo) >= 0) & (f(hi) <= 0)
    for _ in range(60):
        mid = 0.5 * (lo + hi)
        up = f(mid) >= 0
        lo, hi = torch.where(up, mid, lo), torch.where(up, hi, mid)
    k = torch.where(inside, 0.5 * (lo + hi), torch.full_like(t, float("nan")))
    return {"predicted": out(X).numpy(), "kappa": k.numpy()}
