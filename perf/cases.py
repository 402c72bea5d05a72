"""Timed cases of the library: what its users run, through its public entry points.

A case is a plain dict; "family" names the path:

  josephson   Eq. 1 ensembles on the persistent schedule (Ensemble.run_josephson), FP32
  noalloc     one Eq. 1 point through the allocation-free entry point, FP32
  fp64        one Eq. 1 point in double precision
  meanfield   Kuramoto, mean-field sums (Eq. 3): a replica per CTA or cluster, or over the whole grid
  pairwise    Kuramoto, direct all-pairs sums (Alg. 3)
  general     Kuramoto, matrix coupling: BF16 tensor-core GEMM or the FP32 form
  forward     surrogate network ensemble, inference
  train       surrogate network ensemble, Adam steps (forward, backward, update)

Sizes are the benchmark's and the tests' (inputs.py), shortened in steps where
a full run takes longer than the measurement needs, and ragged ones between.
"""
import math

import numpy as np
import torch

from paper_0903_3852_gb300 import inputs, sde

DEV = "cuda"
TWO_PI = 2.0 * math.pi
FIG2 = dict(gamma=0.9, a=4.2, omega=4.9, f=0.1, D=1e-3)  # the point of the paper's Fig. 2


# --------------------------------------------------------------------- cases

def listed():
    return [
        # The smallest call: a stroboscopic record of the Fig. 2 point, one
        # call per drive period (200 steps), 1024 paths; launches and latency.
        dict(name="josephson period", family="josephson", points=1, paths_lo=1024, paths_hi=1024, steps_lo=400,
             steps_hi=400, P=200, calls=2),
        # One parameter point at the size of the benchmark's plain run: 1024
        # paths for 100 drive periods, <<v>> read back.
        dict(name="josephson point", family="josephson", points=1, paths_lo=1024, paths_hi=1024, steps_lo=20000,
             steps_hi=20000, P=200, calls=1),
        # The benchmark's default: 512 points of f and D, ragged path and step
        # counts, 1.13 million paths; the largest call.
        dict(name="josephson sweep", family="josephson", points=512, paths_lo=256, paths_hi=8192, steps_lo=10000,
             steps_hi=100000, P=200, calls=1),
        # The double-precision check of FP32 trajectories over the first drive
        # periods, before chaos separates them: 2^16 paths, the Fig. 2 step.
        dict(name="josephson fp64", family="fp64", paths=65536, steps=400, P=100),
        # 64 replicas of 4096 oscillators with r(t) every 100 steps.
        dict(name="meanfield replicas", family="meanfield", osc=4096, replicas=64, steps=2000, K=2.0, D=0.05,
             dt=0.01, M=100, spread=1.0),
        # The ensemble of the paper's Fig. 4: one replica of 2^24 identical
        # oscillators.
        dict(name="meanfield fig4", family="meanfield", osc=2 ** 24, replicas=1, steps=40, K=4.0, D=1.0, dt=0.01,
             M=100, spread=0.0),
        # The all-pairs form at the benchmark's size.
        dict(name="pairwise replicas", family="pairwise", osc=4096, replicas=64, steps=10, K=2.0, D=0.05, dt=0.01,
             M=100, spread=1.0, euler=False),
        # A small ragged population, as in a first look at a model.
        dict(name="pairwise small", family="pairwise", osc=1000, replicas=3, steps=100, K=2.0, D=0.05, dt=0.01,
             M=100, spread=1.0, euler=False),
        # Matrix coupling at the benchmark's size, sub-steps in the GEMM's epilogue.
        dict(name="general bf16", family="general", osc=8192, replicas=256, steps=40, K=3.0, D=0.02, dt=0.005,
             M=100, f32=False, fused=True),
        # The FP32 form, for sizes and accuracies the BF16 form does not take.
        dict(name="general fp32", family="general", osc=3000, replicas=100, steps=20, K=3.0, D=0.02, dt=0.005,
             M=100, f32=True, fused=False),
        # Surrogate predictions for the benchmark's batch.
        dict(name="surrogate forward", family="forward", batch=100000, members=4, max_batch=131072),
        # Eight bootstrap batches of the surrogate's fit.
        dict(name="surrogate training", family="train", batch=1024, members=4, steps=8, max_batch=131072),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    family = rng.choice(["josephson", "josephson", "noalloc", "fp64", "meanfield", "meanfield", "pairwise",
                         "general", "general f32", "forward", "train"])
    if family == "josephson":
        points = _log_int(rng, 1, 512)
        lo = _log_int(rng, 100, 2000)
        steps = _log_int(rng, 200, 5000)
        return dict(family=family, points=points, paths_lo=lo, paths_hi=_log_int(rng, lo, 4 * lo), steps_lo=steps,
                    steps_hi=_log_int(rng, steps, 4 * steps), P=rng.choice([200, 200, 100, 90]),
                    calls=rng.choice([1, 1, 2]))
    if family == "noalloc":
        return dict(family=family, paths=_log_int(rng, 100, 500000), steps=_log_int(rng, 100, 2000),
                    P=rng.choice([200, 100]))
    if family == "fp64":
        return dict(family=family, paths=_log_int(rng, 100, 500000), steps=rng.randint(50, 400), P=100)
    if family == "meanfield":
        osc = _log_int(rng, 200, 2 ** 24)
        replicas = _log_int(rng, 1, max(1, min(64, 2 ** 20 // osc)))
        steps = max(20, min(_log_int(rng, 100, 2000), 2 ** 30 // (osc * replicas)))
        return dict(family=family, osc=osc, replicas=replicas, steps=steps, K=rng.choice([2.0, 4.0]),
                    D=rng.choice([0.05, 1.0]), dt=0.01, M=rng.choice([100, 25]), spread=rng.choice([1.0, 0.0]))
    if family == "pairwise":
        osc = _log_int(rng, 100, 6000)
        replicas = _log_int(rng, 1, 64)
        steps = max(5, min(_log_int(rng, 10, 200), int(4e10 / (osc * osc * replicas))))
        return dict(family=family, osc=osc, replicas=replicas, steps=steps, K=2.0, D=0.05, dt=0.01,
                    M=rng.choice([100, 25]), spread=1.0, euler=rng.choice([False, False, True]))
    if family == "general":
        return dict(family=family, osc=128 * _log_int(rng, 2, 64), replicas=64 * rng.randint(1, 4),
                    steps=_log_int(rng, 10, 40), K=3.0, D=0.02, dt=0.005, M=100, f32=False,
                    fused=rng.choice([True, True, False]))
    if family == "general f32":
        return dict(family="general", osc=8 * _log_int(rng, 16, 500), replicas=_log_int(rng, 1, 128),
                    steps=_log_int(rng, 10, 40), K=3.0, D=0.02, dt=0.005, M=100, f32=True, fused=False)
    if family == "forward":
        return dict(family=family, batch=_log_int(rng, 1, 131072), members=rng.choice([4, 4, 2]), max_batch=131072)
    return dict(family=family, batch=_log_int(rng, 200, 2048), members=rng.choice([4, 4, 2]),
                steps=rng.randint(1, 8), max_batch=131072)


# -------------------------------------------------------------------- inputs

def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _uniform(g, shape, lo, hi):
    return torch.rand(shape, generator=g, device=DEV) * (hi - lo) + lo


def _josephson_table(case):
    """Parameter points, paths and steps of a case: the same for every seed."""
    n = case["points"]
    if n == 1:
        return [FIG2], np.array([case["paths_lo"]]), np.array([case["steps_lo"]])
    rng = np.random.default_rng(1)
    paths = inputs.log_uniform_int(rng, case["paths_lo"], case["paths_hi"], n)
    steps = inputs.log_uniform_int(rng, case["steps_lo"], case["steps_hi"], n)
    return inputs.sweep_grid(n), paths, steps


def _paths_of(case):
    if case["family"] == "josephson":
        return int(_josephson_table(case)[1].sum())
    return case["paths"]


def _josephson_inputs(case, seed):
    """x0 ~ U[0, 1), v0 ~ U[-2, 2)."""
    g, n = _gen(seed), _paths_of(case)
    dt = torch.float64 if case["family"] == "fp64" else torch.float32
    return _uniform(g, n, 0.0, 1.0).to(dt), _uniform(g, n, -2.0, 2.0).to(dt)


def _kuramoto_inputs(case, seed):
    """phi0 ~ U[0, 2 pi), omega ~ spread N(0, 1); matrix coupling as in inputs.kuramoto_general."""
    g = _gen(seed)
    R, N = case["replicas"], case["osc"]
    phi = _uniform(g, (R, N), 0.0, TWO_PI).clamp_(max=6.2831845)
    omega = torch.randn((R, N), generator=g, device=DEV) * case.get("spread", 1.0)
    Kmat = None
    if case["family"] == "general":
        Kmat = (_uniform(g, (N, N), -1.0, 1.0) * 0.5 + 1.0) * (case["K"] / N)
    return phi, omega, Kmat


H, LAYERS, N_IN = 256, 3, 5  # the surrogate's network: 5 -> 256 x 3 -> 1


def _mlp_inputs(case, seed):
    """Weights U(+-1/sqrt(fan_in)), features U[-1, 1], labels a smooth function of them."""
    g = _gen(seed)
    fan = [N_IN] + [H] * LAYERS
    out = [H] * LAYERS + [1]
    members = []
    for _ in range(case["members"]):
        members.append([(_uniform(g, (o, i), -1.0, 1.0) / math.sqrt(i), _uniform(g, o, -1.0, 1.0) / math.sqrt(i))
                        for i, o in zip(fan, out)])
    if case["family"] == "forward":
        return members, _uniform(g, (case["batch"], N_IN), -1.0, 1.0), None
    X = _uniform(g, (case["steps"], case["members"], case["batch"], N_IN), -1.0, 1.0)
    y = torch.sin(3.0 * X[..., 0]) * X[..., 1] + 0.5 * X[..., 2]
    return members, X, y.contiguous()


def _flat(layers):
    return torch.cat([t.reshape(-1) for w, b in layers for t in (w, b)]).contiguous()


def _rows(case):
    return -(-case["steps"] // case["M"]) + 1


MODELS = {"meanfield": sde.SDE_KURAMOTO_MEANFIELD, "pairwise": sde.SDE_KURAMOTO_PAIRWISE}


# ----------------------------------------------------------- prepare and run

def prepare(case, seed):
    f = case["family"]
    s = dict(case=case, seed=seed)
    if f == "josephson":
        points, paths, steps = _josephson_table(case)
        s["x0"], s["v0"] = _josephson_inputs(case, seed)
        s["ens"] = sde.Ensemble.josephson(points, paths, steps, seed, steps_per_period=case["P"])
        s["n_end"] = int(steps.max())
    elif f in ("noalloc", "fp64"):
        s["x0"], s["v0"] = _josephson_inputs(case, seed)
    elif f in ("forward", "train"):
        members, s["X"], s["y"] = _mlp_inputs(case, seed)
        s["mlp"] = sde.Mlp(members=case["members"], max_batch=case["max_batch"])
        for m, layers in enumerate(members):
            s["mlp"].set_params(m, _flat(layers))
        s["loss"] = torch.empty((case.get("steps", 1), case["members"]), device=DEV)
        return s
    else:
        s["phi0"], s["omega"], Kmat = _kuramoto_inputs(case, seed)
        flags = 0
        if f == "general":
            model = sde.SDE_KURAMOTO_GENERAL_FP32 if case["f32"] else sde.SDE_KURAMOTO_GENERAL
            flags = sde.SDE_FLAG_FUSED if case["fused"] else 0
        else:
            model = MODELS[f]
            flags = sde.SDE_FLAG_EULER if case.get("euler") else 0
        s["ens"] = sde.Ensemble.kuramoto(model, case["osc"], case["replicas"], case["K"], case["D"], case["dt"], seed,
                                         sample_every=case["M"], flags=flags)
        if Kmat is not None:
            s["ens"].set_coupling(Kmat)
            torch.cuda.synchronize()
        s["phi"] = torch.empty_like(s["phi0"])
        s["r"] = torch.empty((_rows(case), case["replicas"]), dtype=torch.float64, device=DEV)
        s["one"] = torch.ones_like(s["phi0"])
        return s
    n = s["x0"].numel()
    s["x"], s["v"] = torch.empty_like(s["x0"]), torch.empty_like(s["v0"])
    s["w"] = torch.empty(n, dtype=torch.int32, device=DEV)
    s["vsum"] = torch.empty(n, dtype=torch.float64, device=DEV)
    s["obs"] = torch.empty(5, dtype=torch.float64, device=DEV)
    return s


def run(s):
    case = s["case"]
    f = case["family"]
    if f == "josephson":
        ens, calls, n_end = s["ens"], case["calls"], s["n_end"]
        x, v, w, vsum = s["x"], s["v"], s["w"], s["vsum"]
        n0 = 0
        for c in range(calls):  # successive windows of one run, the state kept in x, v, w, vsum
            n1 = n_end * (c + 1) // calls
            if c == 0:
                ens.run_josephson(n0, n1, s["x0"], s["v0"], x, v, w, vsum)
            else:
                ens.run_josephson(n0, n1, x, v, x, v, w, vsum, w_in=w, vsum_in=vsum)
            n0 = n1
        obs = ens.observables()  # <<v>> and its standard error per point: the result of the sweep
        return dict(x=x, v=v, w=w, vsum=vsum, mean=obs["mean"], se=obs["se"])
    if f == "noalloc":
        sde.josephson_run_noalloc(FIG2, case["P"], case["paths"], case["steps"], s["seed"], 0, case["steps"], s["x0"],
                                  s["v0"], s["x"], s["v"], s["w"], s["vsum"], s["obs"])
        return dict(x=s["x"], v=s["v"], w=s["w"], vsum=s["vsum"], obs=s["obs"])
    if f == "fp64":
        sde.josephson_run_fp64(FIG2, case["P"], case["steps"], s["seed"], 0, case["steps"], s["x0"], s["v0"], s["x"],
                               s["v"], vsum_out=s["vsum"])
        return dict(x=s["x"], v=s["v"], vsum=s["vsum"])
    if f == "forward":
        mean, spread = s["mlp"].forward(s["X"])
        return dict(mean=mean, spread=spread)
    if f == "train":
        for k in range(case["steps"]):
            s["mlp"].train_step_members(s["X"][k], s["y"][k], s["loss"][k])
        return dict(loss=s["loss"], params=[s["mlp"].get_params(m) for m in range(case["members"])])
    s["ens"].run_kuramoto(0, case["steps"], s["phi0"], s["phi"], s["omega"], s["r"])
    # A phase is a point on a circle: the complex field e^{i phi}, which local
    # order parameters are taken from, has no jump at 2 pi.  r(t) is stored in
    # FP64 but formed from 32-bit phases and FP32 sines: a program plots it in FP32.
    return dict(z=torch.polar(s["one"], s["phi"]), r=s["r"].float())


# ---------------------------------------------------------------------- work

def work(case):
    """Bytes: inputs read once, outputs written once.  FLOP: per path-step of
    Eq. 1 the 52 FP32 (79 FP64, Table 1 of the paper) operations of one SRK2
    step with its Gaussian, per oscillator-step of Eq. 3 66, per pair term 6
    (the paper's counts), the multiply-adds of a GEMM."""
    f = case["family"]
    if f == "josephson":
        _, paths, steps = _josephson_table(case)
        return dict(bytes=28.0 * float(paths.sum()), flops=52.0 * float((paths * steps).sum()))
    if f == "noalloc":
        return dict(bytes=28.0 * case["paths"], flops=52.0 * case["paths"] * case["steps"])
    if f == "fp64":
        return dict(bytes=40.0 * case["paths"], flops=79.0 * case["paths"] * case["steps"])
    if f in ("forward", "train"):
        per_point = 2.0 * (N_IN * H + (LAYERS - 1) * H * H + H)
        P = N_IN * H + H + (LAYERS - 1) * (H * H + H) + H + 1
        if f == "forward":
            return dict(bytes=4.0 * (case["batch"] * (N_IN + 2) + case["members"] * P),
                        flops=per_point * case["batch"] * case["members"])
        n = case["steps"] * case["members"]
        # parameters and both Adam moments are read and written in each step
        return dict(bytes=4.0 * n * (case["batch"] * (N_IN + 1) + 6 * P), flops=3.0 * n * case["batch"] * per_point)
    N, R, steps = float(case["osc"]), float(case["replicas"]), float(case["steps"])
    if f == "meanfield":
        return dict(bytes=12.0 * N * R, flops=66.0 * N * R * steps)
    if f == "pairwise":
        return dict(bytes=12.0 * N * R, flops=(6.0 if case["euler"] else 12.0) * N * N * R * steps)
    return dict(bytes=(4.0 if case["f32"] else 2.0) * N * N + 12.0 * N * R, flops=2.0 * 2.0 * N * N * 2.0 * R * steps)


# ----------------------------------------------------------- 64-bit reference

M32 = 0xFFFFFFFF


def _mul32(a, m):
    """(high, low) words of a * m, a an int64 tensor of 32-bit words."""
    al, ah, ml, mh = a & 0xFFFF, a >> 16, m & 0xFFFF, m >> 16
    ll, lh, hl = al * ml, al * mh, ah * ml
    mid = (ll >> 16) + (lh & 0xFFFF) + (hl & 0xFFFF)
    return ah * mh + (lh >> 16) + (hl >> 16) + (mid >> 16), ((mid & 0xFFFF) << 16) | (ll & 0xFFFF)


def _philox(c0, c1, c2, c3, seed):
    """Philox4x32-10 (Salmon et al., SC'11) of int64 tensors of 32-bit words."""
    k0, k1 = seed & M32, (seed >> 32) & M32
    for _ in range(10):
        h0, l0 = _mul32(c0, 0xD2511F53)
        h1, l1 = _mul32(c2, 0xCD9E8D57)
        c0, c1, c2, c3 = h1 ^ c1 ^ k0, l1, h0 ^ c3 ^ k1, l0
        k0, k1 = (k0 + 0x9E3779B9) & M32, (k1 + 0xBB67AE85) & M32
    return c0, c1, c2, c3


def _gauss4(block, index, group, tag, seed):
    """The four Gaussians of Philox block `block` for every (index, group)."""
    z = torch.zeros_like(index)
    w = _philox(z + block, index, group, z + tag, seed)
    u = [((a >> 8) + 1).double() * 2.0 ** -24 for a in w]
    out = []
    for a, b in ((u[0], u[1]), (u[2], u[3])):
        rho = torch.sqrt(-2.0 * torch.log(a))
        out += [rho * torch.cos(TWO_PI * b), rho * torch.sin(TWO_PI * b)]
    return out


def _exact_josephson(case, seed):
    if case["family"] == "josephson":
        points, paths, steps = _josephson_table(case)
    else:
        points, paths, steps = [FIG2], np.array([case["paths"]]), np.array([case["steps"]])
    P, last = case["P"], int(steps.max())
    # Trajectories at these parameters separate by a factor of ~25 per drive
    # period: over more than a few periods no path has a value to compare with.
    if last > 4 * P:
        return None
    group = np.repeat(np.arange(len(points)), paths)
    index = np.concatenate([np.arange(n) for n in paths])

    def column(values):
        return torch.from_numpy(np.asarray(values, dtype=np.float64)[group]).to(DEV)

    gamma, a, omega, fb, D = (column([p[k] for p in points]) for k in ("gamma", "a", "omega", "f", "D"))
    S = column(steps)
    gi, ii = torch.from_numpy(group).to(DEV), torch.from_numpy(index).to(DEV)
    dt = TWO_PI / (omega * P)
    s = torch.sqrt(2.0 * gamma * D * dt)
    start = S - torch.floor(S / 2)
    x, v = (t.double() for t in _josephson_inputs(case, seed))
    vsum = torch.zeros_like(x)

    def force(x, v, n):
        return -gamma * v - TWO_PI * torch.cos(TWO_PI * x) + a * math.cos(TWO_PI * (n % P) / P) + fb

    for n in range(last):
        if n % 4 == 0:
            z = _gauss4(n // 4, ii, gi, 1, seed)
        noise = s * z[n % 4]
        on = n < S
        F1 = force(x, v, n)
        vt = v + dt * F1 + noise
        F2 = force(x + dt * v, vt, n + 1)
        x1, v1 = x + 0.5 * dt * (v + vt), v + 0.5 * dt * (F1 + F2) + noise
        x, v = torch.where(on, x1, x), torch.where(on, v1, v)
        vsum = torch.where(on & (n + 1 > start), vsum + v, vsum)
    if case["family"] == "fp64":
        return dict(x=x, v=v, vsum=vsum)
    frac = x - torch.floor(x)
    if case["family"] == "noalloc":
        return dict(x=frac, v=v, w=None, vsum=vsum, obs=None)
    avg = torch.split(vsum / torch.floor(S / 2), [int(n) for n in paths])
    return dict(x=frac, v=v, w=None, vsum=vsum, mean=torch.stack([t.mean() for t in avg]), se=None)


def _exact_kuramoto(case, seed):
    phi, omega, Kmat = _kuramoto_inputs(case, seed)
    R, N = phi.shape
    f, dt = case["family"], case["dt"]
    if f == "general" and N * N * R * case["steps"] > 8e11:
        return None
    x, omega = phi.double(), omega.double()
    if Kmat is not None:
        Kt = Kmat.double().t()
    index = torch.arange(N, device=DEV).repeat(R, 1)
    group = torch.arange(R, device=DEV)[:, None].expand(R, N).contiguous()
    amp = math.sqrt(2.0 * case["D"] * dt)
    r = []

    def drift(x):
        s, c = torch.sin(x), torch.cos(x)
        if Kmat is None:  # sum_j sin(x_j - x_i) by Eq. 3
            k = case["K"] / N
            return omega + k * (c * s.sum(1, keepdim=True) - s * c.sum(1, keepdim=True))
        return omega + c * (s @ Kt) - s * (c @ Kt)

    for n in range(case["steps"]):
        if n % case["M"] == 0:
            r.append(torch.polar(torch.ones_like(x), x).mean(1).abs())
        if n % 4 == 0:
            z = _gauss4(n // 4, index, group, 2, seed)
        noise = amp * z[n % 4]
        F1 = drift(x)
        if case.get("euler"):
            x = x + dt * F1 + noise
        else:
            x = x + 0.5 * dt * (F1 + drift(x + dt * F1 + noise)) + noise
    z = torch.polar(torch.ones_like(x), x)
    r.append(z.mean(1).abs())
    return dict(z=z, r=torch.stack(r))


def _exact_mlp(case, seed):
    members, X, y = _mlp_inputs(case, seed)
    members = [[(w.double(), b.double()) for w, b in m] for m in members]

    def net(layers, h):
        for k, (w, b) in enumerate(layers):
            h = h @ w.t() + b
            if k < LAYERS:
                h = h * torch.sigmoid(h)
        return h[:, 0]

    if case["family"] == "forward":
        out = torch.stack([net(m, X.double()) for m in members])
        return dict(mean=out.mean(0), spread=out.std(0))
    params, losses = [], torch.zeros(case["steps"], case["members"], dtype=torch.float64, device=DEV)
    for q, layers in enumerate(members):
        leaves = [t.clone().requires_grad_() for w, b in layers for t in (w, b)]
        opt = torch.optim.Adam(leaves, lr=1e-3, betas=(0.9, 0.999), eps=1e-8)
        for k in range(case["steps"]):
            loss = ((net(list(zip(leaves[::2], leaves[1::2])), X[k, q].double()) - y[k, q].double()) ** 2).mean()
            opt.zero_grad()
            loss.backward()
            opt.step()
            losses[k, q] = loss.detach()
        params.append(torch.cat([t.detach().reshape(-1) for t in leaves]))
    return dict(loss=losses, params=params)


def exact(case, seed):
    f = case["family"]
    if f in ("josephson", "noalloc", "fp64"):
        return _exact_josephson(case, seed)
    if f in ("forward", "train"):
        return _exact_mlp(case, seed)
    return _exact_kuramoto(case, seed)
