"""The work that users of this library have it do, as cases to be timed.

Four kinds of program, each through the Python binding of the C ABI:

* ``advance`` -- one lattice that exists already is advanced by ``steps`` time
  steps and its density and velocity are read back (the loop of every
  simulation: run, look, run on);
* ``simulate`` -- the whole call: a density field goes in, ``steps`` steps are
  run, density and velocity come back;
* ``sweep`` -- many flat-interface lattices are started from their coexistence
  densities and advanced together, window by window (parameter sweeps, and the
  narrow slabs that the warm-start network is trained on);
* ``mlp_train`` / ``mlp_predict`` -- training and evaluation of that network.

Sizes are those of the repository's configurations, tests and benchmark (the
64^2 slab, the 200^2 and 256^2 droplets, the 1024^2 and 8192^2 spinodal
decompositions, sweep slabs of 32-512 x 128-512, narrow slabs of 32 columns, the
4 -> 64 -> 64 -> 3 network) or generic ones beside them.
"""
import math

import numpy as np
import torch

from paper_1204_4098_gb300 import inputs, lbm, warmstart

SCHEMES = {"sc": lbm.SC, "edm": lbm.EDM, "improved": lbm.IMPROVED, "noforce": lbm.NOFORCE,
           "edm_mod": lbm.EDM_MOD, "ladd": lbm.LADD, "mrt": lbm.MRT}
PRECISIONS = {"fp32": lbm.FP32, "fp64": lbm.FP64, "bf16": lbm.BF16DEV, "fp16": lbm.FP16DEV}
MRT_RATES = (0.8, 1.1, 1.3)  # energy, energy square, energy flux


def _lattice(name, kind, nx, ny, steps, scheme, tau, sigma=0.0, T=0.85, precision="fp32",
             field="spinodal"):
    return dict(name=name, kind=kind, nx=nx, ny=ny, steps=steps, scheme=scheme, tau=tau,
                sigma=sigma, T=T, precision=precision, field=field)


def listed():
    return [
        # the network asked for the 256 held-out sweep points: the smallest call
        dict(name="mlp_predict_256", kind="mlp_predict", n=256),
        # the flat-interface slab every forcing scheme is checked on: a lattice
        # whose steps are shorter than a launch
        _lattice("slab_64", "advance", 64, 64, 500, "sc", 1.0, T=0.8, field="slab"),
        # the droplet of the stability figures, modified exact difference method
        _lattice("droplet_200", "advance", 200, 200, 500, "edm_mod", 0.7, T=0.8,
                 field="droplet"),
        # spinodal decomposition at the size the golden run is stored for
        _lattice("spinodal_1024", "advance", 1024, 1024, 100, "improved", 0.8, 0.1),
        # a lattice whose sides are no multiple of anything
        _lattice("ragged_1501x997", "advance", 1501, 997, 60, "edm", 0.9, T=0.88),
        # the multiple-relaxation-time form of the improved scheme
        _lattice("mrt_2048", "advance", 2048, 2048, 60, "mrt", 0.8, 0.1),
        # 16-bit deviation storage, chosen to fit larger lattices
        _lattice("bf16_4096", "advance", 4096, 4096, 60, "improved", 0.8, 0.1,
                 precision="bf16"),
        # the double-precision run a user checks the others against
        _lattice("fp64_512", "advance", 512, 512, 50, "sc", 0.8, precision="fp64",
                 T=0.9, field="droplet"),
        # the benchmark's lattice, from the host's density to the host's moments
        _lattice("simulate_8192", "simulate", 8192, 8192, 200, "improved", 0.8, 0.1),
        # a parameter sweep over mixed sizes, temperatures and schemes (some
        # points are unstable and leave at the first check)
        dict(name="sweep_48", kind="sweep", count=48, nx_lo=32, nx_hi=512, sizes=4, windows=6),
        # the narrow slabs that the network's training data come from
        dict(name="narrow_slabs_96", kind="sweep", count=96, nx_lo=32, nx_hi=32, sizes=40,
             windows=8),
        # training on the converged runs of a data set of the usual size
        dict(name="mlp_train_2048", kind="mlp_train", n=2048, epochs=10, batch=128),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["advance"] * 5 + ["simulate", "sweep", "mlp_train", "mlp_predict"])
    if kind == "mlp_predict":
        return dict(kind=kind, n=_log_int(rng, 1, 20000))
    if kind == "mlp_train":
        return dict(kind=kind, n=_log_int(rng, 100, 4000), epochs=rng.randint(3, 10),
                    batch=rng.choice([32, 64, 100, 128]))
    if kind == "sweep":
        narrow = rng.random() < 0.4
        return dict(kind=kind, count=rng.randint(6, 96 if narrow else 40), nx_lo=32,
                    nx_hi=32 if narrow else 512, sizes=rng.randint(0, 10 ** 6),
                    windows=rng.randint(2, 4))
    precision = rng.choice(["fp32"] * 4 + ["bf16", "fp16", "fp64"])
    hi = 1000 if precision == "fp64" else 5000
    nx, ny = _log_int(rng, 30, hi), _log_int(rng, 30, hi)
    steps = _log_int(rng, 4, 300)
    most = 1.2e7 if precision == "fp64" else 1.5e9
    steps = max(1, min(steps, int(most / (nx * ny))))
    scheme = rng.choice(["sc", "edm", "improved", "improved", "edm_mod", "mrt", "noforce"])
    case = _lattice("", kind, nx, ny, steps, scheme, round(rng.uniform(0.7, 1.3), 3),
                    round(rng.uniform(0.05, 0.15), 3), T=round(rng.uniform(0.87, 0.95), 3),
                    precision=precision, field=rng.choice(["slab", "droplet", "spinodal"]))
    del case["name"]
    return case


# ---- inputs ----------------------------------------------------------------


def _cs_z(e):
    """(g, g', g'') of g(eta) = eta (1 + eta + eta^2 - eta^3) / (1 - eta)^3: the
    Carnahan-Starling pressure is T g(rho) - rho^2 for a = 1, b = 4, R = 1."""
    n = 1 + 4 * e + 4 * e ** 2 - 4 * e ** 3 + e ** 4
    dn = 4 + 8 * e - 12 * e ** 2 + 4 * e ** 3
    return (e * (1 + e + e * e - e ** 3) / (1 - e) ** 3, n / (1 - e) ** 4,
            (dn * (1 - e) + 4 * n) / (1 - e) ** 5)


def _bisect(f, lo, hi):
    flo = f(lo)
    for _ in range(200):
        mid = 0.5 * (lo + hi)
        if (f(mid) > 0) == (flo > 0):
            lo = mid
        else:
            hi = mid
    return 0.5 * (lo + hi)


def _critical():
    """(rho, T) of the critical point: both derivatives of the pressure vanish."""
    e = _bisect(lambda x: _cs_z(x)[1] - x * _cs_z(x)[2], 0.05, 0.3)
    return e, 2.0 / _cs_z(e)[2]


def _coexistence(t):
    """(rho_g, rho_l) at t = T / Tc: equal pressure and chemical potential."""
    rc, Tc = _critical()
    T = t * Tc
    p = lambda e: T * _cs_z(e)[0] - e * e  # noqa: E731
    dp = lambda e: T * _cs_z(e)[1] - 2 * e  # noqa: E731
    mu = lambda e: T * (math.log(e) + (8 * e - 9 * e * e + 3 * e ** 3) / (1 - e) ** 3) - 2 * e  # noqa: E731
    s_g, s_l = _bisect(dp, 1e-9, rc), _bisect(dp, rc, 0.9)  # spinodal densities

    def at(press):
        return (_bisect(lambda e: p(e) - press, 1e-12, s_g),
                _bisect(lambda e: p(e) - press, s_l, 0.95))

    def gap(press):
        g, l = at(press)
        return mu(g) - mu(l)

    return at(_bisect(gap, max(p(s_l), 1e-12), p(s_g)))


def _field(case, seed):
    """Density field [ny][nx] in FP64: a slab, a droplet or the middle of the
    spinodal region, with a seeded multiplicative noise on every cell."""
    nx, ny = case["nx"], case["ny"]
    g, l = _coexistence(case["T"])
    if case["field"] == "slab":
        rho, amp = inputs.slab_tanh(nx, ny, g, l, W=5.0), 1e-3
    elif case["field"] == "droplet":
        rho, amp = inputs.droplet(nx, ny, g, l, 0.15 * min(nx, ny) + 5.0, W=5.0), 1e-3
    else:
        rho, amp = np.full((ny, nx), 0.5 * (g + l)), 1e-2
    gen = torch.Generator(device="cuda").manual_seed(seed)
    noise = torch.rand((ny, nx), dtype=torch.float64, device="cuda", generator=gen)
    noise.mul_(2.0 * amp).add_(1.0 - amp)
    return noise.mul_(torch.from_numpy(rho).cuda()).cpu().numpy()


def _flow(case, seed):
    """Initial velocity (ux, uy): slabs and droplets sit in a slow shear flow in
    both directions, a spinodal decomposition starts at u = 0 (None, None)."""
    if case["field"] == "spinodal":
        return None, None
    nx, ny = case["nx"], case["ny"]
    u, v = np.random.default_rng(seed).uniform(0.005, 0.01, 2)
    ux = u * np.sin(2.0 * np.pi * np.arange(ny) / ny)[:, None]
    uy = v * np.sin(2.0 * np.pi * np.arange(nx) / nx)[None, :]
    return (np.ascontiguousarray(np.broadcast_to(a, (ny, nx))) for a in (ux, uy))


def _instances(case, seed):
    """The sweep's draws, above the temperature below which nearly every point
    is unstable; the lattice sizes belong to the case."""
    sized = inputs.sweep_instances(case["count"], seed=case["sizes"],
                                   nx_range=(case["nx_lo"], case["nx_hi"]))
    drawn = inputs.sweep_instances(case["count"], seed=seed, t_range=(0.7, 0.95))
    return [dict(d, nx=s["nx"], ny=s["ny"]) for s, d in zip(sized, drawn)]


def _samples(n, seed):
    """Network inputs over the sweep's ranges and smooth standardised targets."""
    inst = inputs.sweep_instances(n, seed=seed)
    X = warmstart.features(inst)
    x = X.astype(np.float64)
    Y = np.stack([np.tanh(x[:, 0] + 0.5 * x[:, 1]), x[:, 0] * x[:, 2] - 0.3 * x[:, 3],
                  np.sin(2.0 * x[:, 0]) + 0.2 * x[:, 1] * x[:, 3]], 1)
    return X, ((Y - Y.mean(0)) / (Y.std(0) + 1e-12)).astype(np.float32)


def _order(case, seed):
    rng = np.random.default_rng(seed)
    return np.stack([rng.permutation(case["n"]) for _ in range(case["epochs"])]).astype(np.int32)


# ---- the calls ---------------------------------------------------------------


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("advance", "simulate"):
        nx, ny = case["nx"], case["ny"]
        rho = lbm.host_array((ny, nx))  # page-locked, as the copies want it
        rho[...] = _field(case, seed)
        ux, uy = _flow(case, seed)
        lat = lbm.Lattice(nx, ny, case["T"], precision=PRECISIONS[case["precision"]])
        if case["scheme"] == "mrt":
            lat.set_mrt_rates(*MRT_RATES)
        out = tuple(lbm.host_array((ny, nx)) for _ in range(3))
        if kind == "advance":
            lat.init_density(rho, ux, uy)
        return dict(case=case, lat=lat, rho=rho, ux=ux, uy=uy, out=out)
    if kind == "sweep":
        inst = _instances(case, seed)
        dens = np.array([_coexistence(d["T_over_Tc"]) for d in inst])
        return dict(case=case, batch=lbm.Batch(inst), rho_g=dens[:, 0].copy(),
                    rho_l=dens[:, 1].copy(), width=np.zeros(len(inst)))
    X, Y = _samples(case["n"], seed)
    state = dict(case=case, X=X, Y=Y, params=warmstart.glorot_params(seed))
    if kind == "mlp_train":
        state.update(mlp=lbm.MLP(), order=_order(case, seed))
    else:
        state.update(mlp=lbm.MLP(state["params"]))
    return state


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind in ("advance", "simulate"):
        lat = state["lat"]
        if kind == "simulate":
            lat.init_density(state["rho"], state["ux"], state["uy"])
        lat.step(case["steps"], SCHEMES[case["scheme"]], case["tau"], case["sigma"])
        rho, vx, vy = lat.observe(state["out"])
        return dict(rho=rho, vx=vx, vy=vy)
    if kind == "sweep":
        batch = state["batch"]
        batch.init_slabs(state["rho_g"], state["rho_l"], state["width"])
        left = batch.run(case["windows"])
        res = batch.results()
        ok = np.array([r["status"] != lbm.RUN_DIVERGED for r in res])  # else unspecified
        out = {k: np.where(ok, [r[k] for r in res], 0.0)
               for k in ("rho_g", "rho_l", "width", "mass")}
        out.update(left=left, steps=np.array([r["steps"] for r in res]),
                   status=np.array([r["status"] for r in res]))
        # the profiles of the first points, to look at
        out["density"] = [batch.density(i) if ok[i] else np.zeros(
            (batch.instances[i]["ny"], batch.instances[i]["nx"])) for i in range(6)]
        return out
    mlp = state["mlp"]
    if kind == "mlp_predict":
        return mlp.predict(state["X"])
    mlp.set_params(state["params"])
    loss = mlp.train(state["X"], state["Y"], state["order"], case["batch"], 2e-3)
    return dict(params=mlp.params(), loss=np.float32(loss))


def work(case):
    """One read of what goes in and one write of what comes out, and the
    arithmetic: about 250 operations per cell and step, 2 per weight and sample."""
    kind = case["kind"]
    if kind in ("advance", "simulate"):
        cells = case["nx"] * case["ny"]
        state = {"fp32": 36, "fp64": 72, "bf16": 22, "fp16": 22}[case["precision"]]
        given = state
        if kind == "simulate":
            given = 8 if case["field"] == "spinodal" else 24
        return dict(bytes=cells * (given + state + 24), flops=250.0 * cells * case["steps"])
    if kind == "sweep":
        cells = sum(d["nx"] * d["ny"] for d in _instances(case, 0))
        return dict(bytes=cells * 36, flops=250.0 * cells * 1000 * case["windows"])
    if kind == "mlp_predict":
        return dict(bytes=4 * (4675 + 7 * case["n"]), flops=2.0 * 4544 * case["n"])
    return dict(bytes=4 * (7 * case["n"] + case["n"] * case["epochs"] + 2 * 4675),
                flops=6.0 * 4544 * case["n"] * case["epochs"])


# ---- the same in 64 bits, in plain torch --------------------------------------

_E = ((0, 0), (1, 0), (0, 1), (-1, 0), (0, -1), (1, 1), (-1, 1), (-1, -1), (1, -1))
_W = (4 / 9,) + (1 / 9,) * 4 + (1 / 36,) * 4


def _feq(rho, u, v):
    uu = u * u + v * v
    out = []
    for (ex, ey), w in zip(_E, _W):
        eu = ex * u + ey * v
        out.append(w * rho * (1.0 + 3.0 * eu + 4.5 * eu * eu - 1.5 * uu))
    return out


def _force(rho, T, roll):
    """psi and F of the interaction (G = -1) from the density."""
    num = rho * (1.0 + rho + rho * rho - rho ** 3)
    p = T * num / (1.0 - rho) ** 3 - rho * rho
    psi = torch.sqrt(-2.0 * (p - rho / 3.0))
    fx = fy = 0.0
    for ex, ey in _E[1:]:
        w = 1.0 / 3.0 if ex * ex + ey * ey == 1 else 1.0 / 12.0
        n = roll(psi, -ex, -ey)  # the neighbour at x + e
        fx, fy = fx + w * ex * n, fy + w * ey * n
    return psi, psi * fx, psi * fy


_MRT = np.array([[1] * 9, [-4, -1, -1, -1, -1, 2, 2, 2, 2], [4, -2, -2, -2, -2, 1, 1, 1, 1],
                 [0, 1, 0, -1, 0, 1, -1, -1, 1], [0, -2, 0, 2, 0, 1, -1, -1, 1],
                 [0, 0, 1, 0, -1, 1, 1, -1, -1], [0, 0, -2, 0, 2, 1, 1, -1, -1],
                 [0, 1, -1, 1, -1, 0, 0, 0, 0], [0, 0, 0, 0, 0, 1, -1, 1, -1]], dtype=np.float64)


def _guo(be, ce, fx, fy, vx, vy):
    """w [3 B (e.F) + C (9 (e.V)(e.F) - 3 V.F)] for the nine directions."""
    vf = vx * fx + vy * fy
    out = []
    for (ex, ey), w in zip(_E, _W):
        ef, ev = ex * fx + ey * fy, ex * vx + ey * vy
        out.append(w * (3.0 * be * ef + ce * (9.0 * ev * ef - 3.0 * vf)))
    return out


def _step(f, T, scheme, tau, sigma, roll):
    rho = sum(f)
    ux = (f[1] - f[3] + f[5] - f[6] - f[7] + f[8]) / rho
    uy = (f[2] - f[4] + f[5] + f[6] - f[7] - f[8]) / rho
    om = 1.0 / tau
    if scheme == "noforce":
        post = [a + om * (e - a) for a, e in zip(f, _feq(rho, ux, uy))]
        return [roll(a, ex, ey) for a, (ex, ey) in zip(post, _E)]
    psi, fx, fy = _force(rho, T, roll)
    vx, vy = ux + 0.5 * fx / rho, uy + 0.5 * fy / rho
    sg = sigma / (tau - 0.5) / (psi * psi)
    guo = 1.0 - 0.5 * om
    if scheme == "sc":
        eq, term = _feq(rho, ux + tau * fx / rho, uy + tau * fy / rho), [0.0] * 9
    elif scheme == "edm":
        eq, term = _feq(rho, ux, uy), _guo(1.0, 1.0, fx, fy, vx, vy)
    elif scheme == "edm_mod":
        eq, term = _feq(rho, ux, uy), _guo(1.0, om, fx, fy, vx, vy)
    elif scheme == "ladd":
        eq, term = _feq(rho, ux, uy), _guo(1.0, 1.0, fx, fy, ux, uy)
    elif scheme == "improved":
        eq, term = _feq(rho, vx, vy), _guo(guo, guo, fx, fy, vx + sg * fx, vy + sg * fy)
    else:  # mrt: relax the moments, each at its own rate
        M = torch.from_numpy(_MRT).to(rho.device)
        s = torch.tensor([0.0, MRT_RATES[0], MRT_RATES[1], 0.0, MRT_RATES[2], 0.0, MRT_RATES[2],
                          om, om], dtype=torch.float64, device=rho.device)
        mm = lambda m, a: torch.einsum("ij,j...->i...", m, torch.stack(a))  # noqa: E731
        m = mm(M, f)
        meq = mm(M, _feq(rho, vx, vy))
        mf = mm(M, _guo(1.0, 1.0, fx, fy, vx + sg * fx, vy + sg * fy))
        col = (slice(None),) + (None,) * rho.dim()
        m = m - s[col] * (m - meq) + (1.0 - 0.5 * s)[col] * mf
        # the momentum relaxes towards j + F / 2 at no rate: it gains F
        m[3], m[5] = rho * ux + fx, rho * uy + fy
        post = list(torch.einsum("ij,j...->i...", torch.linalg.inv(M), m))
        return [roll(a, ex, ey) for a, (ex, ey) in zip(post, _E)]
    post = [a + om * (e - a) + t for a, e, t in zip(f, eq, term)]
    return [roll(a, ex, ey) for a, (ex, ey) in zip(post, _E)]


def _exact_lattice(case, seed):
    T = case["T"] * _critical()[1]
    rho = torch.from_numpy(_field(case, seed)).cuda()
    roll = lambda a, ex, ey: torch.roll(a, (ey, ex), (0, 1)) if ex or ey else a  # noqa: E731
    ux, uy = (torch.zeros_like(rho) if a is None else torch.from_numpy(a).cuda()
              for a in _flow(case, seed))
    f = _feq(rho, ux, uy)
    for _ in range(case["steps"]):
        f = _step(f, T, case["scheme"], case["tau"], case["sigma"], roll)
    rho = sum(f)
    fx = fy = 0.0
    if case["scheme"] != "noforce":
        _, fx, fy = _force(rho, T, roll)
    vx = (f[1] - f[3] + f[5] - f[6] - f[7] + f[8] + 0.5 * fx) / rho
    vy = (f[2] - f[4] + f[5] + f[6] - f[7] - f[8] + 0.5 * fy) / rho
    return dict(rho=rho.cpu().numpy(), vx=vx.cpu().numpy(), vy=vy.cpu().numpy())


def _exact_mlp(case, seed):
    X, Y = (a.astype(np.float64) for a in _samples(case["n"], seed))
    p = warmstart.glorot_params(seed).astype(np.float64)
    cut = np.cumsum([256, 64, 4096, 64, 192])

    def forward(p, x):
        w1, b1, w2, b2, w3, b3 = np.split(p, cut)
        h1 = np.tanh(x @ w1.reshape(4, 64) + b1)
        h2 = np.tanh(h1 @ w2.reshape(64, 64) + b2)
        return h1, h2, h2 @ w3.reshape(64, 3) + b3

    if case["kind"] == "mlp_predict":
        return forward(p, X)[2]
    order, m, v, t, loss = _order(case, seed), np.zeros_like(p), np.zeros_like(p), 0, 0.0
    for e in range(case["epochs"]):
        for k in range(0, case["n"], case["batch"]):
            idx = order[e, k:k + case["batch"]]
            h1, h2, y = forward(p, X[idx])
            d = y - Y[idx]
            loss = float(np.mean(d * d))
            dy = 2.0 * d / d.size
            dz2 = (dy @ p[4480:4672].reshape(64, 3).T) * (1 - h2 * h2)
            dz1 = (dz2 @ p[320:4416].reshape(64, 64).T) * (1 - h1 * h1)
            g = np.concatenate([(X[idx].T @ dz1).ravel(), dz1.sum(0), (h1.T @ dz2).ravel(),
                                dz2.sum(0), (h2.T @ dy).ravel(), dy.sum(0)])
            t += 1
            m, v = 0.9 * m + 0.1 * g, 0.999 * v + 0.001 * g * g
            p = p - 2e-3 * (m / (1 - 0.9 ** t)) / (np.sqrt(v / (1 - 0.999 ** t)) + 1e-8)
    return dict(params=p, loss=np.float64(loss))


def exact(case, seed):
    if case["kind"] in ("mlp_predict", "mlp_train"):
        return _exact_mlp(case, seed)
    if case["kind"] == "sweep":  # thousands of steps of every instance: too long
        return None
    if case["nx"] * case["ny"] * case["steps"] > 2e9:
        return None
    return _exact_lattice(case, seed)
