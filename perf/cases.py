"""Timed cases: what a user of the library has it do, through its public entry points.

Four kinds of work:

* ``project``: a block of intervals of one population (``LrdmcSystem.step``),
  then its trace entries and the walkers read back, as a production run or a
  sampling run does between two blocks;
* ``batch``: the same for several systems in one ``LrdmcBatch``;
* ``evaluate``: one stateless evaluation of every lattice move of n
  configurations (``LrdmcSystem.evaluate``);
* ``train``: forward and backward pass of the neural pair Jastrow's
  objective over one minibatch.

Systems, spacings, interval lengths and population sizes are those of the
repository's benchmark, experiments and tests (a = 1/(3.5 Z) or 0.2, about
10 jumps per walker and interval); odd sizes stand for a user's own.
"""
import math

import numpy as np
import torch

import lrdmc_synth as S
import paper_1909_01589_gb300 as pkg

TRACE_CAPACITY = 1 << 16
RECOMPUTE_EVERY = 5
KINDS = {"single": pkg.SINGLE, "this_work": pkg.THIS_WORK, "previous": pkg.PREVIOUS}
PRECISIONS = {"df64": pkg.PRECISION_DF64, "fp64": pkg.PRECISION_FP64, "fp32": pkg.PRECISION_FP32}
E_TRIAL = {"He": -2.90, "Ne": -128.9, "Ar": -527.5, "Kr": -2753.0, "H2O": -76.0}
Z_MAX = {"He": 2, "Ne": 10, "Ar": 18, "Kr": 36, "H2O": 8}
# tau for about 10 jumps per walker and interval at a = 1/(3.5 Z_max)
TAU = {
    ("He", "single"): 0.0343, ("He", "this_work"): 0.0482, ("He", "previous"): 0.0429,
    ("Ne", "single"): 2.49e-4, ("Ne", "this_work"): 7.93e-4, ("Ne", "previous"): 9.80e-4,
    ("Ar", "single"): 4.51e-5, ("Ar", "this_work"): 1.919e-4, ("Ar", "previous"): 2.932e-4,
    ("Kr", "single"): 5.72e-6, ("Kr", "this_work"): 3.336e-5, ("Kr", "previous"): 6.42e-5,
    ("H2O", "single"): 4.11e-4, ("H2O", "this_work"): 1.338e-3, ("H2O", "previous"): 1.659e-3,
}


def _spacing(name):
    return pkg.Spacing(KINDS[name])


def _project(name, system, walkers, spacing, intervals, precision="df64", neural=False, equil=8, a=None, tau=None,
             jumps=10.0):
    return {"name": name, "kind": "project", "system": system, "walkers": walkers, "spacing": spacing,
            "precision": precision, "neural": neural, "a": a or 1.0 / (3.5 * Z_MAX[system]),
            "tau": tau or TAU[system, spacing], "jumps": jumps, "intervals": intervals, "equil": equil}


def listed():
    return [
        # the smallest production run: He, the population of the long parity test, latency bound
        _project("he_256_single", "He", 256, "single", 20, a=0.2, tau=0.068),
        # the benchmark's headline workload in the default arithmetic
        _project("ne_4096", "Ne", 4096, "this_work", 20, a=0.2, tau=0.025, equil=20, jumps=7.3),
        # the same in the mixed arithmetic (single-precision moves)
        _project("ne_4096_fp32", "Ne", 4096, "this_work", 20, "fp32", a=0.2, tau=0.025, jumps=7.3),
        # the same with a neural pair Jastrow installed
        _project("ne_4096_neural", "Ne", 4096, "this_work", 20, neural=True, a=0.2, tau=0.025, jumps=7.3),
        # the plain FP64 form that the efficiency metric is quoted against, an odd population
        _project("ne_1021_fp64", "Ne", 1021, "this_work", 4, "fp64", a=0.2, tau=0.025, jumps=7.3),
        # a molecule on the earlier double grid, an odd population
        _project("h2o_3001_previous", "H2O", 3001, "previous", 8),
        # the heavier atoms of the paper's scaling study; Kr is the largest system
        _project("ar_8192", "Ar", 8192, "this_work", 6),
        _project("kr_4096", "Kr", 4096, "this_work", 6),
        # a few configurations checked by a caller of its own
        {"name": "eval_h2o_37", "kind": "evaluate", "system": "H2O", "n": 37, "spacing": "this_work",
         "precision": "df64", "a": 1.0 / 28.0},
        # every lattice move of a large sample of configurations
        {"name": "eval_kr_16384", "kind": "evaluate", "system": "Kr", "n": 16384, "spacing": "this_work",
         "precision": "df64", "a": 1.0 / 126.0},
        # one optimisation step's gradient of the neural pair Jastrow, the default minibatch
        {"name": "train_ne_16384", "kind": "train", "system": "Ne", "n": 16384, "bf16": True},
        # five systems of one study projected together
        {"name": "batch_5x2048", "kind": "batch", "systems": "He,Ne,Ar,Kr,H2O", "walkers": 2048,
         "spacing": "this_work", "intervals": 4, "equil": 4},
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["project"] * 6 + ["evaluate"] * 3 + ["train", "batch"])
    if kind == "project":
        system = rng.choice(["He", "Ne", "Ne", "H2O", "Ar", "Kr"])
        most = {"He": 16384, "Ne": 8192, "H2O": 8192, "Ar": 8192, "Kr": 4096}[system]
        precision = rng.choice(["df64"] * 6 + ["fp32", "fp64"])
        neural = precision == "df64" and system in ("He", "Ne", "H2O") and rng.random() < 0.25
        if precision == "fp64":
            most //= 8
        W = _log_uniform(rng, 64, most)
        spacing = rng.choice(["single", "this_work", "this_work", "previous"])
        c = _project("", system, W, spacing, rng.choice([4, 5, 6]), precision, neural, equil=4)
    elif kind == "evaluate":
        system = rng.choice(["He", "Ne", "H2O", "Ar", "Kr"])
        c = {"kind": kind, "system": system, "n": _log_uniform(rng, 1, 16384),
             "spacing": rng.choice(["single", "this_work", "previous"]),
             "precision": rng.choice(["df64"] * 3 + ["fp32"]), "a": 1.0 / (3.5 * Z_MAX[system])}
    elif kind == "train":
        c = {"kind": kind, "system": rng.choice(["He", "Ne", "H2O"]), "n": _log_uniform(rng, 256, 16384),
             "bf16": rng.random() < 0.75}
    else:
        names = ["He", "Ne", "Ar", "Kr", "H2O"]
        c = {"kind": kind, "systems": ",".join(rng.sample(names, rng.randint(2, 4))),
             "walkers": _log_uniform(rng, 200, 2048), "spacing": rng.choice(["single", "this_work", "previous"]),
             "intervals": 4, "equil": 2}
    c.pop("name", None)
    return c


# ------------------------------------------------------------------ prepare and run
def _neural(system, seed, out_scale=0.5):
    spec = S.default_neural_spec(system)
    return spec, S.neural_init(spec, seed, out_scale=out_scale)


def _population(case, name, seed):
    """A system with its walkers after a few intervals."""
    system = S.make_system(name)
    g = pkg.LrdmcSystem(system).set_precision(PRECISIONS[case.get("precision", "df64")])
    if case.get("neural"):
        # a term as small as a trained one: it changes the energy's spread by a part of itself
        g.set_neural_jastrow(*_neural(system, seed, 0.2))
    tau = case.get("tau") or TAU[name, case["spacing"]]
    x0 = torch.tensor(S.initial_positions(system, case["walkers"], seed), device="cuda")
    g.init_walkers(x0, seed=seed, tau=tau, e_trial=E_TRIAL[name], recompute_every=RECOMPUTE_EVERY,
                   trace_capacity=TRACE_CAPACITY)
    return g


def prepare(case, seed):
    sp = _spacing(case.get("spacing", "this_work"))
    if case["kind"] == "project":
        g = _population(case, case["system"], seed)
        g.step(case["equil"], case["a"], sp)
        g.sync()
        trace = torch.zeros((3, TRACE_CAPACITY), dtype=torch.float64).pin_memory()
        return {"case": case, "g": g, "sp": sp, "k": case["equil"], "trace": trace}
    if case["kind"] == "batch":
        names = case["systems"].split(",")
        gs = [_population(case, name, seed + 17 * q) for q, name in enumerate(names)]
        batch = pkg.LrdmcBatch(gs, [1.0 / (3.5 * Z_MAX[name]) for name in names], [sp] * len(names))
        batch.set_carveout(100)  # the plan that the autotuner keeps for such a batch
        batch.step(case["equil"])
        batch.sync()
        trace = torch.zeros((len(names), 3, TRACE_CAPACITY), dtype=torch.float64).pin_memory()
        return {"case": case, "batch": batch, "gs": gs, "k": case["equil"], "trace": trace}
    system = S.make_system(case["system"])
    g = pkg.LrdmcSystem(system)
    x = torch.tensor(S.initial_positions(system, case["n"], seed), device="cuda")
    if case["kind"] == "evaluate":
        g.set_precision(PRECISIONS[case["precision"]])
        rot = torch.tensor(S.random_rotations(case["n"], seed + 1), device="cuda")
        return {"case": case, "g": g, "sp": sp, "x": x, "rot": rot}
    spec, params = _neural(system, seed)
    grad_base, e_base = g.base_terms(x)
    return {"case": case, "g": g, "spec": spec, "x": x, "grad_base": grad_base, "e_base": e_base,
            "params": torch.tensor(params, device="cuda", requires_grad=True)}


def run(state):
    case = state["case"]
    if case["kind"] == "project":
        g, k, n = state["g"], state["k"], case["intervals"]
        g.step(n, case["a"], state["sp"])
        g.energy_trace_async(k, n, state["trace"])
        state["k"] = k + n
        walkers = g.walkers()
        return {"trace": state["trace"][:, k:k + n], "walkers": walkers}
    if case["kind"] == "batch":
        k, n = state["k"], case["intervals"]
        state["batch"].step(n)
        state["batch"].sync()
        state["k"] = k + n
        out = []
        for q, g in enumerate(state["gs"]):
            g.energy_trace_async(k, n, state["trace"][q])
            out.append({"trace": state["trace"][q, :, k:k + n], "walkers": g.walkers()})
        return out
    if case["kind"] == "evaluate":
        ratio, T, b, el = state["g"].evaluate(state["x"], state["rot"], case["a"], state["sp"])
        return {"ratio": ratio, "T": T, "b": b, "el": el}
    from paper_1909_01589_gb300 import neural

    params = state["params"]
    params.grad = None
    el, j = neural.NeuralJastrowTerms.apply(params, state["g"], state["spec"], state["x"], state["grad_base"],
                                            state["e_base"], case["bf16"])
    loss = neural.variance_loss(el, j, True, 5.0)
    loss.backward()
    return {"el": el.detach(), "j": j.detach(), "loss": loss.detach(), "grad": params.grad}


# ------------------------------------------------------------------ necessary work
def _evaluation_ops(system, G):
    """Operations of one evaluation of all 6 G N moves and the local energy, from the formulas."""
    N, n_ao, n_nuc = system.N, system.n_ao, system.n_nuc
    exps = sum(len(s.alpha) if s.kind == S.GTO else 1 for s in system.shells)
    pairs = N - 1 + n_nuc
    move = 3 + 9 * n_nuc + 2 * exps + 4 * n_ao + 13 * pairs + 6
    local = N * (2 * exps + 12 * n_ao + 25 * pairs + n_ao * system.n_up)
    return 6 * G * N * move + local


def _projection_work(system, G, walkers, intervals, jumps):
    P = 6 * G * system.N
    update = 3 * system.n_up ** 2 + system.n_ao * (8 + system.n_up) + 2 * P
    record = 3 * system.N + system.n_up ** 2 + system.n_dn ** 2 + 9 + P + 2
    return (2.0 * 8 * record * walkers * intervals,
            (jumps * (_evaluation_ops(system, G) + update) + P) * float(walkers) * intervals)


def work(case):
    G = 1 if case.get("spacing") == "single" else 2
    if case["kind"] in ("project", "batch"):
        total = [0.0, 0.0]
        for name in (case["systems"].split(",") if case["kind"] == "batch" else [case["system"]]):
            w = _projection_work(S.make_system(name), G, case["walkers"], case["intervals"], case.get("jumps", 10.0))
            total = [a + b for a, b in zip(total, w)]
        return {"bytes": total[0], "flops": total[1]}
    system, n = S.make_system(case["system"]), case["n"]
    N = system.N
    if case["kind"] == "evaluate":
        P = 6 * G * N
        inverse = 2 * (system.n_up ** 3 + system.n_dn ** 3)
        return {"bytes": 8.0 * n * (3 * N + 9 + 2 * P + 2), "flops": float(n) * (_evaluation_ops(system, G) + inverse)}
    spec = S.default_neural_spec(system)
    H, D = spec.hidden, spec.n_in
    n_pairs = N * (N - 1) // 2 + N * system.n_nuc
    # value, first and second radial derivative through both layers, forward once and backward twice that
    network = 3 * 2 * (H * D + H * H + H)
    return {"bytes": 4.0 * (n * (4 * 3 * N + 2 + 4) + 2 * spec.n_params), "flops": 3.0 * n * n_pairs * network}


# ------------------------------------------------------------------ 64-bit values
def _slater_groups(Z):
    """(zeta, n*, electrons) of the groups of Slater's rules for a neutral atom."""
    fill = [(1, 0), (2, 0), (2, 1), (3, 0), (3, 1), (4, 0), (3, 2), (4, 1)]
    groups = [(1, 0), (2, 0), (3, 0), (3, 2), (4, 0)]
    nstar = {1: 1.0, 2: 2.0, 3: 3.0, 4: 3.7}
    occ, left = dict.fromkeys(groups, 0), Z
    for n, l in fill:
        put = min(left, 2 * (2 * l + 1))
        occ[n, 0 if l <= 1 else l] += put
        left -= put
    out = []
    for g, (n, t) in enumerate(groups):
        if not occ[n, t]:
            continue
        s = (occ[n, t] - 1) * (0.30 if n == 1 else 0.35)
        for h, (m, u) in enumerate(groups):
            if h == g:
                continue
            if t == 0:
                s += occ[m, u] * (0.85 if m == n - 1 else 1.0 if m < n - 1 else 0.0)
            elif h < g:
                s += occ[m, u]
        out.append(((Z - s) / nstar[n], nstar[n], occ[n, t]))
    return out


def _lattice(Z, a, spacing):
    """(G, a', r_c) of a spacing choice: S-13 with Eq. 6 and 7, or Eq. 4."""
    if spacing == "single":
        return 1, a, 1.0
    if spacing == "previous":
        return 2, a * math.sqrt(Z * Z / 4.0 + 1.0), Z / 2.0
    q = (a * Z) ** 2
    rc = 0.75 * (2.5 * q + 1.0) / (q + 1.0) * Z ** (-5.0 / 7.0)
    groups = _slater_groups(int(Z))
    # Eq. 7 by Gauss-Legendre panels; the Gaussian ends the integral at 40 r_c
    top = min(40.0 * rc, 80.0 / min(z for z, _, _ in groups))
    t, w = np.polynomial.legendre.leggauss(64)
    edges = np.linspace(0.0, top, 257)
    mid, half = 0.5 * (edges[1:] + edges[:-1]), 0.5 * (edges[1:] - edges[:-1])
    r = (mid[:, None] + half[:, None] * t).ravel()
    wr = (half[:, None] * w).ravel()
    f = sum(o * (2 * z) ** (2 * n + 1) / math.gamma(2 * n + 1) * r ** (2 * n) * np.exp(-2 * z * r) for z, n, o in groups)
    core = float(np.sum(wr * f * np.exp(-r * r / (2 * rc * rc))))
    return 2, a * math.sqrt((Z - core) / core), rc


def _solid(l, d):
    """Real solid harmonics of degree l and their gradients (lists over the components)."""
    x, y, z = d.unbind(-1)
    o, I = torch.zeros_like(x), torch.ones_like(x)
    if l == 0:
        return [I], [(o, o, o)]
    if l == 1:
        return [x, y, z], [(I, o, o), (o, I, o), (o, o, I)]
    return ([x * y, y * z, z * x, x * x - y * y, 2 * z * z - x * x - y * y],
            [(y, x, o), (o, z, y), (z, o, x), (2 * x, -2 * y, o), (-2 * x, -2 * y, 4 * z)])


def _radial(sh, r, derivatives):
    """R, R'/r and R'' of a shell."""
    if sh.kind == S.STO:
        m = sh.n_eff - 1 - sh.l
        R = r ** m * torch.exp(-sh.zeta * r)
        if not derivatives:
            return R, None, None
        t = m / r - sh.zeta
        return R, t * R / r, (t * t - m / (r * r)) * R
    R, R1, R2 = 0.0, 0.0, 0.0
    for al, c in zip(sh.alpha, sh.coef):
        g = c * torch.exp(-al * r * r)
        R = R + g
        if derivatives:
            R1 = R1 - 2 * al * g
            R2 = R2 + (4 * al * al * r * r - 2 * al) * g
    return R, R1, R2


def _orbital_dot(system, p, v, derivatives=False):
    """sum_mu v_mu chi_mu(p) and, on request, its gradient and Laplacian; v[..., n_ao] goes with p[..., 3]."""
    val, grad, lap, mu = 0.0, 0.0, 0.0, 0
    for sh in system.shells:
        d = p - torch.tensor(system.nuc_xyz[sh.center], device=p.device)
        r = torch.linalg.norm(d, dim=-1)
        R, R1, R2 = _radial(sh, r, derivatives)
        Sv, gS = _solid(sh.l, d)
        for s, g in zip(Sv, gS):
            c = v[..., mu]
            mu += 1
            val = val + c * s * R
            if derivatives:
                grad = grad + (c * R)[..., None] * torch.stack(g, -1) + (c * s * R1)[..., None] * d
                lap = lap + c * s * (R2 + 2 * (sh.l + 1) * R1)
    return val, grad, lap


def _orbitals(system, x):
    """chi_mu at every electron, [m][N][n_ao]."""
    out = []
    for sh in system.shells:
        d = x - torch.tensor(system.nuc_xyz[sh.center], device=x.device)
        R, _, _ = _radial(sh, torch.linalg.norm(d, dim=-1), False)
        out += [s * R for s in _solid(sh.l, d)[0]]
    return torch.stack(out, -1)


def _projected(system, x):
    """v[m][i][mu] = sum_o C[mu][o] Ainv[o][i] of the electron's spin block."""
    C = torch.tensor(system.C, device=x.device)
    chi, v = _orbitals(system, x), []
    for lo, n in ((0, system.n_up), (system.n_up, system.n_dn)):
        if n:
            inv = torch.linalg.inv(chi[:, lo:lo + n] @ C[:, :n])
            v.append((C[:, :n] @ inv).transpose(1, 2))
    return torch.cat(v, 1)


def _pair_strength(system, device):
    """c[i][j] of the electron pair's Pade term, 0 on the diagonal."""
    spin = torch.arange(system.N, device=device) < system.n_up
    c = torch.where(spin[:, None] == spin[None, :], float(system.c_par), float(system.c_anti)).double()
    return c * (1.0 - torch.eye(system.N, device=device, dtype=torch.float64))


def _base(system, x, v):
    """grad_i log|psi|, E_L and the Jastrow sum of every electron."""
    dev, N = x.device, system.N
    _, gD, lD = _orbital_dot(system, x, v, True)
    eye = torch.eye(N, device=dev, dtype=torch.float64)
    d = x[:, :, None] - x[:, None]
    r = torch.linalg.norm(d, dim=-1) + eye
    c, b = _pair_strength(system, dev), system.b_ee
    q = 1.0 / (1.0 + b * r)
    u1, u2 = c * q * q, -2.0 * b * c * q ** 3
    J = (c * r * q).sum(2)
    gJ = ((u1 / r)[..., None] * d).sum(2)
    lJ = (u2 + 2.0 * u1 / r).sum(2)
    V = (((1.0 - eye) / r).sum((1, 2)) * 0.5) if system.ee_on else 0.0
    en = system.en_b1 if system.en_b1 is not None else np.zeros(system.n_nuc)
    for I in range(system.n_nuc):
        d = x - torch.tensor(system.nuc_xyz[I], device=dev)
        r = torch.linalg.norm(d, dim=-1)
        q = 1.0 / (1.0 + system.en_b2 * r)
        u1, u2 = -en[I] * q * q, 2.0 * system.en_b2 * en[I] * q ** 3
        J = J - en[I] * r * q
        gJ = gJ + (u1 / r)[..., None] * d
        lJ = lJ + u2 + 2.0 * u1 / r
        V = V - (system.Z[I] / r).sum(1)
    for I in range(system.n_nuc):
        for K in range(I):
            V = V + system.Z[I] * system.Z[K] / float(np.linalg.norm(system.nuc_xyz[I] - system.nuc_xyz[K]))
    el = -0.5 * (lD + 2 * (gD * gJ).sum(-1) + lJ + (gJ * gJ).sum(-1)).sum(1) + V
    return gD + gJ, el, J


def _jastrow_at(system, x, p):
    """Jastrow sum of electron i displaced to p[m][i][q] against the others at x."""
    dev = x.device
    eye = torch.eye(system.N, device=dev, dtype=torch.float64)
    r = torch.linalg.norm(p[:, :, :, None] - x[:, None, None], dim=-1)
    J = (_pair_strength(system, dev)[:, None] * r / (1.0 + system.b_ee * r) * (1.0 - eye)[:, None]).sum(-1)
    en = system.en_b1 if system.en_b1 is not None else np.zeros(system.n_nuc)
    for I in range(system.n_nuc):
        r = torch.linalg.norm(p - torch.tensor(system.nuc_xyz[I], device=dev), dim=-1)
        J = J - en[I] * r / (1.0 + system.en_b2 * r)
    return J


def _exact_evaluate(case, seed):
    system = S.make_system(case["system"])
    a, Z = case["a"], float(np.max(system.Z))
    G, ap, rc = _lattice(Z, a, case["spacing"])
    x_all = torch.tensor(S.initial_positions(system, case["n"], seed), device="cuda")
    rot_all = torch.tensor(S.random_rotations(case["n"], seed + 1), device="cuda")
    parts = []
    for s in range(0, case["n"], 512):
        x, rot = x_all[s:s + 512], rot_all[s:s + 512].view(-1, 3, 3)
        v = _projected(system, x)
        _, el, J0 = _base(system, x, v)
        h = torch.tensor([a, ap][:G], device="cuda", dtype=torch.float64)
        # [m][1][g][axis][sign][3] displacements, flattened over the moves of an electron
        step = rot.transpose(1, 2)[:, None, None, :, None, :] * h[:, None, None, None]
        step = torch.cat([step, -step], 4).reshape(len(x), 1, 6 * G, 3)
        p = x[:, :, None] + step
        det, _, _ = _orbital_dot(system, p, v[:, :, None])
        ratio = det * torch.exp(_jastrow_at(system, x, p) - J0[:, :, None])
        if G == 2:
            mid = x[:, :, None] + 0.5 * step
            heavy = [I for I in range(system.n_nuc) if system.Z[I] == Z]
            d2 = torch.stack([((mid - torch.tensor(system.nuc_xyz[I], device="cuda")) ** 2).sum(-1) for I in heavy])
            d2 = d2.amin(0)
            pm = torch.exp(-d2 / (2 * rc * rc)) if case["spacing"] == "this_work" else 1.0 / (1.0 + rc * rc * d2)
            w = torch.cat([pm[..., :6], 1.0 - pm[..., 6:]], -1)
        else:
            w = torch.ones_like(ratio)
        scale = (0.5 / h ** 2).repeat_interleave(6)
        T = w * scale * ratio.clamp(min=0.0)
        parts.append((ratio.reshape(len(x), -1), T.reshape(len(x), -1), T.sum((1, 2)), el))
    ratio, T, b, el = (torch.cat(q) for q in zip(*parts))
    return {"ratio": ratio, "T": T, "b": b, "el": el}


def _silu_chain(z, z1, z2):
    """silu of z with the first and second radial derivative of its argument carried along."""
    sg = torch.sigmoid(z)
    d1 = sg * (1.0 + z * (1.0 - sg))
    d2 = sg * (1.0 - sg) * (2.0 + z * (1.0 - 2.0 * sg))
    return z * sg, d1 * z1, d2 * z1 * z1 + d1 * z2


def _pair_function(theta, spec, r, ch):
    """g_c(r), g' and g'' of the pair network with its cut-off."""
    H, D, o = spec.hidden, spec.n_in, 0
    parts = []
    for shape in ((H, D), (H,), (H, H), (H,), (H,), (1,)):
        n = int(np.prod(shape))
        parts.append(theta[o:o + n].view(shape))
        o += n
    W1, b1, W2, b2, w3, b3 = parts
    l2 = torch.tensor(spec.ell, device=r.device, dtype=torch.float64) ** 2
    r2 = (r * r)[:, None]
    den = r2 + l2
    hot = torch.nn.functional.one_hot(ch, spec.n_ch).double()
    z = torch.zeros_like(hot)
    f = [torch.cat(q, 1) for q in ((r2 / den, hot), (2.0 * r[:, None] * l2 / den ** 2, z),
                                   (2.0 * l2 * (l2 - 3.0 * r2) / den ** 3, z))]
    h = _silu_chain(f[0] @ W1.T + b1, f[1] @ W1.T, f[2] @ W1.T)
    h = _silu_chain(h[0] @ W2.T + b2, h[1] @ W2.T, h[2] @ W2.T)
    m, m1, m2 = h[0] @ w3 + b3, h[1] @ w3, h[2] @ w3
    rc = torch.tensor(spec.r_cut, device=r.device, dtype=torch.float64)[ch]
    t = (r / rc).clamp(max=1.0)
    s = 1 - 10 * t ** 3 + 15 * t ** 4 - 6 * t ** 5
    s1 = (-30 * t ** 2 + 60 * t ** 3 - 30 * t ** 4) / rc
    s2 = (-60 * t + 180 * t ** 2 - 120 * t ** 3) / rc ** 2
    return m * s, m1 * s + m * s1, m2 * s + 2 * m1 * s1 + m * s2


def _exact_train(case, seed):
    system = S.make_system(case["system"])
    spec, params = _neural(system, seed)
    dev, N = torch.device("cuda"), system.N
    x = torch.tensor(S.initial_positions(system, case["n"], seed), device=dev)
    grad_base, e_base, _ = _base(system, x, _projected(system, x))
    theta32 = torch.tensor(params, device=dev)
    theta = theta32.double().requires_grad_(True)
    used = theta + (theta32.bfloat16().double() - theta.detach()) if case["bf16"] else theta
    J, lap, G = 0.0, 0.0, torch.zeros_like(x)
    i, j = torch.triu_indices(N, N, 1, device=dev)
    pairs = [(i, j, x[:, i] - x[:, j], ((i < system.n_up) != (j < system.n_up)).long())] if N > 1 else []
    for I in range(system.n_nuc):
        e = torch.arange(N, device=dev)
        pairs.append((e, None, x - torch.tensor(system.nuc_xyz[I], device=dev),
                      torch.full((N,), 2 + int(spec.species[I]), device=dev)))
    for e, other, d, ch in pairs:
        r = torch.linalg.norm(d, dim=-1)
        g, g1, g2 = (q.view(r.shape) for q in _pair_function(used, spec, r.reshape(-1), ch.repeat(len(x))))
        gv = (g1 / r)[..., None] * d
        G = G.index_add(1, e, gv)
        l = (g2 + 2.0 * g1 / r).sum(1)
        if other is not None:
            G, l = G.index_add(1, other, -gv), 2.0 * l
        J, lap = J + g.sum(1), lap + l
    el = e_base - 0.5 * (2.0 * (grad_base * G).sum((1, 2)) + (G * G).sum((1, 2)) + lap)
    med = el.detach().median()
    mad = (el.detach() - med).abs().mean()
    lim = torch.minimum(torch.maximum(el, med - 5.0 * mad), med + 5.0 * mad)
    w = torch.exp(2.0 * (J - J.max().detach()))
    ebar = (w * lim).sum() / w.sum()
    loss = (w * (lim - ebar) ** 2).sum() / w.sum()
    loss.backward()
    return {"el": el.detach(), "j": J.detach(), "loss": loss.detach(), "grad": theta.grad}


def exact(case, seed):
    """What ``run`` returns in 64 bits; a projection's outcome is a chain of
    decisions over thousands of evaluations, for which there is no such value."""
    if case["kind"] == "evaluate":
        return _exact_evaluate(case, seed)
    if case["kind"] == "train":
        return _exact_train(case, seed)
    return None
