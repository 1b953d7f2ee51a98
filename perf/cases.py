"""The calls a program makes of this library, as measurable cases.

listed()  the cases; draw(rng) more of the same ranges; prepare(case, seed)
builds inputs and the handles such a program keeps; run(state) is one pass
through the public entry points; work(case) the bytes and operations a pass
cannot do without; exact(case, seed) the same outputs from plain torch in
complex double precision, where that is feasible.

Kinds of case:
  solve    hc.batched_solve: a batch of dense complex n x n systems.
  request  one instance, numpy in and out (Problem.track).
  track    a batch of dense total-degree instances on device tensors.
  plan     the same through a captured plan, pinned host buffers in and out.
  family   a batch of parameter-homotopy instances (computer vision scenes).
  serve    a burst of mixed requests through the continuous-batching server.
"""
import math
import os

import numpy as np
import torch

from paper_2112_03444_gb300 import hc, inputs

START_DIR = os.path.join(os.path.dirname(os.path.abspath(inputs.__file__)), "startsets")

FAMILIES = {  # family, scene generator, start set, tracked with sign symmetries
    "triangulation4": (lambda: inputs.triangulation_family(4),
                       lambda s: inputs.triangulation_scene(s)[0], "triangulation4", False),
    "triangulation2": (lambda: inputs.triangulation_family(2),
                       lambda s: inputs.triangulation_scene(s, views=2)[0], "triangulation2", False),
    "p3p": (inputs.p3p_family, lambda s: inputs.p3p_scene(s)[0], "p3p", True),
    "pose5_depth": (inputs.pose5_depth_family, lambda s: inputs.pose5_scene(s)[0], "pose5_depth",
                    True),
    "trifocal_f": (inputs.trifocal_family, lambda s: inputs.trifocal_scene(s)[0], "trifocal_f",
                   True),
}
STARTS = {"triangulation4": 296, "triangulation2": 8, "p3p": 8, "pose5_depth": 40,
          "trifocal_f": 5344}
# of the family's tracked starts: orbits of the sign symmetries
TRACKED = {"triangulation4": 296, "triangulation2": 8, "p3p": 4, "pose5_depth": 20,
           "trifocal_f": 1336}
PRECISION = {"fp64": hc.HC_PREC_FP64, "mixed": hc.HC_PREC_MIXED, "df": hc.HC_PREC_DF}


def listed():
    return [
        # the paper's standalone linear solver at its own batch size (Fig. 3):
        # latency of one launch
        dict(name="solve_c64_n8", kind="solve", n=8, batch=1000, dtype="c64"),
        # the solver in double precision at an odd size
        dict(name="solve_c128_n13", kind="solve", n=13, batch=40_000, dtype="c128"),
        # the solver at the paper's largest matrices, a batch larger than L2
        dict(name="solve_c64_n20", kind="solve", n=20, batch=100_000, dtype="c64"),
        # the smallest tracking call: one system of six quadratics, arrays on
        # the host, waited for -- a single hypothesis of an interactive program
        dict(name="request_quad6", kind="request", n=6, deg=2, instances=1, precision="mixed"),
        # a ragged cubic batch replayed from a plan with pinned buffers: the
        # steady loop of a program that tracks one batch size again and again
        dict(name="plan_cubic5", kind="plan", n=5, deg=3, instances=24, precision="mixed"),
        # the two heaviest classes of the dense sweep (mixed precision)
        dict(name="sweep_quad12", kind="track", n=12, deg=2, instances=16, precision="mixed"),
        dict(name="sweep_cubic8", kind="track", n=8, deg=3, instances=16, precision="mixed"),
        # plain double precision, six quadratics, for programs that want no
        # mixed precision at all
        dict(name="fp64_quad6", kind="track", n=6, deg=2, instances=64, precision="fp64"),
        # robust estimation loops: many scenes in one batch
        dict(name="triangulation4", kind="family", family="triangulation4", instances=600),
        dict(name="p3p", kind="family", family="p3p", instances=3000),
        # trifocal pose with unknown focal length: many starts, ill-conditioned
        # paths re-tracked in high precision; the step limit keeps a program
        # from waiting seconds for the few that crawl towards a failure
        dict(name="trifocal", kind="family", family="trifocal_f", instances=4, max_steps=800),
        # a burst of requests of all sizes through the server
        dict(name="serve_mix", kind="serve", requests=64),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["solve", "solve", "track", "track", "track", "plan", "family", "family"])
    if kind == "solve":
        n = rng.randint(3, 24)
        return dict(kind=kind, n=n, batch=_log(rng, 500, 4_000_000 // (n * n) * 10),
                    dtype=rng.choice(["c64", "c128"]))
    if kind == "family":
        name = rng.choice(["triangulation4", "triangulation2", "p3p", "pose5_depth"])
        most = {"triangulation4": 400, "triangulation2": 2000, "p3p": 3000, "pose5_depth": 400}
        return dict(kind=kind, family=name, instances=_log(rng, 1, most[name]))
    deg = rng.choice([2, 2, 3])
    n = rng.randint(3, 11) if deg == 2 else rng.randint(2, 7)
    precision = rng.choice(["mixed", "mixed", "mixed", "fp64", "df"])
    most = 40_000 if precision == "mixed" else 4_000  # paths
    return dict(kind=kind, n=n, deg=deg, instances=_log(rng, 1, max(2, most // deg ** n)),
                precision=precision)


# ---------------------------------------------------------------- inputs
def _dense_inputs(case, seed):
    """One system structure, its gamma, and coefficients [instances, terms]."""
    n, d, count = case["n"], case["deg"], case["instances"]
    base = inputs.dense_system(n, d, seed)
    rng = np.random.default_rng([seed, 0xC0, n, d, count])
    coef = rng.standard_normal((count, base.n_terms)) + 1j * rng.standard_normal(
        (count, base.n_terms))
    return base, inputs.unit_gamma(seed), coef


def _solve_inputs(case, seed):
    n, batch = case["n"], case["batch"]
    dt = torch.complex64 if case["dtype"] == "c64" else torch.complex128
    g = torch.Generator(device="cuda").manual_seed(seed * 7919 + n)
    A = torch.randn((batch, n, n), dtype=dt, device="cuda", generator=g)
    b = torch.randn((batch, n), dtype=dt, device="cuda", generator=g)
    return A, b


def _device_outputs(instances, paths, n):
    return dict(x=torch.zeros((instances, paths, n), dtype=torch.complex128, device="cuda"),
                status=torch.zeros((instances, paths), dtype=torch.uint8, device="cuda"),
                steps=torch.zeros((instances, paths, 3), dtype=torch.int32, device="cuda"),
                be=torch.zeros((instances, paths), dtype=torch.float64, device="cuda"))


def _family_problem(name, **settings):
    make, scene, starts, sym = FAMILIES[name]
    fam = make()
    z = np.load(os.path.join(START_DIR, starts + ".npz"))
    return hc.Problem(fam.system, kind=hc.HC_PARAMETER, p0=z["p0"], start=z["start"],
                      symmetries=fam.sign_masks if sym else (), settings=settings), scene


SERVE_SIZES = (4, 5, 6, 7, 8, 9, 10, 11, 12)


def prepare(case, seed):
    kind = case["kind"]
    s = dict(kind=kind, case=case)
    if kind == "solve":
        s["A"], s["b"] = _solve_inputs(case, seed)
        s["x"] = torch.empty_like(s["b"])
        s["info"] = torch.empty(case["batch"], dtype=torch.int32, device="cuda")
    elif kind in ("request", "track", "plan"):
        base, gamma, coef = _dense_inputs(case, seed)
        pr = hc.Problem(base, gamma=gamma, settings=dict(precision=PRECISION[case["precision"]]))
        s["problem"] = pr
        count, n = case["instances"], case["n"]
        if kind == "request":
            s["coef"] = coef
        elif kind == "track":
            s["coef"] = torch.from_numpy(coef).cuda()
            s["out"] = _device_outputs(count, pr.paths, n)
        else:
            s["plan"] = pr.plan(count)
            s["coef"] = torch.from_numpy(coef).pin_memory()
            s["out"] = {k: torch.zeros(v.shape, dtype=v.dtype, pin_memory=True)
                        for k, v in _device_outputs(count, pr.paths, n).items()}
    elif kind == "family":
        limit = dict(max_steps=case["max_steps"]) if "max_steps" in case else {}
        pr, scene = _family_problem(case["family"], **limit)
        count = case["instances"]
        p1 = np.stack([scene(1_000_003 * seed + k) for k in range(count)])
        s["problem"] = pr
        s["p1"] = torch.from_numpy(p1).cuda()
        s["out"] = _device_outputs(count, pr.paths, pr.n)
    elif kind == "serve":
        probs, gens = [], []
        for n in SERVE_SIZES:
            probs.append(hc.Problem(inputs.dense_system(n, 2, 700 + n),
                                    gamma=inputs.unit_gamma(700 + n)))
            gens.append(lambda k, n=n: inputs.dense_coefficients(n, 2, k).reshape(-1))
        for name in ("triangulation4", "p3p"):
            pr, scene = _family_problem(name)
            probs.append(pr)
            gens.append(scene)
        s["requests"] = [(probs[k % len(probs)], gens[k % len(probs)](1_000_003 * seed + k))
                         for k in range(case["requests"])]
        s["server"] = hc.Server()
    else:
        raise ValueError(kind)
    return s


# ---------------------------------------------------------------- one pass
def run(s):
    kind, case = s["kind"], s["case"]
    if kind == "solve":
        hc.batched_solve(s["A"], s["b"], s["x"], s["info"],
                         torch.cuda.current_stream().cuda_stream)
        return dict(x=s["x"], info=s["info"])
    if kind == "request":
        b = s["problem"].track(n_instances=case["instances"], coef=s["coef"]).wait()
        out = dict(x=b.x, status=b.status, steps=b.steps, be=b.be)
        b.close()
        return out
    if kind == "serve":
        srv = s["server"]
        ids = [(srv.submit(pr, data), pr) for pr, data in s["requests"]]
        got = [srv.wait(rid, pr) for rid, pr in ids]
        return dict(x=np.concatenate([x.reshape(-1) for x, _, _ in got]),
                    status=np.concatenate([st for _, st, _ in got]))
    o = s["out"]
    bufs = dict(x_out=o["x"], status_out=o["status"], steps_out=o["steps"], be_out=o["be"])
    if kind == "plan":
        b = s["plan"].run(coef=s["coef"], **bufs).wait()
    elif kind == "track":
        b = s["problem"].track(n_instances=case["instances"], coef=s["coef"], device=True,
                               **bufs).wait()
    else:
        b = s["problem"].track(n_instances=case["instances"], p1=s["p1"], device=True,
                               **bufs).wait()
    b.close()
    return dict(o)


# ---------------------------------------------------------------- work
# Steps (taken and rejected) and Newton iterations of a path, on average over
# seeded inputs of each class: what the method needs, whatever tracks it.
STEPS = {2: (38.0, 50.0), 3: (36.0, 48.0)}  # dense, by degree
FAMILY_STEPS = {"triangulation4": (61.0, 106.0), "triangulation2": (43.0, 59.0),
                "p3p": (34.0, 49.0), "pose5_depth": (52.0, 95.0), "trifocal_f": (107.0, 280.0)}


def _solve_cfma(n):
    return sum(j * (j + 1) for j in range(n)) + n * (n + 1) // 2


def _dense_work(n, d, instances):
    M = math.comb(n + d, d)
    e_h = n * M
    e_hx = n * sum(k * math.comb(n, k) * math.comb(d, k) for k in range(1, d + 1))
    steps, newton = STEPS[d]
    paths = instances * d ** n
    cfma = steps * 4 * (e_hx + e_h + _solve_cfma(n)) + newton * (e_h + e_hx + _solve_cfma(n))
    return dict(bytes=instances * n * M * 16 + paths * (16 * n + 21), flops=8.0 * cfma * paths)


def _family_work(name, instances):
    """One evaluation of H, dH/dx and dH/dt: three multiply-adds per factor of
    every term (prefix product, suffix product, derivative)."""
    system = FAMILIES[name][0]().system
    n = system.n
    factors = system.term_exp.astype(int).sum(1) + (system.term_param >= 0).sum(1)
    steps, newton = FAMILY_STEPS[name]
    cfma = (4 * steps + newton) * (3 * int(factors.sum()) + _solve_cfma(n))
    return dict(bytes=instances * (16 * system.n_params + STARTS[name] * (16 * n + 21)),
                flops=8.0 * cfma * instances * TRACKED[name])


def work(case):
    kind = case["kind"]
    if kind == "solve":
        n, batch, e = case["n"], case["batch"], 8 if case["dtype"] == "c64" else 16
        return dict(bytes=batch * ((n * n + 2 * n) * e + 4), flops=8.0 * batch * _solve_cfma(n))
    if kind == "family":
        return _family_work(case["family"], case["instances"])
    if kind == "serve":
        parts = [_dense_work(n, 2, 1) for n in SERVE_SIZES]
        parts += [_family_work(name, 1) for name in ("triangulation4", "p3p")]
        return {k: case["requests"] * sum(p[k] for p in parts) / len(parts)
                for k in ("bytes", "flops")}
    return _dense_work(case["n"], case["deg"], case["instances"])


# ---------------------------------------------------------------- 64-bit values
class _Dense64:
    """H = (1 - t) gamma G + t F of dense instances, in torch complex128."""

    def __init__(self, n, d, gamma, coef, exps):
        self.n, self.d, self.gamma = n, d, gamma
        self.C = coef.reshape(coef.shape[0], n, -1)  # [I, n, M]
        idx = [[v for v in range(n) for _ in range(int(e[v]))] for e in exps]
        idx = [r + [n] * (d - len(r)) for r in idx]  # n: the constant 1
        self.idx = torch.tensor(idx, device=coef.device)  # [M, d]

    def __call__(self, x, t):
        """x [I, P, n], t [I, P] -> H, Hx, Ht."""
        n, d = self.n, self.d
        x1 = torch.cat([x, torch.ones_like(x[..., :1])], -1)
        f = x1[..., self.idx]  # [I, P, M, d]
        F = torch.einsum("ipm,inm->ipn", f.prod(-1), self.C)
        J = torch.zeros(x.shape + (n,), dtype=x.dtype, device=x.device)
        for a in range(d):
            rest = torch.ones_like(f[..., 0])
            for b in range(d):
                if b != a:
                    rest = rest * f[..., b]
            for j in range(n):
                m = self.idx[:, a] == j
                J[..., j] += torch.einsum("ipm,inm->ipn", rest[..., m], self.C[..., m])
        G = x ** d - 1
        tt, gm = t[..., None], self.gamma
        Hx = tt[..., None] * J + torch.diag_embed((1 - tt) * gm * d * x ** (d - 1))
        return tt * F + (1 - tt) * gm * G, Hx, F - gm * G


def _track64(H, x):
    """The endpoints at t = 1 of the paths from x at t = 0 (Runge-Kutta 4 and
    Newton in complex double precision, small steps); None if one is lost."""
    t = torch.zeros(x.shape[:2], dtype=torch.float64, device=x.device)
    dt = torch.full_like(t, 0.01)
    good = torch.zeros_like(t)

    def rate(y, s):
        _, Hx, Ht = H(y, s)
        return torch.linalg.solve(Hx, -Ht[..., None])[..., 0]

    for _ in range(1500):
        if bool((t >= 1).all()):
            break
        h = torch.minimum(dt, 1 - t)
        k1 = rate(x, t)
        k2 = rate(x + 0.5 * h[..., None] * k1, t + 0.5 * h)
        k3 = rate(x + 0.5 * h[..., None] * k2, t + 0.5 * h)
        k4 = rate(x + h[..., None] * k3, t + h)
        y = x + h[..., None] / 6 * (k1 + 2 * k2 + 2 * k3 + k4)
        t1 = torch.where(h >= 1 - t, torch.ones_like(t), t + h)
        ok = torch.ones_like(t, dtype=torch.bool)
        for it in range(3):
            v, Hx, _ = H(y, t1)
            c = torch.linalg.solve(Hx, -v[..., None])[..., 0]
            y = y + c
            size = c.abs().amax(-1) / (1 + y.abs().amax(-1))
            if it == 0:
                ok = size <= 1e-3
        ok = ok & (size <= 1e-10)
        x = torch.where(ok[..., None], y, x)
        t = torch.where(ok, t1, t)
        good = torch.where(ok, good + 1, torch.zeros_like(good))
        dt = torch.where(ok, dt, dt / 2)
        grow = good >= 3
        dt = torch.where(grow, torch.clamp(2 * dt, max=0.05), dt)
        good = torch.where(grow, torch.zeros_like(good), good)
        if bool((dt < 1e-7).any()):
            return None
    if not bool((t >= 1).all()):
        return None
    for _ in range(3):
        v, Hx, _ = H(x, t)
        x = x - torch.linalg.solve(Hx, v[..., None])[..., 0]
    # two paths at one root: a path has been lost
    for one in x:
        if one.shape[0] > 1:
            far = torch.cdist(torch.view_as_real(one).flatten(1), torch.view_as_real(one).flatten(1))
            far.fill_diagonal_(math.inf)
            if float(far.min()) < 1e-6:
                return None
    return x


def exact(case, seed):
    kind = case["kind"]
    if kind == "solve":
        A, b = _solve_inputs(case, seed)
        x = torch.linalg.solve(A.to(torch.complex128), b.to(torch.complex128)[..., None])[..., 0]
        return dict(x=x, info=None)
    if kind not in ("request", "track", "plan"):
        return None
    n, d = case["n"], case["deg"]
    paths = d ** n
    if case["instances"] * paths * math.comb(n + d, d) * n > 4_000_000:
        return None
    base, gamma, coef = _dense_inputs(case, seed)
    exps = base.term_exp[:math.comb(n + d, d)]
    dev = torch.device("cuda")
    H = _Dense64(n, d, gamma, torch.from_numpy(coef).to(dev), exps)
    digits = (np.arange(paths)[:, None] // d ** np.arange(n)[None, :]) % d
    start = np.exp(2j * np.pi * digits / d)
    x0 = torch.from_numpy(start).to(dev).expand(case["instances"], paths, n).clone()
    x = _track64(H, x0)
    return None if x is None else dict(x=x, status=None, steps=None, be=None)
