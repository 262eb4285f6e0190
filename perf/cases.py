"""The measured workloads: what programs that use this library have it do, through ``native``.

Four kinds of call:

* ``solve``  -- one Hamilton-Jacobi problem: initial data from a device array, whole RK3 steps (to a final
  time, or a number of them), the solution back into a device array.  FP64 returns float64; FP32 and MIXED
  return float32, the type their stencil computes in.
* ``batch``  -- many independent instances of uneven size from host arrays to host arrays.
* ``serve``  -- a burst of requests to a resident server, from submission to the last result.

The problems are the paper's examples at the sizes of the library's tests and benchmark; every seed moves
the phase (or the kinks) of the initial data.
"""
import math

import numpy as np
import torch

from paper_1909_13263_gb300 import native

# name: (dim, Hamiltonian, lo, hi, boundary, time unit)
PROBLEMS = {
    "ex6": (1, "burgers1d", -1.0, 1.0, "periodic", 1.0 / math.pi**2),
    "ex2": (1, "negcos1d", -1.0, 1.0, "periodic", 1.0 / math.pi**2),
    "ex3": (2, "burgers2d", -2.0, 2.0, "periodic", 1.0 / math.pi**2),
    "ex4": (2, "negcos2d", -2.0, 2.0, "periodic", 1.0 / math.pi**2),
    "ex10": (2, "sin2d", -1.0, 1.0, "linextrap", 1.0),
    "ex12": (2, "eikonal2d", 0.0, 1.0, "periodic", 1.0),
}


def _solve(name, problem, nx, ny, precision, steps=0, t=0.0, weights="arclength"):
    return {"name": name, "kind": "solve", "problem": problem, "nx": nx, "ny": ny, "precision": precision,
            "steps": steps, "t": t, "weights": weights}


def listed():
    return [
        # the smallest call: one accuracy-table run in 1D (smooth Burgers solution), about a dozen steps
        _solve("1d_80_fp64", "ex6", 80, 1, "fp64", t=0.5),
        # the longest 1D run of the paper's examples: through the kink, some four hundred steps
        _solve("1d_320_kink_fp64", "ex6", 320, 1, "fp64", t=3.5),
        # a whole 2D solve in double at a table size
        _solve("2d_400_fp64", "ex3", 400, 400, "fp64", t=0.5),
        # a large grid in double: a few steps of a longer run
        _solve("2d_2048_fp64", "ex3", 2048, 2048, "fp64", steps=3),
        # kinks and extrapolated boundaries in double (the reference arm of the precision study)
        _solve("ex10_1024_fp64", "ex10", 1024, 1024, "fp64", steps=4),
        # plain float storage on an ordinary grid
        _solve("2d_2048_fp32", "ex3", 2048, 2048, "fp32", steps=40),
        # a whole 2D solve in mixed precision on a small, ragged grid: latency and launches
        _solve("2d_403x397_mixed", "ex3", 403, 397, "mixed", t=0.5),
        # the largest grid, the benchmark's size
        _solve("2d_8192_mixed", "ex3", 8192, 8192, "mixed", steps=10),
        # kinks and extrapolated boundaries in mixed precision
        _solve("ex10_1024_mixed", "ex10", 1024, 1024, "mixed", steps=60),
        # the classical indicators, a rectangular ragged grid, a Hamiltonian with sines
        _solve("2d_1500x901_mixed_jp", "ex4", 1500, 901, "mixed", steps=60, weights="jp"),
        # many small and middle instances at once, two Hamiltonians, host to host
        {"name": "batch_48", "kind": "batch", "count": 48, "lo_side": 64, "hi_side": 512, "mix": 1,
         "precision": "mixed"},
        # a burst of requests to a resident server
        {"name": "serve_24", "kind": "serve", "count": 24, "lo_side": 128, "hi_side": 768, "mix": 2,
         "precision": "mixed"},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


# nodes x steps of a drawn solve, by precision: no more work than the largest listed case of that precision
_CAP_2D = {"fp64": 1.1e7, "fp32": 6.0e8, "mixed": 6.0e8}


def draw(rng):
    kind = rng.choices(["1d", "2d", "batch", "serve"], weights=[2, 6, 1, 1])[0]
    if kind == "batch" or kind == "serve":
        lo = 64 if kind == "batch" else 128
        count = _log_int(rng, 6, 48 if kind == "batch" else 24)
        hi = _log_int(rng, 160, 512 if kind == "batch" else 768)
        return {"kind": kind, "count": count, "lo_side": lo, "hi_side": hi, "mix": rng.randrange(1 << 16),
                "precision": rng.choice(["mixed", "mixed", "fp32"])}
    weights = rng.choice(["arclength", "arclength", "arclength", "jp"])
    if kind == "1d":
        n = _log_int(rng, 40, 320)
        c = _solve("", rng.choice(["ex6", "ex6", "ex2"]), n, 1, "fp64", t=round(rng.uniform(0.2, 3.5), 3), weights=weights)
    else:
        precision = rng.choice(["fp64", "fp32", "mixed", "mixed"])
        problem = rng.choice(["ex3", "ex3", "ex4", "ex10", "ex10", "ex12"])
        nx = _log_int(rng, 64, 2048 if precision == "fp64" else 8192)
        ny = min(8192, max(48, int(nx * rng.uniform(0.6, 1.4))))
        nodes = nx * ny
        if precision == "fp64" and nodes > 2048 * 2048:
            ny = 2048 * 2048 // nx
            nodes = nx * ny
        most = _CAP_2D[precision] / nodes
        c = _solve("", problem, nx, ny, precision, steps=max(1, min(_log_int(rng, 4, 80), int(most))), weights=weights)
    del c["name"]
    return c


# ---------------------------------------------------------------- inputs

def _axis(n, lo, hi, bc):
    dx = (hi - lo) / (n if bc == "periodic" else n - 1)
    return lo + dx * np.arange(n, dtype=np.float64), dx


def _phi0(problem, nx, ny, rng):
    """Initial data as float64 numpy values of the two axes combined on the GPU; (tensor, dx, dy)."""
    dim, _, lo, hi, bc, _ = PROBLEMS[problem]
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    x, dx = _axis(nx, lo, hi, bc)
    x = torch.from_numpy(x).to(dev)
    th = rng.uniform(0.0, 2.0 * math.pi)
    if dim == 1:
        return -torch.cos(math.pi * x + th), dx, dx
    y, dy = _axis(ny, lo, hi, bc)
    x, y = x[None, :], torch.from_numpy(y).to(dev)[:, None]
    if problem in ("ex3", "ex4"):
        return -torch.cos(0.5 * math.pi * (x + y) + th), dx, dy
    if problem == "ex10":  # kinks through a point near the middle
        x0, y0 = rng.uniform(-0.05, 0.05), rng.uniform(-0.05, 0.05)
        return math.pi * ((y - y0).abs() - (x - x0).abs()), dx, dy
    a, b = rng.uniform(0.0, 2.0 * math.pi), rng.uniform(0.0, 2.0 * math.pi)
    return 0.25 * (torch.cos(2 * math.pi * x + a) - 1.0) * (torch.cos(2 * math.pi * y + b) - 1.0) - 1.0, dx, dy


def _instances(case, rng):
    """Square periodic grids, log-uniform sides, both Hamiltonians (by the case's mix); random phase and end time."""
    mix = np.random.default_rng(case["mix"])
    out = []
    for _ in range(case["count"]):
        n = int(round(math.exp(mix.uniform(math.log(case["lo_side"]), math.log(case["hi_side"])))))
        problem = "ex3" if mix.random() < 0.5 else "ex4"
        phi0, dx, _ = _phi0(problem, n, n, rng)
        out.append((problem, n, phi0, dx, float(rng.uniform(0.1, 0.5) / math.pi**2)))
    return out


def prepare(case, seed):
    native.load()
    native.use_torch_allocator(True)
    rng = np.random.default_rng(seed)
    if case["kind"] == "solve":
        dim, ham, lo, hi, bc, unit = PROBLEMS[case["problem"]]
        phi0, _, _ = _phi0(case["problem"], case["nx"], case["ny"], rng)
        solver = native.Solver(dim=dim, nx=case["nx"], ny=case["ny"], bc=bc, xlo=lo, xhi=hi, ylo=lo, yhi=hi, ham=ham,
                               weights=case["weights"], precision=case["precision"])
        return {"kind": "solve", "solver": solver, "phi0": phi0, "steps": case["steps"], "t": case["t"] * unit,
                "dtype": torch.float64 if case["precision"] == "fp64" else torch.float32}
    st = {"kind": case["kind"], "precision": case["precision"], "jobs": []}
    for problem, n, phi0, _, tf in _instances(case, rng):
        _, ham, lo, hi, _, _ = PROBLEMS[problem]
        st["jobs"].append(dict(nx=n, ny=n, xlo=lo, xhi=hi, ylo=lo, yhi=hi, ham=ham, phi0=phi0.cpu().numpy(),
                               t_final=tf))
    if case["kind"] == "serve":
        st["server"] = native.Server(hbm_budget_bytes=2 << 30, max_slots=64, max_side=768, precision=case["precision"])
    return st


def run(state):
    if state["kind"] == "solve":
        s = state["solver"]
        s.set_phi0(state["phi0"])
        if state["steps"]:
            s.advance(state["steps"])
        else:
            s.step_to(state["t"])
        out = torch.empty(state["phi0"].shape, dtype=state["dtype"], device="cuda")
        return s.get_phi_device(out)
    # results of the float stencil are kept as float32
    if state["kind"] == "batch":
        with native.Batch(precision=state["precision"]) as b:
            for job in state["jobs"]:
                b.add(**job)
            b.run()
            return [b.get_phi(i).astype(np.float32) for i in range(len(state["jobs"]))]
    server = state["server"]
    ids = [server.submit(**job) for job in state["jobs"]]
    out = []
    for i in ids:
        done, info, phi = server.poll(i, timeout=60.0)
        if not done or info["status"] != 0:
            raise RuntimeError("request %d failed: %r" % (i, info))
        out.append(phi.astype(np.float32))
    return out


# ---------------------------------------------------------------- work

def _steps_of(case, n, t):
    """About the number of RK3 steps to time t (CFL 0.6 with the largest |dH/dp| of the problem)."""
    dim, ham, lo, hi, _, _ = PROBLEMS[case]
    alpha = {"burgers1d": math.pi + 1.0, "burgers2d": math.pi / 2 * 1.0 + 1.0 + math.pi / 2}.get(ham, 1.0)
    return max(1.0, math.ceil(t * dim * alpha / (0.6 * (hi - lo) / n)))


def work(case):
    """Per RK3 step: phi read and written once at its storage width; about 250 (2D) or 120 (1D) operations per
    node and stage; plus the input and the output array."""
    if case["kind"] == "solve":
        dim, _, _, _, _, unit = PROBLEMS[case["problem"]]
        nodes = case["nx"] * case["ny"]
        steps = case["steps"] or _steps_of(case["problem"], case["nx"], case["t"] * unit)
        width = 4 if case["precision"] == "fp32" else 8
        out = 8 if case["precision"] == "fp64" else 4
        return {"bytes": nodes * (2.0 * width * steps + 8 + out),
                "flops": nodes * steps * 3.0 * (250 if dim == 2 else 120)}
    # instances: the mean over the log-uniform sides of n^2 x steps (steps proportional to n), mean end time
    lo, hi = case["lo_side"], case["hi_side"]
    ln = math.log(hi / lo)
    n2, n3 = (hi**2 - lo**2) / (2 * ln), (hi**3 - lo**3) / (3 * ln)
    per_n = 0.5 * (_steps_of("ex3", 1000, 0.3 / math.pi**2) + _steps_of("ex4", 1000, 0.3 / math.pi**2)) / 1000.0
    width = 4 if case["precision"] == "fp32" else 8
    return {"bytes": case["count"] * (n3 * per_n * 2.0 * width + n2 * 16.0),
            "flops": case["count"] * n3 * per_n * 750.0}


# ---------------------------------------------------------------- the same in 64 bits, plainly

def _ghosts(phi, bc, axis):
    """phi with three ghost values on either side along `axis`."""
    n = phi.shape[axis]

    def at(i):
        return phi.narrow(axis, i, 1)

    if bc == "periodic":
        left = [at((-k) % n) for k in (3, 2, 1)]
        right = [at((n - 1 + k) % n) for k in (1, 2, 3)]
    else:
        left = [(1.0 + k) * at(0) - k * at(1) for k in (3, 2, 1)]
        right = [(1.0 + k) * at(n - 1) - k * at(n - 2) for k in (1, 2, 3)]
    return torch.cat(left + [phi] + right, dim=axis)


def _mean_length(a, b):
    """Mean of sqrt(1 + u^2) over [a, b].  With sigma = sqrt(1+a^2) + sqrt(1+b^2) and t = (b - a) / sigma it is
    sigma / 2 - (1 / (1 - t^2) - atanh(t) / t) / sigma; by its series for short intervals and by the
    primitive (u sqrt(1+u^2) + asinh u) / 2 for long ones."""
    sa, sb, h = torch.sqrt(1.0 + a * a), torch.sqrt(1.0 + b * b), b - a
    sg = sa + sb
    x = (h / sg) ** 2
    c = torch.full_like(x, 20.0 / 21.0)
    for k in range(9, 0, -1):
        c = c * x + 2.0 * k / (2.0 * k + 1.0)
    series = 0.5 * sg - c * x / sg
    prim = (b * sb + torch.asinh(b) - a * sa - torch.asinh(a)) / (2.0 * torch.where(h == 0, torch.ones_like(h), h))
    return torch.where(x < 0.01, series, prim)


def _one_sided(p, dx, weights, eps):
    """phi_x^-, phi_x^+ along the last axis of p, which holds three ghosts on either side."""
    n = p.shape[-1] - 6
    v = (p[..., 1:] - p[..., :-1]) / dx

    def at(q, m):  # q's entries for the nodes 0..n-1 at offset m
        return q[..., m:m + n]

    if weights == "arclength":
        d2 = (v[..., 1:] - v[..., :-1]) / dx          # d2[m - 1] belongs to m
        i = d2[..., 1:-1]                             # m = 2 ..
        def q(a, b):
            return (eps + (dx * _mean_length(a, b)) ** 2) ** 2
        qx = q(i, 2.0 * i - d2[..., :-2])             # entry m - 2
        qy = q(i, d2[..., 2:])
        qz = q(2.0 * i - d2[..., 2:], i)
        minus = (at(qx, 0), at(qy, 0), at(qz, 1))
        plus = (at(qz, 2), at(qy, 1), at(qx, 1))
    else:
        s = v[..., 1:] - v[..., :-1]                  # s[m - 1] belongs to m
        x, y = s[..., :-1], s[..., 1:]                # entry m - 1
        d = 13.0 * (x - y) ** 2
        qx, qy, qz = ((eps + d + 3.0 * w ** 2) ** 2 for w in (x - 3.0 * y, x + y, 3.0 * x - y))
        minus = (at(qx, 0), at(qy, 1), at(qz, 2))
        plus = (at(qz, 3), at(qy, 2), at(qx, 1))

    def combine(q3, a, b, c, d, e):
        w = [g / q for g, q in zip((0.1, 0.6, 0.3), q3)]
        k = [(2.0 * a - 7.0 * b + 11.0 * c) / 6.0, (-b + 5.0 * c + 2.0 * d) / 6.0, (2.0 * c + 5.0 * d - e) / 6.0]
        return (w[0] * k[0] + w[1] * k[1] + w[2] * k[2]) / (w[0] + w[1] + w[2])

    return (combine(minus, at(v, 0), at(v, 1), at(v, 2), at(v, 3), at(v, 4)),
            combine(plus, at(v, 5), at(v, 4), at(v, 3), at(v, 2), at(v, 1)))


def _hamiltonian(ham):
    """(H(p, q), |H_p|(p, q), |H_q|(p, q))"""
    if ham in ("burgers1d", "burgers2d"):
        a = lambda p, q: (p + q + 1.0).abs()  # noqa: E731
        return (lambda p, q: 0.5 * (p + q + 1.0) ** 2), a, a
    if ham in ("negcos1d", "negcos2d"):
        a = lambda p, q: torch.sin(p + q + 1.0).abs()  # noqa: E731
        return (lambda p, q: -torch.cos(p + q + 1.0)), a, a
    if ham == "sin2d":
        a = lambda p, q: torch.cos(p + q).abs()  # noqa: E731
        return (lambda p, q: torch.sin(p + q)), a, a
    root = lambda p, q: torch.sqrt(p * p + q * q + 1.0)  # noqa: E731
    return root, (lambda p, q: p.abs() / root(p, q)), (lambda p, q: q.abs() / root(p, q))


def _max4(f, um, up, vm, vp):
    return torch.maximum(torch.maximum(f(um, vm), f(um, vp)), torch.maximum(f(up, vm), f(up, vp)))


def _rhs(phi, alpha, dim, ham, bc, dx, dy, weights, eps=1e-6):
    """L(phi) with the given flux alpha (1D: each node's own), and the grid maxima of |H_p|, |H_q|."""
    h, hp, hq = _hamiltonian(ham)
    if dim == 1:
        um, up = _one_sided(_ghosts(phi, bc, 0), dx, weights, eps)
        zero = torch.zeros_like(um)
        a = torch.maximum(hp(um, zero), hp(up, zero))
        return -(h(0.5 * (um + up), zero) - 0.5 * a * (up - um)), (a.max(), torch.zeros((), dtype=a.dtype, device=a.device))
    ny, nx = phi.shape
    px, py = _ghosts(phi, bc, 1), _ghosts(phi, bc, 0)
    out, ax, ay = torch.empty_like(phi), [], []
    band = max(1, (1 << 23) // nx)
    for j in range(0, ny, band):
        k = min(ny, j + band)
        um, up = _one_sided(px[j:k], dx, weights, eps)
        vm, vp = _one_sided(py[j:k + 6].t(), dy, weights, eps)
        vm, vp = vm.t(), vp.t()
        ax.append(_max4(hp, um, up, vm, vp).max())
        ay.append(_max4(hq, um, up, vm, vp).max())
        if alpha is not None:
            out[j:k] = -(h(0.5 * (um + up), 0.5 * (vm + vp)) - 0.5 * alpha[0] * (up - um) - 0.5 * alpha[1] * (vp - vm))
    return out, (torch.stack(ax).max(), torch.stack(ay).max())


def _integrate(phi, problem, dx, dy, weights, steps, t_final, cfl=0.6):
    """RK3 steps (a number of them, or to t_final): the maxima of the stage before give alpha (2D) and dt."""
    dim, ham, _, _, bc, _ = PROBLEMS[problem]
    args = (dim, ham, bc, dx, dy, weights)
    _, alpha = _rhs(phi, None, *args)
    t, n = 0.0, 0
    while n < steps if steps else t < t_final:
        dt = cfl / (float(alpha[0]) / dx + (float(alpha[1]) / dy if dim == 2 else 0.0))
        last = not steps and t + dt >= t_final
        if last:
            dt = t_final - t
        k, a = _rhs(phi, alpha, *args)
        p1 = phi + dt * k
        k, b = _rhs(p1, a, *args)
        p2 = 0.75 * phi + 0.25 * (p1 + dt * k)
        k, alpha = _rhs(p2, b, *args)
        phi = phi / 3.0 + 2.0 * (p2 + dt * k) / 3.0
        t, n = (t_final if last else t + dt), n + 1
    return phi


def exact(case, seed):
    rng = np.random.default_rng(seed)
    if case["kind"] == "solve":
        phi0, dx, dy = _phi0(case["problem"], case["nx"], case["ny"], rng)
        unit = PROBLEMS[case["problem"]][5]
        return _integrate(phi0, case["problem"], dx, dy, case["weights"], case["steps"], case["t"] * unit)
    return [_integrate(phi0, problem, dx, dx, "arclength", 0, tf).cpu().numpy()
            for problem, _, phi0, dx, tf in _instances(case, rng)]
