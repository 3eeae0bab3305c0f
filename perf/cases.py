"""The work whose speed is followed: what a user of this package has it do, through its public entry points.

A case is a dict of plain values.  `prepare` builds what a program holds before the call (host fields of the
state, the tank's or batch's handle, or device buffers), `run` is one pass: the state handed in, physical steps of
dual time stepping, the new state read back.  `exact` is the same pass in plain FP64 torch.
"""
import math

import numpy as np
import torch

from paper_2108_08769_gb300 import ac
from paper_2108_08769_gb300 import workloads as W

# --------------------------------------------------------------------------------------------- cases


def listed():
    return [
        # The smallest runs of the paper (Sec. 3.1): a one-dimensional Riemann problem in pure pseudo-time, to its
        # output pseudo-time.  Every kernel's latency counts, nothing else.
        dict(name="riemann_problem_100x1_fp64", kind="pseudo", problem=1, nx=100),
        # The Riemann tank of the tests and the benchmark: 800 cells, a few tiles.
        dict(name="riemann_tank_200x4_fp64", kind="tank", scene="riemann", form="fp64", nx=200, ny=4, iters=200, steps=1),
        # The benchmark's headline tank (water under air, closed walls), its fluids moving.
        dict(name="tank_256x256_fp64", kind="tank", scene="layers", form="fp64", nx=256, ny=256, iters=100, steps=1),
        # The same tank in the mixed form, at the stated number of pseudo-iterations of a step.
        dict(name="tank_256x256_mixed", kind="tank", scene="layers", form="mixed", nx=256, ny=256, iters=500, steps=1),
        # The collapsing water column of the configurations, both forms.
        dict(name="water_column_1024x512_fp64", kind="tank", scene="column", form="fp64", nx=1024, ny=512, iters=20,
             steps=1),
        dict(name="water_column_1024x512_mixed", kind="tank", scene="column", form="mixed", nx=1024, ny=512, iters=300,
             steps=1),
        # The largest configuration: the Rayleigh-Taylor tank, one whole physical step of 500 pseudo-iterations.
        dict(name="rayleigh_taylor_2048x8192_mixed", kind="tank", scene="rayleigh_taylor", form="mixed", nx=2048,
             ny=8192, iters=500, steps=1),
        # Many uneven tanks at once.
        dict(name="batch_24_tanks_mixed", kind="batch", count=24, nmin=64, nmax=512, iters=50),
        # A ragged grid off every tile size with the options a study of the scheme varies: second-order real-time
        # levels over two steps, the Roe flux, open and no-slip sides.
        dict(name="ragged_371x193_fp64_roe_bdf2", kind="tank", scene="wavy", form="fp64", nx=371, ny=193, iters=20,
             steps=2, riemann="roe", bdf_order=2, bc="slip,transmissive,noslip,slip"),
        # The same kind of study in the mixed form: third-order real-time levels, periodic sides.
        dict(name="ragged_389x211_mixed_bdf3", kind="tank", scene="wavy", form="mixed", nx=389, ny=211, iters=60,
             steps=3, bdf_order=3, bc="periodic,periodic,slip,slip"),
        # The stage sweep on the caller's own device buffers (callers that may not allocate).
        dict(name="stage_sweeps_600x401_fp64", kind="sweeps", scene="column", nx=600, ny=401),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["tank"] * 5 + ["batch", "sweeps", "pseudo"])
    if kind == "pseudo":
        return dict(kind="pseudo", problem=rng.randint(1, 5), nx=rng.randint(40, 400))
    if kind == "sweeps":
        return dict(kind="sweeps", scene=rng.choice(["column", "layers"]), nx=_log_int(rng, 64, 1500),
                    ny=_log_int(rng, 64, 1500))
    if kind == "batch":
        nmin = _log_int(rng, 24, 128)
        return dict(kind="batch", count=rng.randint(4, 24), nmin=nmin, nmax=rng.randint(nmin + 1, 420),
                    iters=rng.randint(10, 50))
    form = rng.choice(["fp64", "mixed"])
    hi = 900 if form == "fp64" else 1800
    nx, ny = _log_int(rng, 20, hi), _log_int(rng, 4, hi)
    # pseudo-iterations so that a pass stays far below the largest listed case
    most = 6e6 if form == "fp64" else 6e7
    iters = max(8, min(rng.randint(40, 240), int(most / (nx * ny))))
    case = dict(kind="tank", scene=rng.choice(["layers", "column", "wavy", "rayleigh_taylor"]), form=form, nx=nx, ny=ny,
                iters=iters, steps=1)
    if rng.random() < 0.3:
        case["bc"] = rng.choice(["slip,slip,slip,slip", "noslip,noslip,noslip,noslip",
                                 "slip,transmissive,noslip,slip", "periodic,periodic,slip,slip"])
    if rng.random() < 0.15:
        case["limiter_k"] = 2
    if rng.random() < 0.1:
        case["riemann"] = "roe"
    if rng.random() < 0.1:
        case["bdf_order"], case["steps"] = 2, 2
    return case


# --------------------------------------------------------------------------------------------- inputs


def _waves(seed, nx, ny, lx, ly, amplitude):
    """Smooth seeded velocities: three products of sines that vanish at the walls."""
    rng = np.random.default_rng(seed)
    x = (np.arange(nx) + 0.5) / nx
    y = (np.arange(ny) + 0.5) / ny
    u = np.zeros((ny, nx))
    v = np.zeros((ny, nx))
    for k in range(1, 4):
        a, b = rng.uniform(-amplitude, amplitude, 2)
        px, py = rng.uniform(0.0, 1.0, 2)
        u += (a / k) * np.outer(np.cos(math.pi * (k * y + py)), np.sin(math.pi * k * x))
        v += (b / k) * np.outer(np.sin(math.pi * k * y), np.cos(math.pi * (k * x + px)))
    return u, v


def _problem(case, seed):
    """The workloads.Case of one tank, its velocities seeded."""
    nx, ny = case["nx"], case["ny"]
    scene = case["scene"]
    if scene == "riemann":
        c = W.riemann_tank(nx, ny)
        amplitude = 0.05
    elif scene == "column":
        c = W.water_column(nx, ny)
        amplitude = 0.3
    elif scene == "rayleigh_taylor":
        c = W.rayleigh_taylor(nx, ny)
        amplitude = 0.1
    elif scene == "layers":
        c = W.hydrostatic_tank(ny) if nx == ny else _layers(nx, ny)
        amplitude = 0.2
    else:
        c = W.random_two_fluid(nx, ny, seed=seed, ratio=500.0, c0=10.0, velocity=0.02)
        amplitude = 0.1
    u, v = _waves(seed, nx, ny, c.lx, c.ly, amplitude)
    c.rhou += c.rho * u
    c.rhov += c.rho * v
    if "bc" in case:
        c.bc = tuple(case["bc"].split(","))
    c.options.riemann = case.get("riemann", "osher")
    c.options.bdf_order = case.get("bdf_order", 1)
    c.options.limiter_k = case.get("limiter_k", 1)
    return c


def _layers(nx, ny):
    """W.hydrostatic_tank on a grid that is not square (cells stay square)."""
    lx, ly = 1.0, ny / nx
    _, Y = W.cell_centres(nx, ny, lx, ly)
    rho = np.where(Y < 0.5 * ly, 1000.0, 1.0)
    p = W.hydrostatic_columns(rho, ly / ny, -9.81)
    z = np.zeros_like(rho)
    return W.Case(f"layers_{nx}x{ny}", nx, ny, lx, ly, 0.0, -9.81, W.beta_from_speed(20.0, 1000.0), ("slip",) * 4, rho,
                  z.copy(), z.copy(), p, dt=1e-3)


def _riemann_problem(case, seed):
    """Riemann problem `problem` with a seeded tangential velocity on either side."""
    c = W.riemann_problem(case["problem"], case["nx"])
    vl, vr = np.random.default_rng(seed).uniform(-0.5, 0.5, 2)
    c.rhov = c.rho * np.where(c.x < 0.0, vl, vr).reshape(c.rho.shape)
    return c


def _batch_problems(case, seed):
    sizes = np.random.default_rng(2108).integers(case["nmin"], case["nmax"] + 1, case["count"])
    cases = W.batched_tanks(case["count"], seed=seed, sizes=[int(n) for n in sizes])
    for k, c in enumerate(cases):
        u, v = _waves(seed + 1000 * k, c.nx, c.ny, 1.0, 1.0, 0.2)
        c.rhou += c.rho * u
        c.rhov += c.rho * v
    return cases


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        cases = _batch_problems(case, seed)
        return dict(case=case, cases=cases, states=[c.state() for c in cases], batch=ac.Batch(cases))
    if kind == "sweeps":
        c = _problem(case, seed)
        dev = torch.device("cuda", 0)
        q0 = [torch.from_numpy(a.reshape(-1)).to(dev) for a in c.state()]
        out = [[torch.empty_like(x) for x in q0] for _ in range(c.options.s_max)]
        return dict(case=case, c=c, q0=q0, qn=[x.clone() for x in q0[:3]], out=out, options=ac.options_from(c.options),
                    norms=torch.zeros(4, dtype=torch.float64, device=dev))
    c = _riemann_problem(case, seed) if kind == "pseudo" else _problem(case, seed)
    form = case.get("form", "fp64")
    tank = ac.Tank(c.nx, c.ny, c.lx, c.ly, c.gx, c.gy, c.beta, c.bc, ac.options_from(c.options, form))
    return dict(case=case, c=c, fields=c.state(), tank=tank)


# --------------------------------------------------------------------------------------------- passes

FIELDS = ("rho", "rhou", "rhov", "p")


def _kept(form, fields):
    # the mixed form computes in single precision: its results are kept in it
    if form == "mixed":
        fields = [f.astype(np.float32) for f in fields]
    return dict(zip(FIELDS, fields))


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "sweeps":
        c = state["c"]
        stream = torch.cuda.current_stream().cuda_stream
        q0 = [x.data_ptr() for x in state["q0"]]
        qn = [x.data_ptr() for x in state["qn"]]
        prev = None
        for stage, out in enumerate(state["out"], start=1):
            ptr = [x.data_ptr() for x in out]
            ac.ac_stage_sweep_noalloc(c.nx, c.ny, c.lx, c.ly, c.gx, c.gy, c.beta, c.bc, state["options"], stage, c.dt,
                                      prev, q0, qn, ptr, state["norms"].data_ptr() if stage == 1 else 0, stream)
            prev = ptr
        return dict(zip(FIELDS, state["out"][-1]), norms=state["norms"])
    if kind == "batch":
        b, cases = state["batch"], state["cases"]
        for k, s in enumerate(state["states"]):
            b.set_state(k, *s)
        _, iters, _ = b.physical_step([c.dt for c in cases], -1.0, case["iters"])
        out = [np.concatenate(f, axis=None) for f in zip(*(b.get_state(k) for k in range(len(cases))))]
        return dict(_kept("mixed", out), iters=np.array(iters))
    tank, c = state["tank"], state["c"]
    tank.set_state(*state["fields"])
    if kind == "pseudo":
        _, iters = tank.pseudo_time_run(c.tau_end)
        return dict(_kept("fp64", tank.get_state()), iters=iters)
    for _ in range(case["steps"]):
        _, iters = tank.physical_step(c.dt, -1.0, case["iters"])
    return dict(_kept(case["form"], tank.get_state()), iters=iters)


# --------------------------------------------------------------------------------------------- work


def work(case):
    """Operations of the method per cell and Runge-Kutta stage (483 in FP64 with the Osher flux, the mixed form's about
    420 counted the same way), three stages to a pseudo-iteration; the state in and out once as FP64 fields."""
    if case["kind"] == "pseudo":
        cells, stages = case["nx"], 3 * case["nx"] // 2
    elif case["kind"] == "batch":
        sizes = np.random.default_rng(2108).integers(case["nmin"], case["nmax"] + 1, case["count"])
        cells, stages = int((sizes.astype(np.int64) ** 2).sum()), 3 * case["iters"]
    elif case["kind"] == "sweeps":
        cells, stages = case["nx"] * case["ny"], 3
    else:
        cells, stages = case["nx"] * case["ny"], 3 * case["iters"] * case["steps"]
    mixed = case["kind"] == "batch" or case.get("form") == "mixed"
    return dict(bytes=64.0 * cells + (24.0 * cells if case["kind"] == "sweeps" else 0.0),
                flops=(420.0 if mixed else 483.0) * cells * stages)


# --------------------------------------------------------------------------------------------- exact values


class _Exact:
    """The scheme (arXiv 2108.08769) on whole arrays in FP64: ghost-padded fields, every operation of the paper in its
    own order, |A| dQ in eigenvector form."""

    BDF = {1: (1.0, -1.0, 0.0, 0.0), 2: (1.5, -2.0, 0.5, 0.0), 3: (11.0 / 6.0, -3.0, 1.5, -1.0 / 3.0)}
    NODES = ((0.5 - math.sqrt(0.15), 5.0 / 18.0), (0.5, 8.0 / 18.0), (0.5 + math.sqrt(0.15), 5.0 / 18.0))

    def __init__(self, c):
        self.c, self.o = c, c.options
        self.dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
        self.ix, sx, tx, gx = self._axis(c.nx, c.bc[0], c.bc[1])
        self.iy, sy, ty, gy = self._axis(c.ny, c.bc[2], c.bc[3])
        # signs of (rho u, rho v) of the padded cells: a wall flips the normal momentum, no-slip the tangential too
        self.su = sx[None, :] * ty[:, None]
        self.sv = sy[:, None] * tx[None, :]
        self.sg = torch.where(gx[None, :] | gy[:, None], -1.0, 1.0).to(self.dev, torch.float64)

    def _axis(self, n, lo, hi):
        src, flip, tang, wall = [], [], [], []
        for i in range(-2, n + 2):
            f, t = 1.0, 1.0
            outside = lo if i < 0 else hi if i >= n else None
            while i < 0 or i >= n:
                kind = lo if i < 0 else hi
                if kind == "periodic":
                    i += n if i < 0 else -n
                elif kind == "transmissive":
                    i = 0 if i < 0 else n - 1
                else:
                    i = -1 - i if i < 0 else 2 * n - 1 - i
                    f = -f
                    t = -t if kind == "noslip" else t
            src.append(i), flip.append(f), tang.append(t), wall.append(outside in ("slip", "noslip"))
        f64 = dict(dtype=torch.float64, device=self.dev)
        return (torch.tensor(src, device=self.dev), torch.tensor(flip, **f64), torch.tensor(tang, **f64),
                torch.tensor(wall, device=self.dev))

    def pad(self, a, sign=None):
        a = a[self.iy][:, self.ix]
        return a if sign is None else a * sign

    @staticmethod
    def limit(a, b, k):
        s = torch.sign(b)
        m = torch.maximum(torch.minimum(k * b.abs(), s * a), torch.minimum(b.abs(), k * s * a))
        return s * torch.clamp(m, min=0.0)

    def flux(self, L, R):
        """Flux in the face-normal frame; L, R = (rho, un, ut, p)."""
        beta = self.c.beta
        (rL, uL, vL, pL), (rR, uR, vR, pR) = L, R
        QL, QR = (rL, rL * uL, rL * vL, pL / beta), (rR, rR * uR, rR * vR, pR / beta)
        dr, dm, dn, dq = (b - a for a, b in zip(QL, QR))
        D = [0.0, 0.0, 0.0, 0.0]
        if self.o.riemann == "roe":
            wl, wr = torch.sqrt(rL), torch.sqrt(rR)
            points = [(1.0, wl * wr, (wl * uL + wr * uR) / (wl + wr), (wl * vL + wr * vR) / (wl + wr))]
        else:
            points = []
            for t, w in self.NODES:
                r = QL[0] + t * dr
                points.append((w, r, (QL[1] + t * dm) / r, (QL[2] + t * dn) / r))
        for w, r, u, v in points:
            c = torch.sqrt(u * u + 4.0 * beta / r)
            l4, l5 = 0.5 * (u + c), 0.5 * (u - c)
            a = (dm - u * dr) / beta
            s4, s5 = (r / c) * (l4 * a + dq), -(r / c) * (l5 * a + dq)
            f4, f5 = (l4.abs() - u.abs()) * s4, (l5.abs() - u.abs()) * s5
            # acoustic right eigenvectors (l4, u l4 + beta/rho, v l4, -l5/rho) and the same with l4, l5 exchanged
            for k, (x, r4, r5) in enumerate(((dr, l4, l5), (dm, u * l4 + beta / r, u * l5 + beta / r),
                                             (dn, v * l4, v * l5), (dq, -l5 / r, -l4 / r))):
                D[k] = D[k] + w * (u.abs() * x + f4 * r4 + f5 * r5)
        FL, FR = (QL[1], QL[1] * uL + pL, QL[1] * vL, uL), (QR[1], QR[1] * uR + pR, QR[1] * vR, uR)
        return [0.5 * (a + b - d) for a, b, d in zip(FL, FR, D)]

    def bracket(self, Q, rt, rho_m):
        """The bracket of Eq. RK2 at stage state Q; real-time terms and body force stay those of Q^m."""
        c, dx, dy = self.c, self.c.dx, self.c.dy
        rho = self.pad(Q[0])
        u, v, p = self.pad(Q[1], self.su) / rho, self.pad(Q[2], self.sv) / rho, self.pad(Q[3])
        ring = (slice(1, -1), slice(1, -1))
        k = float(self.o.limiter_k)

        def slopes(a, kk):
            m = a[ring]
            return (self.limit(a[1:-1, 2:] - m, m - a[1:-1, :-2], kk), self.limit(a[2:, 1:-1] - m, m - a[:-2, 1:-1], kk))

        (rx, ry), (ux, uy), (vx, vy) = slopes(rho, k), slopes(u, k), slopes(v, k)
        r, U, V, P, sg = rho[ring], u[ring], v[ring], p[ring], self.sg[ring]
        if self.o.gradp == "new":
            tu, tv = self.pad(rt[1], self.su)[ring], self.pad(rt[2], self.sv)[ring]
            gx = (-tu - (U * U * rx + 2.0 * r * U * ux) / dx - (U * V * ry + r * U * vy + r * V * uy) / dy + r * c.gx * sg)
            gy = (-tv - (V * V * ry + 2.0 * r * V * vy) / dy - (U * V * rx + r * V * ux + r * U * vx) / dx + r * c.gy * sg)
            px, py = gx * dx, gy * dy
        else:
            px, py = slopes(p, 1.0)
        W = (r, U, V, P)
        lo = [a[1:-1, :-1] + 0.5 * s[1:-1, :-1] for a, s in zip(W, (rx, ux, vx, px))]
        hi = [a[1:-1, 1:] - 0.5 * s[1:-1, 1:] for a, s in zip(W, (rx, ux, vx, px))]
        F = self.flux(lo, hi)
        lo = [a[:-1, 1:-1] + 0.5 * s[:-1, 1:-1] for a, s in zip(W, (ry, uy, vy, py))]
        hi = [a[1:, 1:-1] - 0.5 * s[1:, 1:-1] for a, s in zip(W, (ry, uy, vy, py))]
        G = self.flux([lo[0], lo[2], lo[1], lo[3]], [hi[0], hi[2], hi[1], hi[3]])
        G = [G[0], G[2], G[1], G[3]]
        b = [-(f[:, 1:] - f[:, :-1]) / dx - (g[1:] - g[:-1]) / dy for f, g in zip(F, G)]
        b[0] = b[0] - rt[0]
        b[1] = b[1] - rt[1] + rho_m * c.gx
        b[2] = b[2] - rt[2] + rho_m * c.gy
        return b

    def local_dtau(self, Q):
        c = self.c
        u, v, f = Q[1] / Q[0], Q[2] / Q[0], 4.0 * c.beta / Q[0]
        den = 0.5 * (u.abs() + torch.sqrt(u * u + f)) * c.dy + 0.5 * (v.abs() + torch.sqrt(v * v + f)) * c.dx
        return self.o.cfl_tau * c.dx * c.dy / den

    def iteration(self, Qm, rt, B0dt, dtau):
        """One pseudo-iteration from Q^m: the new state and the RMS of the first stage's bracket."""
        Q, norms = Qm, None
        for s in range(1, self.o.s_max + 1):
            alpha = 1.0 / (self.o.s_max - s + 1)
            b = self.bracket(Q, rt, Qm[0])
            if s == 1:
                norms = [torch.sqrt((x * x).mean()) for x in b[:3]] + [self.c.beta * torch.sqrt((b[3] * b[3]).mean())]
            k = alpha * dtau / (1.0 + B0dt * alpha * dtau)
            Q = [Qm[0] + k * b[0], Qm[1] + k * b[1], Qm[2] + k * b[2], Qm[3] + self.c.beta * k * b[3]]
        return Q, torch.stack(norms)

    def tensors(self, fields):
        return [torch.tensor(a, dtype=torch.float64, device=self.dev) for a in fields]

    def steps(self, fields, dt, iters, steps):
        Q, levels, norms = self.tensors(fields), [], None
        for n in range(steps):
            levels = [Q[:3]] + levels[:2]
            B = self.BDF[min(self.o.bdf_order, n + 1)]
            for _ in range(iters):
                rt = [(B[0] * Q[f] + sum(b * lev[f] for b, lev in zip(B[1:], levels))) / dt for f in range(3)]
                Q, norms = self.iteration(Q, rt, B[0] / dt, self.local_dtau(Q))
        return Q, norms

    def pseudo(self, fields, tau_end):
        Q, tau, iters = self.tensors(fields), 0.0, 0
        zero = [torch.zeros_like(Q[0])] * 3
        while tau < tau_end:
            dtau = min(float(self.local_dtau(Q).min()), tau_end - tau)
            Q, _ = self.iteration(Q, zero, 0.0, dtau)
            tau += dtau
            iters += 1
        return Q, iters


def exact(case, seed):
    kind = case["kind"]
    if kind == "tank" and case["nx"] * case["ny"] * case["iters"] * case["steps"] > 4e8:
        return None
    if kind == "batch":
        cases = _batch_problems(case, seed)
        out = [_Exact(c).steps(c.state(), c.dt, case["iters"], 1)[0] for c in cases]
        return dict(zip(FIELDS, [np.concatenate([a.cpu().numpy() for a in f], axis=None) for f in zip(*out)]))
    c = _riemann_problem(case, seed) if kind == "pseudo" else _problem(case, seed)
    e = _Exact(c)
    if kind == "pseudo":
        Q, iters = e.pseudo(c.state(), c.tau_end)
        return dict(zip(FIELDS, [a.cpu().numpy() for a in Q]))
    if kind == "sweeps":
        Q, norms = e.steps(c.state(), c.dt, 1, 1)
        return dict(zip(FIELDS, [a.reshape(-1) for a in Q]), norms=norms)
    Q, _ = e.steps(c.state(), c.dt, case["iters"], case["steps"])
    return dict(zip(FIELDS, [a.cpu().numpy() for a in Q]))
