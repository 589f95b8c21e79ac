"""The work that a user of this framework has it do, as cases that can be timed.

Almost everything here is one kind of call: a dynamic optimal transport solve from
two host densities to the density path, the momenta, the potential and W2^2.  The
cases take it over both precisions, two and three dimensions, with and without
obstacles, from the 32^2 x 16 grid to the 1024^2 x 32 one, on axes of every kind of
length (powers of two, multiples of four, odd).  A whole solve runs thousands of
iterations of one fixed cost; a pass here runs the first few hundred of them, with
the stopping measures and the penalty rule at the period that the case names, and
reads the results back.  Two more cases are the serving runtime (a burst of small
requests) and the allocation-free Poisson operator on device buffers.

The mixed path computes in FP32 (its multipliers in two-float), so the fields it
returns in the binding's float64 arrays are taken as FP32 tensors; the FP64 path's
are taken as they are.
"""
import math

import numpy as np
import torch

from paper_2505_05424_gb300.solver import DotServer, DotSolver, dot_poisson_f32_noalloc


def listed():
    return [
        # the smallest call: a Poisson solve inside another program's device loop that may not allocate
        dict(name="poisson64", kind="poisson", D=2, T=16, N0=64, N1=48),
        # a small interactive solve: two Gaussians, 32^2 x 16, launch-bound
        dict(name="gauss32", kind="solve", prec="mixed", D=2, T=16, N0=32, N1=32, its=200, check=10,
             data="gauss", masked=False),
        # the paper's grid (its analytic examples), checked every 5 iterations as its tables do
        dict(name="ex128", kind="solve", prec="mixed", D=2, T=32, N0=128, N1=128, its=300, check=5,
             data="gauss", masked=False),
        # transport around obstacles
        dict(name="obst128", kind="solve", prec="mixed", D=2, T=32, N0=128, N1=128, its=300, check=10,
             data="mixture", masked=True),
        # the benchmark's workload
        dict(name="mix256", kind="solve", prec="mixed", D=2, T=64, N0=256, N1=256, its=400, check=10,
             data="mixture", masked=False),
        # volumes
        dict(name="mix3d64", kind="solve", prec="mixed", D=3, T=32, N0=64, N1=64, N2=64, its=120, check=10,
             data="mixture", masked=False),
        # the largest grid the repository solves
        dict(name="mix1024", kind="solve", prec="mixed", D=2, T=32, N0=1024, N1=1024, its=240, check=10,
             data="mixture", masked=False),
        # images and volumes as they come: sides that nothing divides
        dict(name="ragged2d", kind="solve", prec="mixed", D=2, T=37, N0=150, N1=117, its=200, check=10,
             data="mixture", masked=False),
        dict(name="ragged3d", kind="solve", prec="mixed", D=3, T=20, N0=37, N1=21, N2=50, its=150, check=10,
             data="mixture", masked=False),
        # the double-precision path: the reference iteration counts on the paper's grid ...
        dict(name="fp64_ex128", kind="solve", prec="fp64", D=2, T=32, N0=128, N1=128, its=50, check=5,
             data="gauss", masked=False),
        # ... and the comparison on the benchmark's workload
        dict(name="fp64_mix256", kind="solve", prec="fp64", D=2, T=64, N0=256, N1=256, its=20, check=10,
             data="mixture", masked=False),
        # serving: a burst of small requests of two grids, every fifth with obstacles
        dict(name="serve24", kind="serve", small=16, medium=8, its=150),
    ]


def _side(rng, lo, hi):
    """An axis length: log-uniform, as often any integer as a multiple of four or a power of two."""
    v = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    how = rng.randrange(4)
    if how == 0:
        return min(hi, 1 << max(2, round(math.log2(v))))
    if how == 1:
        return max(4, round(v / 4) * 4)
    return max(3, round(v))


def draw(rng):
    pick = rng.random()
    if pick < 0.08:
        return dict(kind="poisson", D=2, T=rng.randint(4, 48), N0=_side(rng, 8, 128), N1=_side(rng, 8, 128))
    if pick < 0.16:
        return dict(kind="serve", small=rng.randint(1, 24), medium=rng.randint(0, 10), its=10 * rng.randint(10, 20))
    fp64 = rng.random() < 0.2
    if rng.random() < 0.25:
        n = _side(rng, 12, 64)
        c = dict(kind="solve", prec="fp64" if fp64 else "mixed", D=3, T=rng.randint(8, 32), N0=n,
                 N1=_side(rng, 12, 64), N2=_side(rng, 12, 64))
        its = 150
    else:
        n = _side(rng, 16, 512)
        near = max(8, n // 2), min(512, 2 * n)   # sides of one image differ by a factor of two at most
        c = dict(kind="solve", prec="fp64" if fp64 else "mixed", D=2, T=rng.randint(8, 64), N0=n,
                 N1=_side(rng, *near))
        its = 300
    if fp64:
        its = 20
        while _nodes(c) > 4_300_000:
            c["T"] //= 2
    while _nodes(c) > 9_000_000:
        c["T"] //= 2
    c.update(its=its, check=rng.choice([5, 10]), data=rng.choice(["gauss", "mixture", "mixture"]),
             masked=c["D"] == 2 and rng.random() < 0.25)
    return c


# ---- inputs -------------------------------------------------------------------------


def _sides(c):
    return [c["N%d" % d] for d in range(c["D"])]


def _nodes(c):
    return (c["T"] + 1) * math.prod(_sides(c))


def _gaussian(X, mu, sig):
    out = 1.0
    for x, m, s in zip(X, mu, sig):
        out = out * (np.exp(-0.5 * ((x - m) / s) ** 2) / (math.sqrt(2 * math.pi) * s))
    return out


def _densities(N, data, masked, rng):
    """(rho0, rho1, mask): cell samples of the kinds that the repository's workloads draw."""
    D = len(N)
    X = np.meshgrid(*[(np.arange(n) + 0.5) / n for n in N], indexing="ij", sparse=True)
    if data == "gauss":   # one Gaussian each way across the square, above a floor
        a, b = rng.uniform(0.2, 0.35, D), rng.uniform(0.65, 0.8, D)
        sig = np.full(D, rng.uniform(0.1, 0.2))
        r = [_gaussian(X, a, sig) + 1e-3, _gaussian(X, b, sig) + 1e-3]
    else:                 # mixtures: with exact zeros in 2D, above a floor in 3D
        r = []
        for _ in range(2):
            k = int(rng.integers(1, 6)) if D == 2 else int(rng.integers(2, 5))
            w = rng.dirichlet(np.ones(k))
            v = 0.0
            for j in range(k):
                sig = np.full(D, rng.uniform(0.03, 0.12)) if D == 2 else rng.uniform(0.05, 0.15, D)
                v = v + w[j] * _gaussian(X, rng.uniform(0.15, 0.85, D), sig)
            r.append(np.where(v < 1e-4, 0.0, v) if D == 2 else v + 1e-4)
    mask = None
    if masked:            # a few rectangles over about a tenth of the cells
        cells = math.prod(N)
        for _ in range(1000):
            mask = np.zeros(N, dtype=bool)
            for _ in range(int(rng.integers(3, 7))):
                e = [np.sort(rng.integers(0, n, 2)) for n in N]
                mask[tuple(slice(int(a), int(b) + 1) for a, b in e)] = True
            clear = all((v * ~mask).sum() > 0.2 * v.sum() for v in r)
            if 0.05 * cells <= mask.sum() <= 0.2 * cells and clear:
                break
        r = [np.where(mask, 0.0, v) for v in r]
    return r[0], r[1], mask


_SMALL, _MEDIUM = (16, [32, 32]), (32, [64, 64])


def _requests(c, seed):
    """[(T, N, rho0, rho1, mask)] of a burst, the two grids in turn as long as both last."""
    rng = np.random.default_rng([seed, 77])
    left, out = [c["small"], c["medium"]], []
    while sum(left):
        k = int(rng.random() < left[1] / sum(left))
        left[k] -= 1
        T, N = (_SMALL, _MEDIUM)[k]
        out.append((T, N, *_densities(N, "mixture", len(out) % 5 == 4, rng)))
    return out


def prepare(case, seed):
    c = dict(case)
    if c["kind"] == "poisson":
        g = torch.Generator().manual_seed(seed)
        b = torch.randn(_nodes(c), generator=g).cuda()
        return dict(case=c, b=b, phi=torch.empty(2 * b.numel(), dtype=torch.float32, device="cuda"))
    if c["kind"] == "serve":
        torch.cuda.init()
        return dict(case=c, reqs=_requests(c, seed), server=DotServer())
    r0, r1, mask = _densities(_sides(c), c["data"], c["masked"], np.random.default_rng([seed, 5]))
    return dict(case=c, r0=r0, r1=r1, mask=mask)


def run(state):
    c = state["case"]
    if c["kind"] == "poisson":
        dot_poisson_f32_noalloc(c["D"], c["T"], _sides(c), state["b"], state["phi"],
                                stream=torch.cuda.current_stream())
        return state["phi"]
    if c["kind"] == "serve":
        srv = state["server"]
        ids = [srv.submit(2, T, N, r0, r1, mask=m, tol=0.0, maxit=c["its"]) for T, N, r0, r1, m in state["reqs"]]
        got = []
        for i in ids:
            srv.wait(i)
            r = srv.result(i)
            srv.release(i)
            got.append((r["rho"], r["m"], r["phi"], r["objective"]))
        # one tensor of each field over the burst, in the order of the requests
        return dict(zip(("rho", "m", "phi"), (_f32(np.concatenate([g[k].ravel() for g in got])) for k in range(3))),
                    objective=torch.tensor([g[3] for g in got], dtype=torch.float32))
    with DotSolver(c["D"], c["T"], _sides(c), state["r0"], state["r1"], mask=state["mask"], prec=c["prec"],
                   check_every=c["check"]) as s:
        s.dot_solve(tol=0.0, maxit=c["its"])
        rho, m, phi, obj, _ = s.dot_get()
    if c["prec"] == "mixed":
        rho, m, phi = _f32(rho), [_f32(v) for v in m], _f32(phi)
    return dict(rho=rho, m=m, phi=phi, objective=obj)


def _f32(a):
    return torch.from_numpy(a).to(torch.float32)


# ---- what a pass cannot do without ----------------------------------------------------


def _iteration_work(D, T, N, word):
    """(bytes, flops) of one iteration of the solver: q (one word), the multipliers (8 bytes)
    and the potential read and written once; a fast transform each way along every axis and
    the projection and updates of each cone."""
    P = math.prod(N)
    nodes, cones, K = (T + 1) * P, T * P, 4 * D + 2
    faces = cones + sum((T + 1) * P // n * (n - 1) for n in N)
    log = sum(math.log2(n) for n in [T + 1, *N])
    return 2 * (word + 8) * faces + 2 * 8 * K * cones + 2 * 8 * nodes, nodes * 5.0 * log + cones * 12.0 * K


def work(case):
    c = dict(case)
    if c["kind"] == "poisson":
        n = _nodes(c)
        return {"bytes": 12.0 * n, "flops": n * 5.0 * sum(math.log2(k) for k in [c["T"] + 1, *_sides(c)])}
    if c["kind"] == "serve":
        parts = [(c[k], *_iteration_work(2, T, N, 4)) for k, (T, N) in (("small", _SMALL), ("medium", _MEDIUM))]
        return {"bytes": c["its"] * float(sum(n * b for n, b, _ in parts)),
                "flops": c["its"] * float(sum(n * f for n, _, f in parts))}
    b, f = _iteration_work(c["D"], c["T"], _sides(c), 8 if c["prec"] == "fp64" else 4)
    return {"bytes": c["its"] * float(b), "flops": c["its"] * float(f)}


# ---- the same in 64 bits with plain torch ----------------------------------------------


def _dct(n, h, dev):
    k = torch.arange(n, dtype=torch.float64, device=dev)
    C = torch.cos(math.pi * k[:, None] * (k[None, :] + 0.5) / n) * math.sqrt(2.0 / n)
    C[0] = math.sqrt(1.0 / n)
    return C, 4.0 / (h * h) * torch.sin(math.pi * k / (2 * n)) ** 2


class _Exact:
    """The inexact proximal ALM on the staggered grid in 64 bits, for a batch of problems of one
    grid: time is axis 1 of every field, space axis d is axis 2 + d."""

    def __init__(self, T, N, dev):
        self.T, self.N, self.D, self.dev = T, list(N), len(N), dev
        self.h = [1.0 / T] + [1.0 / n for n in N]
        self.C, lam = zip(*[_dct(n, h, dev) for n, h in zip([T + 1, *N], self.h)])
        tot = 0.0
        for a, l in enumerate(lam):
            tot = tot + l.reshape([-1] + [1] * (self.D - a))
        tot.view(-1)[0] = math.inf   # the zero mode -> 0
        self.lam = tot

    def poisson(self, b):
        for a, C in enumerate(self.C):
            b = torch.movedim(torch.movedim(b, 1 + a, -1) @ C.T, -1, 1 + a)
        b = b / self.lam
        for a, C in enumerate(self.C):
            b = torch.movedim(torch.movedim(b, 1 + a, -1) @ C, -1, 1 + a)
        return b

    def grad(self, v, a):
        return torch.diff(v, dim=1 + a) / self.h[a]

    def div(self, w):
        """A^* w: +w/h at the node above a face, -w/h at the node below."""
        out = 0.0
        for a, x in enumerate(w):
            pad = [0, 0] * (x.dim() - 2 - a) + [1, 1]
            out = out - torch.diff(torch.nn.functional.pad(x, pad), dim=1 + a) / self.h[a]
        return out

    def spread(self, q):
        """F q: the cone's own q_0, then per axis the faces left / right of it on its two time nodes."""
        out = [q[0]]
        for d in range(self.D):
            ax = 2 + d
            p = [0, 0] * (q[0].dim() - 1 - ax)
            lo = torch.nn.functional.pad(q[1 + d], p + [1, 0])
            hi = torch.nn.functional.pad(q[1 + d], p + [0, 1])
            out += [lo[:, :-1], hi[:, :-1], lo[:, 1:], hi[:, 1:]]
        return out

    def gather(self, u, d):
        """F^* of the components of axis d: what each of its faces collects from the cones around it."""
        ax = 2 + d
        n = self.N[d]
        u1, u2, u3, u4 = u
        now = u1.narrow(ax, 1, n - 1) + u2.narrow(ax, 0, n - 1)
        old = u3.narrow(ax, 1, n - 1) + u4.narrow(ax, 0, n - 1)
        end = [0, 0] * (now.dim() - 2)
        return torch.nn.functional.pad(now, end + [0, 1]) + torch.nn.functional.pad(old, end + [1, 0])

    def start(self, r0, r1, omega):
        """r0, r1, omega: [batch, N...]; densities of mean 1, obstacle cells of weight 1e-6."""
        B, T, N, D = r0.shape[0], self.T, self.N, self.D
        f = dict(dtype=torch.float64, device=self.dev)
        mean = lambda r: r / r.flatten(1).mean(1).reshape([-1] + [1] * D)  # noqa: E731
        self.c = torch.zeros(B, T + 1, *N, **f)
        self.c[:, 0] = mean(r0)
        self.c[:, T] -= mean(r1)
        self.cn = (mean(r0) ** 2 + mean(r1) ** 2).flatten(1).sum(1)
        shapes = [[B, T, *N]] + [[B, T + 1, *N[:d], N[d] - 1, *N[d + 1:]] for d in range(D)]
        self.q = [torch.zeros(s, **f) for s in shapes]
        self.al = [torch.zeros(s, **f) for s in shapes]
        self.K = 4 * D + 2
        self.be = [torch.zeros(B, T, *N, **f) for _ in range(self.K)]
        self.s = torch.sqrt(omega / 2)[:, None]
        s2 = (self.s ** 2).expand(B, T, *N)
        self.den = [3.0] + [1.0 + self.gather([s2] * 4, d) for d in range(D)]
        self.sigma = torch.ones(B, **f)

    def lift(self, x):
        """B F q from F q."""
        return [-x[0]] + [self.s * v for v in x[1:]] + [x[0]]

    def collect(self, u):
        """F^* B^* u."""
        return [u[-1] - u[0]] + [self.gather([self.s * v for v in u[1 + 4 * d:5 + 4 * d]], d) for d in range(self.D)]

    def iterate(self, tau):
        sg = self.sigma.reshape([-1] + [1] * (1 + self.D))
        b = self.div([q - a / sg for q, a in zip(self.q, self.al)]) - self.c / sg
        self.phi = self.poisson(b)
        d = [1.0] + [0.0] * (self.K - 2) + [1.0]
        y = [v + dk - e / sg for v, dk, e in zip(self.lift(self.spread(self.q)), d, self.be)]
        nb = torch.sqrt(sum(v * v for v in y[1:]))
        a = 0.5 * (y[0] + nb)
        inside, below = nb <= y[0], nb <= -y[0]
        scale = torch.where(inside, 1.0, torch.where(below, 0.0, a / torch.where(nb > 0, nb, 1.0)))
        z = [torch.where(inside, y[0], torch.where(below, 0.0, a))] + [scale * v for v in y[1:]]
        del y, nb, a, inside, below, scale
        u = self.collect([v - dk + e / sg for v, dk, e in zip(z, d, self.be)])
        g = [self.grad(self.phi, k) for k in range(self.D + 1)]
        self.q = [(gk + ak / sg + uk) / dk for gk, ak, uk, dk in zip(g, self.al, u, self.den)]
        self.al = [ak + tau * sg * (gk - qk) for ak, gk, qk in zip(self.al, g, self.q)]
        self.inc = [v - w - dk for v, w, dk in zip(z, self.lift(self.spread(self.q)), d)]
        self.be = [e + tau * sg * v for e, v in zip(self.be, self.inc)]

    def rule(self):
        """The penalty rule on the two second-order-cone measures."""
        vol = math.prod(self.h)
        sq = lambda x: sum((v * v).flatten(1).sum(1) for v in x)  # noqa: E731
        n2 = lambda x: torch.sqrt(vol * x)  # noqa: E731
        g = [self.grad(self.phi, k) for k in range(self.D + 1)]
        eta_p = n2(sq([a - b for a, b in zip(g, self.q)])) / (1 + n2(sq(g)) + n2(sq(self.q)))
        cones = self.T * math.prod(self.N)
        psoc = n2(sq(self.inc)) / (1 + math.sqrt(vol * 2 * cones))
        eta_d = n2(sq([self.div(self.al) + self.c])) / (1 + n2(self.cn))
        fb = self.collect(self.be)
        dsoc = n2(sq([a + b for a, b in zip(fb, self.al)])) / (1 + n2(sq(fb)) + n2(sq(self.al)))
        ratio = torch.maximum(eta_p, psoc) / torch.maximum(eta_d, dsoc)
        self.sigma = torch.where(ratio > 2, self.sigma * 1.25, torch.where(ratio < 0.5, self.sigma / 1.25, self.sigma))

    def solve(self, its, check):
        for k in range(1, its + 1):
            self.iterate(1.9)
            if k % check == 0:
                self.rule()
        obj = -2.0 * (self.c * self.phi).flatten(1).sum(1) / math.prod(self.N)
        return self.al[0] * self.T, [a * self.T for a in self.al[1:]], self.phi, obj


def _solve_exact(T, N, problems, its, check, dev):
    e = _Exact(T, N, dev)
    t = lambda a: torch.as_tensor(np.stack(a), dtype=torch.float64, device=dev)  # noqa: E731
    om = [np.ones(N) if m is None else np.where(m, 1e-6, 1.0) for _, _, m in problems]
    e.start(t([p[0] for p in problems]), t([p[1] for p in problems]), t(om))
    return e.solve(its, check)


def exact(case, seed):
    c = dict(case)
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    if c["kind"] == "poisson":
        g = torch.Generator().manual_seed(seed)
        b = torch.randn(_nodes(c), generator=g).to(dev, torch.float64)
        phi = _Exact(c["T"], _sides(c), dev).poisson(b.reshape(1, c["T"] + 1, *_sides(c))).reshape(-1)
        hi = phi.to(torch.float32).to(torch.float64)   # the call's layout: (high, low) pairs
        return torch.stack([hi, phi - hi], dim=1).reshape(-1)
    if c["kind"] == "serve":
        reqs, got = _requests(c, seed), {}
        for T, N in (_SMALL, _MEDIUM):
            at = [i for i, r in enumerate(reqs) if r[0] == T]
            if at:
                rho, m, phi, obj = _solve_exact(T, N, [reqs[i][2:] for i in at], c["its"], 10, dev)
                for j, i in enumerate(at):
                    got[i] = (rho[j].reshape(-1), torch.cat([v[j].reshape(-1) for v in m]), phi[j].reshape(-1), obj[j])
        cat = lambda k: torch.cat([got[i][k] for i in range(len(reqs))])  # noqa: E731
        return dict(rho=cat(0), m=cat(1), phi=cat(2), objective=torch.stack([got[i][3] for i in range(len(reqs))]))
    if _nodes(c) * c["its"] * max(_sides(c)) > 1.2e12:   # over about 20 seconds of 64-bit transforms
        return None
    r0, r1, mask = _densities(_sides(c), c["data"], c["masked"], np.random.default_rng([seed, 5]))
    rho, m, phi, obj = _solve_exact(c["T"], _sides(c), [(r0, r1, mask)], c["its"], c["check"], dev)
    return dict(rho=rho[0], m=[v[0] for v in m], phi=phi[0], objective=float(obj[0]))
