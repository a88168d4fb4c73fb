"""What a user of this package has it compute, as sized cases that can be timed and checked.

Every case is a dict of plain values.  `prepare` builds what a user's program holds before the call
(orbit, plan, strain, data; all from the seed), `run` makes one pass through the package's public entry
points, `work` counts the bytes and operations the path cannot do without, and `exact` evaluates the same
outputs in plain 64-bit torch, without this package.  Sizes and orders are those of this repository's
workloads: dt = 10 s, lengths from a few thousand samples to one year (3 153 600), ragged batches of
2^16 to 2^20 samples per source, Lagrange orders up to 41, Galactic binaries of 0.1 to 10 mHz.
"""
import math

import numpy as np
import torch

import paper_2204_06633_gb300 as lr

DT = 10.0
YEAR_N = 3153600
C = 299792458.0
AU = 149597870700.0
YEAR = 31557600.0
ARM = 2.5e9
MARGIN = 96            # input samples beyond the output span on each side
SIGMA = 1e-21          # noise of the data, per channel
ORDERS = (7, 11, 15, 19, 25, 31, 41)


def listed():
    return [
        # a short stretch of one source, as in a quick look or the inner step of a sampler: latency
        dict(name="short_mixed", kind="response", precision="mixed", order=25, n=4096, orbit="flexing"),
        # the plain method workload: one source on the static triangle, the default precision
        dict(name="config1_fp64", kind="response", precision="fp64", order=25, n=65536, orbit="static"),
        # one year of data in the default precision: the size that response times are quoted on
        dict(name="year_fp64", kind="response", precision="fp64", order=25, n=YEAR_N, orbit="flexing"),
        # the same year in the fast precision
        dict(name="year_mixed", kind="response", precision="mixed", order=25, n=YEAR_N, orbit="flexing"),
        # a small ragged batch in the default precision, as a check of a template bank
        dict(name="batch_fp64", kind="batch", precision="fp64", order=25, sources=6, lo=1 << 16, hi=1 << 18, mix=3,
             orbit="flexing"),
        # the batched workload of the benchmark, with fewer sources of the same lengths
        dict(name="batch_mixed", kind="batch", precision="mixed", order=25, sources=48, lo=1 << 16, hi=1 << 20, mix=3,
             orbit="flexing"),
        # link series and first-generation TDI asked for one after the other (instrument studies): odd
        # length, low order, flexing projection with an equal-arm TDI
        dict(name="split_fp64", kind="split", precision="fp64", order=11, n=200003, orbit="hybrid", generation=1),
        # the likelihood of a set of proposals against their data
        dict(name="like_mixed", kind="like", precision="mixed", order=25, sources=24, lo=1 << 16, hi=1 << 20, mix=3,
             orbit="flexing"),
        # the same with the waveform generated on the device from the binaries' parameters
        dict(name="gb_like_mixed", kind="gb_like", precision="mixed", order=25, sources=24, lo=1 << 16, hi=1 << 20, mix=3,
             orbit="flexing"),
        # a gradient step of a parameter fit: differentiable log-likelihood, forward and backward
        dict(name="grad_fp64", kind="grad", precision="fp64", order=25, n=65536, orbit="static"),
        # the adjoint of one year at the highest order, as in the batched differentiation workload
        dict(name="adjoint_year_mixed", kind="adjoint", precision="mixed", order=41, n=YEAR_N, orbit="flexing"),
        # a batch whose series live in (pinned) host memory, copies included
        dict(name="host_mixed", kind="host", precision="mixed", order=25, sources=8, lo=1 << 16, hi=1 << 20, mix=3,
             orbit="flexing"),
    ]


def draw(rng):
    def size(a, b):
        return int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))

    kind = rng.choice(["response", "response", "response", "batch", "batch", "split", "like", "gb_like", "grad", "adjoint", "host"])
    precision = {"like": "mixed", "gb_like": "mixed", "host": "mixed", "split": "fp64"}.get(kind) or rng.choice(["fp64", "mixed"])
    case = dict(kind=kind, precision=precision, order=rng.choice(ORDERS), orbit=rng.choice(["flexing", "flexing", "static", "hybrid"]))
    fp64 = precision == "fp64"
    if kind in ("batch", "like", "gb_like", "host"):
        case.update(sources=size(2, 8 if fp64 or kind == "host" else 32), lo=1 << 16, hi=1 << (18 if fp64 else 20),
                    mix=rng.randrange(1 << 16))
    elif kind in ("grad", "adjoint"):
        case.update(n=size(4096, (1 << 17) if fp64 else (1 << 20)))
    else:
        case.update(n=size(4096, (1 << 20) if fp64 else YEAR_N))
        if kind == "split":
            case["generation"] = rng.choice([1, 2])
    return case


# ------------------------------------------------------------------ inputs
def _lengths(case):
    if "n" in case:
        return [int(case["n"])]
    r = np.random.default_rng(case["mix"])
    return [int(v) for v in r.integers(case["lo"], case["hi"] + 1, size=case["sources"])]


def _sources(case, seed):
    """Binaries: f log-uniform 0.1-10 mHz (3 mHz +- 10 % where a gradient is taken), isotropic sky."""
    r = np.random.default_rng([int(seed), 2])
    S = len(_lengths(case))
    f = np.exp(r.uniform(np.log(1e-4), np.log(1e-2), S))
    if case["kind"] in ("grad", "adjoint"):
        f = 3e-3 * r.uniform(0.9, 1.1, S)
    ci = r.uniform(-1.0, 1.0, S)
    sky = np.stack([r.uniform(0.0, 2 * np.pi, S), np.arcsin(r.uniform(-0.95, 0.95, S)), r.uniform(0.0, np.pi, S)], 1)
    fdot = np.full(S, 1e-17)
    gb = np.stack([np.full(S, 1e-22), f, fdot, 11.0 * fdot ** 2 / (3.0 * f), r.uniform(0.0, 2 * np.pi, S), np.arccos(ci)], 1)
    return gb, sky


def _knots(n):
    """Knots every 1e5 s over the outputs and the reads around them."""
    k1 = int(math.ceil((n * DT + 3e5) / 1e5)) + 2
    return 1e5 * np.arange(-5, k1 + 1, dtype=np.float64)


def _positions(kind, tk):
    if kind == "static":
        a1, a2 = np.array([0.0, 1.0, 0.0]), np.array([-0.5, 0.0, -math.sqrt(0.75)])
        x = np.empty((3, 3, len(tk)))
        for i in range(3):
            ph = -2.0 * np.pi * i / 3.0
            x[i] = (np.array([AU, 0.0, 0.0]) + ARM / math.sqrt(3.0) * (math.cos(ph) * a1 + math.sin(ph) * a2))[:, None]
        return x
    e, al = ARM / (2.0 * math.sqrt(3.0) * AU), 2.0 * np.pi * tk / YEAR
    x = np.empty((3, 3, len(tk)))
    for i in range(3):
        b = -2.0 * np.pi * i / 3.0
        x[i, 0] = AU * np.cos(al) + 0.5 * e * AU * (np.cos(2 * al - b) - 3 * math.cos(b))
        x[i, 1] = AU * np.sin(al) + 0.5 * e * AU * (np.sin(2 * al - b) - 3 * math.sin(b))
        x[i, 2] = -math.sqrt(3.0) * e * AU * np.cos(al - b)
    centre = x.mean(axis=0)
    for i, (a, ph) in enumerate(((0.0141, 0.3), (-0.0113, 2.1), (0.0085, 4.4))):
        x[i] = centre + (x[i] - centre) * (1.0 + a * np.sin(2 * np.pi * tk / YEAR + ph))
    return x


def _orbits(case, n):
    """(knots, positions, projection delays or None, TDI delays or None)"""
    tk = _knots(n)
    const = np.full((6, len(tk)), ARM / C)
    proj = const if case["orbit"] == "static" else None
    tdi = None if case["orbit"] == "flexing" else const
    return tk, _positions(case["orbit"], tk), proj, tdi


def _strain(gb, n, device):
    """h+, hx of one binary on the input grid -MARGIN .. n + MARGIN."""
    A, f0, fdot, fddot, phi0, iota = (float(v) for v in gb)
    i = torch.arange(-MARGIN, n + MARGIN, dtype=torch.float64, device=device)
    t = i * DT
    hi = float(np.float64(np.float32(f0)))              # f0 t in cycles, modulo one without rounding
    cyc = torch.remainder(hi * t, 1.0) + (f0 - hi) * t + (0.5 * fdot * t + fddot / 6.0 * t * t) * t
    ph = 2.0 * math.pi * torch.remainder(cyc, 1.0) + phi0
    ci = math.cos(iota)
    return A * (1.0 + ci * ci) * torch.cos(ph), 2.0 * A * ci * torch.sin(ph)


def _noise(case, seed, count, device, scale):
    g = torch.Generator(device=device)
    g.manual_seed(int(seed) * 7919 + 13)
    return scale * torch.randn(count, dtype=torch.float64, device=device, generator=g)


def _offsets(lengths, extra=0):
    return np.concatenate([[0], np.cumsum(np.asarray(lengths, dtype=np.int64) + extra)]).astype(np.int64)


def _plan(case, n):
    ctx = lr.Context(0)
    tk, pos, pd, td = _orbits(case, n)
    po = lr.Orbit(ctx, tk, pos, pd)
    to = po if case["orbit"] != "hybrid" else lr.Orbit(ctx, tk, pos, td)
    return lr.Plan(ctx, case["order"], n, DT, po, to, t0=0.0, precision=lr.MIXED if case["precision"] == "mixed" else lr.FP64,
                   generation=case.get("generation", 2))


def prepare(case, seed):
    dev = torch.device("cuda", 0)
    kind, lengths = case["kind"], _lengths(case)
    gb, sky = _sources(case, seed)
    n = max(lengths)
    s = dict(kind=kind, plan=_plan(case, n), t0h=-MARGIN * DT, weights=(1.0 / SIGMA ** 2,) * 3)
    if "n" in case:
        s["hp"], s["hc"] = _strain(gb[0], n, dev)
        s["sky"] = tuple(float(v) for v in sky[0])
        if kind == "grad":
            s["data"] = _noise(case, seed, 3 * n, dev, SIGMA).reshape(3, n)
            s["hp"].requires_grad_(True)
            s["hc"].requires_grad_(True)
            s["sky"] = torch.tensor(s["sky"], dtype=torch.float64, requires_grad=True)
        elif kind == "adjoint":
            s["g"] = _noise(case, seed, 3 * n, dev, 1.0).reshape(3, n)
            s["out"] = (torch.empty_like(s["hp"]), torch.empty_like(s["hc"]), torch.empty(3, dtype=torch.float64, device=dev))
        elif kind == "split":
            s["y"] = torch.empty((6, n), dtype=torch.float64, device=dev)
            s["xyz"] = torch.empty((3, n), dtype=torch.float64, device=dev)
        else:
            s["xyz"] = torch.empty((3, n), dtype=torch.float64, device=dev)
        return s
    S, total = len(lengths), int(sum(lengths))
    oo, ho, t0h = _offsets(lengths), _offsets(lengths, 2 * MARGIN), np.full(S, -MARGIN * DT)
    if kind == "gb_like":
        s["gb"] = torch.tensor(gb, device=dev).reshape(-1)
    else:
        parts = [_strain(gb[i], lengths[i], dev) for i in range(S)]
        s["hp"], s["hc"] = torch.cat([p[0] for p in parts]), torch.cat([p[1] for p in parts])
    if kind == "host":
        s["hp"], s["hc"] = s["hp"].cpu().pin_memory(), s["hc"].cpu().pin_memory()
        s.update(h_off=ho, out_off=oo, t0h=t0h, sky=sky, xyz=torch.empty(3 * total, dtype=torch.float64).pin_memory())
        return s
    s.update(h_off=torch.tensor(ho, device=dev), out_off=torch.tensor(oo, device=dev), t0h=torch.tensor(t0h, device=dev),
             sky=torch.tensor(sky, device=dev).reshape(-1))
    if kind == "batch":
        s["xyz"] = torch.empty(3 * total, dtype=torch.float64, device=dev)
    else:
        s["data"] = _noise(case, seed, 3 * total, dev, SIGMA)
        s["logl"] = torch.empty(S, dtype=torch.float64, device=dev)
    return s


def run(s):
    kind, plan = s["kind"], s["plan"]
    if kind == "response":
        return plan.response(s["hp"], s["hc"], s["t0h"], s["sky"], xyz=s["xyz"])
    if kind == "split":
        y = plan.project(s["hp"], s["hc"], s["t0h"], s["sky"], y=s["y"])
        return y, plan.tdi(y, xyz=s["xyz"])
    if kind == "batch":
        return plan.response_batched(s["h_off"], s["out_off"], s["t0h"], s["sky"], s["hp"], s["hc"], xyz=s["xyz"])
    if kind == "like":
        return plan.log_likelihood_batched(s["h_off"], s["out_off"], s["t0h"], s["sky"], s["hp"], s["hc"], s["data"],
                                           s["weights"], out=s["logl"])
    if kind == "gb_like":
        return plan.log_likelihood_gb_batched(s["out_off"], s["gb"], s["sky"], s["data"], s["weights"], out=s["logl"])
    if kind == "grad":
        logl = lr.log_likelihood(plan, s["hp"], s["hc"], s["sky"], s["t0h"], s["data"], s["weights"])
        g = torch.autograd.grad(logl, (s["hp"], s["hc"], s["sky"]))
        return (logl.detach(),) + g
    if kind == "adjoint":
        a, b, c = s["out"]
        return plan.backward(s["hp"], s["hc"], s["t0h"], s["sky"], s["g"], a, b, c)
    return torch.as_tensor(plan.response_batched_host(s["h_off"], s["out_off"], s["t0h"], s["sky"], s["hp"], s["hc"], xyz=s["xyz"]))


def work(case):
    """Per output sample at T = order + 1 taps: 60 T tap multiply-adds (9 projection reads of two
    polarisations, 42 delayed link reads) and 51 sets of Lagrange weights of 3 T operations; each input
    read once, each output written once.  A gradient does the transposed reads and the reads' derivatives."""
    T = case["order"] + 1
    n = case["n"] if "n" in case else case["sources"] * (case["lo"] + case["hi"]) / 2.0
    reads = 42 if case.get("generation", 2) == 2 else 18
    proj, tdi = 9 * (4 + 3) * T + 500, reads * (2 + 3) * T
    kind = case["kind"]
    byt = {"split": 16 + 48 + 48 + 24, "like": 16 + 24, "gb_like": 24, "grad": 16 + 24 + 16, "adjoint": 16 + 24 + 16}.get(kind, 40)
    flops = {"grad": 2 * (proj + tdi) + 2 * proj, "adjoint": proj + tdi + 2 * proj}.get(kind, proj + tdi)
    return {"bytes": float(byt) * n, "flops": float(flops) * n}


# ------------------------------------------------------------------ plain 64-bit evaluation
RECV, EMIT = (0, 1, 2, 0, 2, 1), (1, 2, 0, 2, 1, 0)     # links 12, 23, 31, 13, 32, 21
CHUNK = 1 << 18


class _Spline:
    """Not-a-knot cubic splines of the rows of v on uniform knots."""

    def __init__(self, tk, v, device):
        n, dk = len(tk), (tk[-1] - tk[0]) / (len(tk) - 1)
        A, rhs = np.zeros((n, n)), np.zeros((n, len(v)))
        A[0, :3], A[-1, -3:] = (1.0, -2.0, 1.0), (1.0, -2.0, 1.0)
        for k in range(1, n - 1):
            A[k, k - 1:k + 2] = (1.0, 4.0, 1.0)
            rhs[k] = 6.0 * (v[:, k + 1] - 2.0 * v[:, k] + v[:, k - 1])
        M = np.linalg.solve(A, rhs).T                     # second derivatives times dk^2
        b = v[:, 1:] - v[:, :-1] - (2.0 * M[:, :-1] + M[:, 1:]) / 6.0
        co = np.stack([v[:, :-1], b, M[:, :-1] / 2.0, (M[:, 1:] - M[:, :-1]) / 6.0])
        self.t0, self.dk, self.n, self.c = float(tk[0]), float(dk), n, torch.tensor(co, device=device)

    def __call__(self, t):
        u = (t - self.t0) / self.dk
        k = torch.clamp(torch.floor(u).to(torch.int64), 0, self.n - 2)
        x = u - k
        a, b, c, d = (self.c[i][:, k] for i in range(4))
        return a + x * (b + x * (c + x * d))


def _light_times(tk, pos, device):
    P = _Spline(tk, pos.reshape(9, -1), device)
    t = torch.tensor(tk, device=device)
    x = P(t)
    L = torch.empty((6, len(tk)), dtype=torch.float64, device=device)
    for l in range(6):
        r = x[3 * RECV[l]:3 * RECV[l] + 3]
        v = torch.linalg.norm(r - x[3 * EMIT[l]:3 * EMIT[l] + 3], dim=0) / C
        for _ in range(20):
            v = torch.linalg.norm(r - P(t - v)[3 * EMIT[l]:3 * EMIT[l] + 3], dim=0) / C
        L[l] = v
    return L.cpu().numpy()


def _weights(eps, T):
    """Lagrange weights of the nodes -h .. h + 1 at eps, as a list of T tensors."""
    h = (T - 2) // 2
    left, right = [torch.ones_like(eps)], [torch.ones_like(eps)]
    for a in range(T - 1):
        left.append(left[-1] * (eps + (h - a)) / (a + 1))
        right.append(right[-1] * (eps + (h - (T - 1 - a))) / (a + 1))
    return [left[a] * right[T - 1 - a] * (-1.0 if (T - 1 - a) % 2 else 1.0) for a in range(T)]


def _split(u):
    fl = torch.floor(u)
    return fl.to(torch.int64), u - fl


def _chains(generation):
    q = 3 if generation == 1 else 7
    link = {(RECV[l], EMIT[l]): l for l in range(6)}
    out = []
    for ch in range(3):
        for sign, seq in ((1.0, (1, 3, 1, 2, 1, 2, 1, 3, 1)), (-1.0, (1, 2, 1, 3, 1, 3, 1, 2, 1))):
            s = [(v - 1 + ch) % 3 for v in seq]
            out.append((ch, sign, [link[(s[i], s[i + 1])] for i in range(q + 1)]))
    return out


class _Plain:
    """The response of one source and its transpose, in chunks of output samples."""

    def __init__(self, case, n, device):
        tk, pos, pd, td = _orbits(case, n)
        self.n, self.T, self.dev = n, case["order"] + 1, device
        solved = _light_times(tk, pos, device) if pd is None or td is None else None
        self.pos = _Spline(tk, pos.reshape(9, -1), device)
        self.pd = _Spline(tk, solved if pd is None else pd, device)
        self.td = _Spline(tk, solved if td is None else td, device)
        self.chains = _chains(case.get("generation", 2))

    def reach(self):
        return 2 * self.T + 24

    def read(self, h, first, u, pad):
        """h at first + i + u[i] (i = 0 .. len(u) - 1), h zero outside; pad: zeros on both sides."""
        m, eps = _split(u)
        base = m + torch.arange(len(u), device=self.dev) + first - (self.T - 2) // 2 + pad
        out = 0.0
        for j, w in enumerate(_weights(eps, self.T)):
            out = out + w * h[base + j]
        return out

    def project(self, hp, hc, sky, k0, k1):
        """y[6] at k0 .. k1 - 1 from the strain padded by `pad` zeros; differentiable in hp, hc and sky."""
        lam, beta, psi = sky[0], sky[1], sky[2]
        sl, cl, sb, cb = torch.sin(lam), torch.cos(lam), torch.sin(beta), torch.cos(beta)
        z = torch.zeros_like(sl)
        kv, uv, vv = torch.stack([-cb * cl, -cb * sl, -sb]), torch.stack([sl, -cl, z]), torch.stack([-sb * cl, -sb * sl, cb])
        c2, s2 = torch.cos(2 * psi), torch.sin(2 * psi)
        t = torch.arange(k0, k1, dtype=torch.float64, device=self.dev) * DT
        x, L = self.pos(t).reshape(3, 3, -1), self.pd(t)
        pad = MARGIN + 64
        sig = [(kv[:, None] * x[i]).sum(0) / C / DT for i in range(3)]
        at = lambda shift: [self.read(h, k0 - self.h0, MARGIN - shift, pad) for h in (hp, hc)]  # noqa: E731
        rec = [at(sig[i]) for i in range(3)]
        y = []
        for l in range(6):
            r, e = RECV[l], EMIT[l]
            d = x[r] - x[e]
            d = d / torch.linalg.norm(d, dim=0)
            un, vn, kn = ((w[:, None] * d).sum(0) for w in (uv, vv, kv))
            p, c = un * un - vn * vn, 2.0 * un * vn
            p, c = c2 * p + s2 * c, c2 * c - s2 * p
            em = at(L[l] / DT + sig[e])
            y.append((p * (em[0] - rec[r][0]) + c * (em[1] - rec[r][1])) / (2.0 * (1.0 - kn)))
        return torch.stack(y)

    h0 = 0

    def terms(self, k0, k1):
        """(channel, sign, link, delay in samples or None) of every read of the outputs k0 .. k1 - 1."""
        L = self.td(torch.arange(k0, k1, dtype=torch.float64, device=self.dev) * DT) / DT
        for ch, sign, links in self.chains:
            D = None
            for i, l in enumerate(links):
                yield ch, sign, l, D
                D = L[l] if D is None else D + L[l]

    def tdi(self, y, k0, k1):
        """X, Y, Z at k0 .. k1 - 1 from y padded by reach() zeros on both sides."""
        pad = self.reach()
        out = torch.zeros((3, k1 - k0), dtype=torch.float64, device=self.dev)
        for ch, sign, l, D in self.terms(k0, k1):
            out[ch] += sign * (y[l, pad + k0:pad + k1] if D is None else self.read(y[l], k0, -D, pad))
        return out

    def padded(self, h):
        return torch.nn.functional.pad(h, (MARGIN + 64, MARGIN + 64))

    def response(self, hp, hc, sky):
        """(y, xyz) of the whole span"""
        sky = torch.tensor(sky, dtype=torch.float64, device=self.dev)
        hp, hc = self.padded(hp), self.padded(hc)
        steps = [(a, min(a + CHUNK, self.n)) for a in range(0, self.n, CHUNK)]
        y = torch.cat([self.project(hp, hc, sky, a, b) for a, b in steps], 1)
        yp = torch.nn.functional.pad(y, (self.reach(), self.reach()))
        return y, torch.cat([self.tdi(yp, a, b) for a, b in steps], 1)

    def transpose(self, hp, hc, sky, g):
        """gradients of sum(g * xyz) with respect to h+, hx and the sky angles"""
        pad, n = self.reach(), self.n
        gy = torch.zeros((6, n + 2 * pad), dtype=torch.float64, device=self.dev)
        for a in range(0, n, CHUNK):
            b = min(a + CHUNK, n)
            i = torch.arange(a, b, device=self.dev) + pad
            for ch, sign, l, D in self.terms(a, b):
                if D is None:
                    gy[l, i] += sign * g[ch, a:b]
                    continue
                m, eps = _split(-D)
                base = i + m - (self.T - 2) // 2
                for j, w in enumerate(_weights(eps, self.T)):
                    gy[l].index_add_(0, base + j, sign * w * g[ch, a:b])
        gy = gy[:, pad:pad + n]
        ang = torch.tensor(sky, dtype=torch.float64, device=self.dev, requires_grad=True)
        hpp, hcc = self.padded(hp), self.padded(hc)
        ghp, ghc, gs = torch.zeros_like(hpp), torch.zeros_like(hcc), torch.zeros(3, dtype=torch.float64, device=self.dev)
        step = CHUNK // 4
        for a in range(0, n, step):
            b = min(a + step, n)
            lo, hi = a, min(len(hpp), b + 4 * MARGIN + 256)   # the strain samples that this chunk reads
            wp, wc = hpp[lo:hi].clone().requires_grad_(True), hcc[lo:hi].clone().requires_grad_(True)
            self.h0 = lo
            with torch.enable_grad():
                v = (self.project(wp, wc, ang, a, b) * gy[:, a:b]).sum()
                d = torch.autograd.grad(v, (wp, wc, ang))
            self.h0 = 0
            ghp[lo:hi] += d[0]
            ghc[lo:hi] += d[1]
            gs += d[2]
        cut = MARGIN + 64
        return ghp[cut:-cut], ghc[cut:-cut], gs


_AET = ((-math.sqrt(0.5), 0.0, math.sqrt(0.5)), (math.sqrt(1 / 6), -2 * math.sqrt(1 / 6), math.sqrt(1 / 6)), (math.sqrt(1 / 3),) * 3)


def exact(case, seed):
    dev = torch.device("cuda", 0) if torch.cuda.is_available() else torch.device("cpu")
    kind, lengths = case["kind"], _lengths(case)
    if dev.type == "cpu" and sum(lengths) > 1 << 16:
        return None
    gb, sky = _sources(case, seed)
    with torch.no_grad():
        if "n" in case:
            n = lengths[0]
            hp, hc = _strain(gb[0], n, dev)
            p = _Plain(case, n, dev)
            if kind == "adjoint":
                return p.transpose(hp, hc, sky[0], _noise(case, seed, 3 * n, dev, 1.0).reshape(3, n))
            y, xyz = p.response(hp, hc, sky[0])
            if kind == "split":
                return y, xyz
            if kind == "response":
                return xyz
            M = torch.tensor(_AET, dtype=torch.float64, device=dev)
            d, h, w = _noise(case, seed, 3 * n, dev, SIGMA).reshape(3, n), M @ xyz, 1.0 / SIGMA ** 2
            logl = w * ((d * h).sum() - 0.5 * (h * h).sum())
            a, b, c = p.transpose(hp, hc, sky[0], M.T @ (w * (d - h)))
            return logl, a, b, c.cpu()
        p = _Plain(case, max(lengths), dev)
        out, off = [], _offsets(lengths)
        data = _noise(case, seed, 3 * int(off[-1]), dev, SIGMA) if kind in ("like", "gb_like") else None
        for s, n in enumerate(lengths):
            p.n = n
            xyz = p.response(*_strain(gb[s], n, dev), sky[s])[1]
            if data is None:
                out.append(xyz.reshape(-1))
                continue
            M = torch.tensor(_AET, dtype=torch.float64, device=dev)
            d, h = data[3 * off[s]:3 * off[s + 1]].reshape(3, n), M @ xyz
            out.append(((d * h).sum() - 0.5 * (h * h).sum())[None] / SIGMA ** 2)
        r = torch.cat(out)
        return r.cpu() if kind == "host" else r
