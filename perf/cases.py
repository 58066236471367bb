"""Timed cases of the library's public entry points: excess chemical potentials
(pnp_excess_mu, pnp_excess_mu_device), Gummel solves (pnp_gummel_solve) and the
serving loop (pnp_submit / pnp_poll), over the sizes, number formats and options
of the workloads, the tests and the benchmark.

`exact` restates the computation in plain FP64 numpy / torch: quadrature
stencils, torch's FFT, and conjugate gradients to rounding.
"""
import math
import time

import numpy as np
import torch

import workloads
from paper_1407_0674_gb300 import pnp

PRECISIONS = ("fp64", "df64", "fp32", "tf32split")


def listed():
    return [
        # one evaluation on a tiny grid: launch latency (the size of the smoke run's order)
        dict(name="mu_16_fp64", kind="mu", nx=16, ny=16, nz=16, pad=0, precision="fp64", fmt=0, host=False),
        # host arrays in, host arrays out, as the README's first example calls it
        dict(name="mu_64_fp32_host", kind="mu", nx=64, ny=64, nz=64, pad=0, precision="fp32", fmt=0, host=True),
        # the mu_ex microbenchmark in its FP64-accuracy, FP32 and plain FP64 forms
        dict(name="mu_128_df64", kind="mu", nx=128, ny=128, nz=128, pad=256, precision="df64", fmt=0, host=False),
        dict(name="mu_128_fp32", kind="mu", nx=128, ny=128, nz=128, pad=256, precision="fp32", fmt=0, host=False),
        dict(name="mu_128_fp64", kind="mu", nx=128, ny=128, nz=128, pad=256, precision="fp64", fmt=0, host=False),
        # ragged box, White Bear functional
        dict(name="mu_ragged_fp64", kind="mu", nx=70, ny=45, nz=101, pad=0, precision="fp64", fmt=1, host=False),
        # the three-species film's mu_ex: periodic in x and y, square wells
        dict(name="mu_film3_df64", kind="mu_film", nx=128, ny=128, nz=256, precision="df64"),
        # the 32^3 film's Gummel iteration (plain Poisson step, geometric relaxation)
        dict(name="gummel_film_32", kind="film", n=32, precision="fp64", sweeps=16),
        # a batch solve: deep wells, screened Poisson step, per-point relaxation
        dict(name="gummel_batch_96", kind="batch", n=96, precision="df64", sweeps=4),
        # a served request at the middle of the size range (no power of two)
        dict(name="gummel_serve_90", kind="serve", n=90, precision="df64", sweeps=4),
        # the large film: equilibrium stage, then the Gummel iteration
        dict(name="gummel_film3", kind="film3", nx=128, ny=128, nz=256, precision="df64", eq=2, sweeps=1),
        # uneven requests through the server, from submission to the last result
        dict(name="server_mix", kind="server", sizes="32,48,36,64", precision="df64", sweeps=16),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _smooth(rng, lo, hi):
    sizes = workloads._smooth_sizes(lo, hi)
    n = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    return min(sizes, key=lambda m: abs(m - n))


def draw(rng):
    kind = rng.choice(["mu", "mu", "mu_film", "film", "batch", "serve", "server"])
    if kind == "mu":
        p = rng.choice(PRECISIONS)
        return dict(kind=kind, nx=_log(rng, 12, 128), ny=_log(rng, 12, 128), nz=_log(rng, 12, 128), pad=0, precision=p,
                    fmt=rng.choice([0, 0, 1]), host=rng.random() < 0.25)
    if kind == "mu_film":
        return dict(kind=kind, nx=_smooth(rng, 24, 128), ny=_smooth(rng, 24, 128), nz=_log(rng, 24, 256),
                    precision=rng.choice(["fp64", "df64", "fp32"]))
    if kind == "server":
        sizes = ",".join(str(_smooth(rng, 24, 64)) for _ in range(rng.randint(2, 4)))
        return dict(kind=kind, sizes=sizes, precision=rng.choice(["fp64", "df64"]), sweeps=rng.randint(8, 16))
    n = _smooth(rng, 20, 40) if kind == "film" else _smooth(rng, 32, 100)
    return dict(kind=kind, n=n, precision=rng.choice(["fp64", "df64"]), sweeps=rng.randint(2, 6))


# ---------------------------------------------------------------------------
# inputs

def _fresh(spec, seed):
    """Sites and fixed charge of `spec` drawn again from the seed."""
    spec.sites = workloads.uniform_sites(np.random.default_rng(seed), len(spec.sites), spec.nx, spec.ny, spec.nz)
    spec.rho_f = np.random.default_rng(seed + 1).normal(0.0, 0.01, size=spec.shape)
    return spec


def _mu_inputs(case, seed):
    if case["kind"] == "mu":
        spec, _ = workloads.mu_microbench(shape=(case["nx"], case["ny"], case["nz"]), fft_len=case["pad"])
        spec.fmt = case["fmt"]
    else:
        spec = _fresh(workloads.film3(case["nx"], case["ny"], case["nz"]), seed)
    return spec, workloads.lognormal_density(spec, seed)


def _solve_spec(kind, n, sweeps, seed, case):
    rng = np.random.default_rng(seed + 7)
    if kind == "film":
        spec = workloads.film_gummel(n, n, n)
    elif kind == "batch":
        spec = workloads.batch_specs(1, seed, grids=[(n, n, n)])[0]
    elif kind == "serve":
        spec = workloads.serving_spec(n, rng.uniform(0.0, 1.0), rng.uniform(250.0, 400.0))
    else:
        spec = workloads.film3(case["nx"], case["ny"], case["nz"], bias=rng.uniform(0.0, 1.0))
        spec.eq_max_iter = case["eq"]
    spec.max_iter = sweeps
    return _fresh(spec, seed)


def _requests(case, seed):
    kinds = ("batch", "serve")
    return [_solve_spec(kinds[j % 2], int(n), case["sweeps"], seed + 100 * j, case)
            for j, n in enumerate(case["sizes"].split(","))]


def prepare(case, seed):
    if case["kind"] in ("mu", "mu_film"):
        spec, rho = _mu_inputs(case, seed)
        P = pnp.Problem(spec, precision=case["precision"])
        if case.get("host"):
            return dict(kind="mu_host", P=P, rho=rho)
        d_rho = torch.from_numpy(rho).cuda()
        d_mu = torch.empty_like(d_rho)
        torch.cuda.synchronize()
        return dict(kind="mu", P=P, rho=d_rho, mu=d_mu)
    if case["kind"] == "server":
        return dict(kind="server", srv=pnp.Server(max_slots=4, policy="smallest_first"), specs=_requests(case, seed),
                    precision=case["precision"])
    spec = _solve_spec(case["kind"], case.get("n"), case["sweeps"], seed, case)
    return dict(kind="solve", P=pnp.Problem(spec, precision=case["precision"]))


def run(state):
    if state["kind"] == "mu":
        state["P"].excess_mu_device(state["rho"], state["mu"])
        return state["mu"]
    if state["kind"] == "mu_host":
        return state["P"].excess_mu(state["rho"])
    if state["kind"] == "solve":
        phi, rho, st = state["P"].gummel_solve(raise_on_error=False)
        return dict(phi=phi, rho=rho, iterations=st["iterations"], status=st["status"])
    srv = state["srv"]
    tickets = [srv.submit(spec, precision=state["precision"])[1] for spec in state["specs"]]
    out = [None] * len(tickets)
    while any(o is None for o in out):
        for j, t in enumerate(tickets):
            if out[j] is None:
                rc, phi, rho, st = srv.poll(t)
                if rc != pnp.PENDING:
                    out[j] = dict(phi=phi, rho=rho, iterations=st["iterations"], status=rc)
        time.sleep(0.0002)
    return out


# ---------------------------------------------------------------------------
# work no implementation can do without

def _mu_flops(n, s, padded):
    # s + s real transforms of the densities and potentials and 10 + 10 of the
    # weighted densities and derivatives (2.5 L log2 L each), the spectral
    # products, the derivatives
    L = float(np.prod([float(v) for v in padded]))
    return (2 * s + 20) * 2.5 * L * math.log2(L) + 10 * s * 4 * L + 60.0 * n


def _solve_work(spec, sweeps, eq):
    n, s = spec.npoints, spec.s
    L = (spec.nx, spec.ny, spec.nz + 6)
    it = sweeps + eq
    # per iteration: mu_ex, one operator application per linear system, exponentials; phi and rho read and written
    return {"bytes": 16.0 * n * (1 + s) * it, "flops": it * (_mu_flops(n, s, L) + 13.0 * n * (1 + s) + 60.0 * n * s)}


def work(case):
    if case["kind"] == "mu":
        n, s = case["nx"] * case["ny"] * case["nz"], 3
        return {"bytes": 16.0 * s * n, "flops": _mu_flops(n, s, [case[a] + 4 for a in ("nx", "ny", "nz")])}
    if case["kind"] == "mu_film":
        n, s = case["nx"] * case["ny"] * case["nz"], 3
        return {"bytes": 16.0 * s * n + 8.0 * n, "flops": _mu_flops(n, s, (case["nx"], case["ny"], case["nz"] + 6))}
    if case["kind"] == "server":
        w = [_solve_work(spec, case["sweeps"], 0) for spec in _requests(case, 0)]
        return {k: sum(v[k] for v in w) for k in ("bytes", "flops")}
    return _solve_work(_solve_spec(case["kind"], case.get("n"), case["sweeps"], 0, case), case["sweeps"],
                       case.get("eq", 0))


# ---------------------------------------------------------------------------
# the same in 64 bits, without the library

def _nodes(r_in, r_out, surface):
    nmu = max(8, math.ceil(2 * math.pi * r_out))
    nth = (2 * nmu + 3) // 4 * 4
    if surface:
        rad, radw = np.array([r_out]), np.array([r_out * r_out])
    else:
        x, w = np.polynomial.legendre.leggauss(max(4, math.ceil(2 * (r_out - r_in))))
        rad = 0.5 * (r_out + r_in) + 0.5 * (r_out - r_in) * x
        radw = 0.5 * (r_out - r_in) * w * rad * rad
    mx, mw = np.polynomial.legendre.leggauss(nmu)
    th = 2 * math.pi * (np.arange(nth) + 0.5) / nth
    sn = np.sqrt(1 - mx * mx)
    u = np.stack([sn[:, None] * np.cos(th), sn[:, None] * np.sin(th), np.broadcast_to(mx[:, None], (nmu, nth))], -1)
    p = rad[:, None, None, None] * u
    w = radw[:, None, None] * mw[None, :, None] * (2 * math.pi / nth) * np.ones(nth)
    return p.reshape(-1, 3), w.reshape(-1), np.broadcast_to(u, p.shape).reshape(-1, 3)


class _Fmt:
    """mu_ex of a spec by torch's FFT on a zero-extended grid."""

    def __init__(self, spec):
        self.spec, self.dev = spec, torch.device("cuda")
        S = max(math.ceil(max(spec.R)) + 1, math.ceil(spec.well_outer) + 1)
        n = (spec.nz, spec.ny, spec.nx)
        self.L = tuple(m if b == "P" else m + S + (m + S) % 2 for m, b in zip(n, (spec.bc[2], spec.bc[1], spec.bc[0])))
        self.K = []
        for R in spec.R:
            p, w, u = _nodes(0.0, R, True)
            ball = _nodes(0.0, R, False)
            self.K.append([self._spectrum(p, w), self._spectrum(ball[0], ball[1])] +
                          [self._spectrum(p, w * u[:, c]) for c in range(3)])
        self.sh = None
        if spec.depth is not None and any(spec.depth) and spec.sites is not None:
            p, w, _ = _nodes(spec.well_inner, spec.well_outer, False)
            U = self._back(self._hat(self._sites()) * self._spectrum(p, w))
            self.sh = [-(0.5 if spec.sw_half else 1.0) * e * U for e in spec.depth]

    def _spectrum(self, p, w):
        base = np.floor(p).astype(np.int64)
        fr = p - base
        k = np.zeros(self.L)
        for c in np.ndindex(2, 2, 2):
            f = np.prod([fr[:, a] if c[a] else 1 - fr[:, a] for a in range(3)], axis=0)
            np.add.at(k, tuple((base[:, a] + c[a]) % self.L[2 - a] for a in (2, 1, 0)), w * f)
        return torch.fft.rfftn(torch.from_numpy(k).to(self.dev))

    def _hat(self, f):
        return torch.fft.rfftn(f, s=self.L, dim=(0, 1, 2))

    def _back(self, F):
        sp = self.spec
        return torch.fft.irfftn(F, s=self.L)[:sp.nz, :sp.ny, :sp.nx].contiguous()

    def _sites(self):
        sp, g = self.spec, []
        reach = math.sqrt(60.0 / sp.site_alpha)
        for a, (n, b) in enumerate(zip((sp.nx, sp.ny, sp.nz), sp.bc)):
            m = math.ceil(reach / n) + 1 if b == "P" else 0
            d = np.arange(n)[None, :, None] - np.asarray(sp.sites)[:, a][:, None, None] - n * np.arange(-m, m + 1)
            g.append(torch.from_numpy(np.exp(-sp.site_alpha * d * d).sum(-1)).to(self.dev))
        out = torch.stack([(g[1] * g[2][:, k:k + 1]).T @ g[0] for k in range(sp.nz)])
        return (sp.site_alpha / math.pi) ** 1.5 * out

    def mu(self, rho):
        sp, pi = self.spec, math.pi
        c0 = [1 / (4 * pi * R * R) for R in sp.R]
        c1 = [1 / (4 * pi * R) for R in sp.R]
        acc = [0.0] * 10
        for i in range(sp.s):
            h, K = self._hat(rho[i]), self.K[i]
            t = [torch.conj(k) * h for k in K]
            for a, f in enumerate([c0[i] * t[0], c1[i] * t[0], t[0], t[1]] + [c1[i] * v for v in t[2:]] + t[2:]):
                acc[a] = acc[a] + f
        n = [self._back(a) for a in acc]
        del acc
        n0, n1, n2, n3, v1, v2 = n[0], n[1], n[2], n[3], n[4:7], n[7:10]
        g = 1 / (1 - n3)
        v12 = v1[0] * v2[0] + v1[1] * v2[1] + v1[2] * v2[2]
        v22 = v2[0] * v2[0] + v2[1] * v2[1] + v2[2] * v2[2]
        if sp.fmt:
            f, df = torch.zeros_like(n3), torch.zeros_like(n3)
            for k in range(40, -1, -1):
                c = (k + 1) * (k + 3) / (k + 2)
                df = df * n3 + f
                f = f * n3 + c
            L, o = torch.log1p(-n3), 1 - n3
            fc = (n3 + o * o * L) / (n3 * n3 * o * o)
            dc = (n3 - 2 * o * L) / (n3 * n3 * o * o) - 2 * (1 - 2 * n3) * fc / (n3 * o)
            far = n3.abs() > 0.2
            f, df = torch.where(far, fc, f), torch.where(far, dc, df)
            c2, c3, cv = f / (12 * pi), df / (36 * pi), f / (6 * pi)
        else:
            c2, c3, cv = g * g / (8 * pi), g ** 3 / (12 * pi), g * g / (4 * pi)
        psi = [-torch.log1p(-n3), n2 * g, n1 * g + (n2 * n2 - v22) * c2,
               n0 * g + (n1 * n2 - v12) * g * g + (n2 ** 3 - 3 * n2 * v22) * c3]
        psi += [-v2[c] * g for c in range(3)] + [-v1[c] * g - n2 * v2[c] * cv for c in range(3)]
        hat = [self._hat(p) for p in psi]
        del psi, n
        out = []
        for i in range(sp.s):
            K = self.K[i]
            F = K[0] * (c0[i] * hat[0] + c1[i] * hat[1] + hat[2]) + K[1] * hat[3]
            for c in range(3):
                F = F + K[2 + c] * (c1[i] * hat[4 + c] + hat[7 + c])
            m = self._back(F)
            out.append(m if self.sh is None else m + self.sh[i])
        return torch.stack(out)

    def bulk(self):
        """Reservoir values: the functional's derivatives in the uniform fluid."""
        sp, pi = self.spec, math.pi
        n = [sum(r * w for r, w in zip(sp.rho_b, ws)) for ws in
             zip(*[(1.0, R, 4 * pi * R * R, 4 * pi * R ** 3 / 3) for R in sp.R])]
        g = 1 / (1 - n[3])
        d = [-math.log1p(-n[3]), n[2] * g, n[1] * g + n[2] ** 2 * g * g / (8 * pi),
             n[0] * g + n[1] * n[2] * g * g + n[2] ** 3 * g ** 3 / (12 * pi)]
        return [d[0] + R * d[1] + 4 * pi * R * R * d[2] + 4 * pi * R ** 3 / 3 * d[3] for R in sp.R]


def _apply(cx, cy, cz, clo, u):
    """7-point operator with face coefficients to +x, +y (periodic), +z and the lower plane."""
    fx, fy = cx * (u - torch.roll(u, -1, 2)), cy * (u - torch.roll(u, -1, 1))
    out = fx - torch.roll(fx, 1, 2) + fy - torch.roll(fy, 1, 1)
    fz = cz * u
    fz[:-1] -= cz[:-1] * u[1:]
    out += fz
    out[1:] -= fz[:-1]
    out[0] += clo * u[0]
    return out


def _cg(cx, cy, cz, clo, dg, b, x):
    diag = cx + torch.roll(cx, 1, 2) + cy + torch.roll(cy, 1, 1) + cz
    diag[1:] += cz[:-1]
    diag[0] += clo
    diag = diag + dg
    r = b - _apply(cx, cy, cz, clo, x) - dg * x
    z = r / diag
    p, rz = z.clone(), (r * z).sum()
    goal = 1e-14 * float(b.norm())
    for it in range(6000):
        Ap = _apply(cx, cy, cz, clo, p) + dg * p
        a = rz / (p * Ap).sum()
        x = x + a * p
        r = r - a * Ap
        if it % 25 == 24 and float(r.norm()) <= goal:
            break
        z = r / diag
        new = (r * z).sum()
        p = z + (new / rz) * p
        rz = new
    return x


def _exact_solve(spec):
    F, dev = _Fmt(spec), torch.device("cuda")
    e, eps0, kB = 1.602176634e-19, 8.8541878128e-12, 1.380649e-23
    four = 4 * math.pi * e * e / (4 * math.pi * eps0 * spec.eps_r * kB * spec.temperature_K) * 1e9 / spec.h_nm
    mub, one = F.bulk(), torch.ones(spec.shape, dtype=torch.float64, device=dev)
    k = torch.arange(1, spec.nz + 1, dtype=torch.float64, device=dev) / (spec.nz + 1)
    phi = (spec.phi_lo + (spec.phi_hi - spec.phi_lo) * k)[:, None, None] * one
    rho = torch.stack([r * one for r in spec.rho_b])
    rho_f = torch.from_numpy(spec.rho_f).to(dev)
    lam = torch.full_like(rho, spec.lambda_rho)
    prev = torch.zeros_like(rho)
    lo = one[0]

    def charge(r):
        b = four * (rho_f + sum(q * r[i] for i, q in enumerate(spec.q)))
        b[0] += spec.phi_lo
        b[-1] += spec.phi_hi
        return b, four * sum(q * q * r[i] for i, q in enumerate(spec.q))

    def newton(r):
        b, dg = charge(r)
        return _cg(one, one, one, lo, dg, b - _apply(one, one, one, lo, phi), torch.zeros_like(phi))

    for _ in range(spec.eq_max_iter if spec.eq_init else 0):
        mu = F.mu(rho)
        cb = [r * math.exp(m) for r, m in zip(spec.rho_b, mub)]
        d = newton([c * torch.exp(-(mu[i] + q * phi)) for i, (c, q) in enumerate(zip(cb, spec.q))]).clamp(-1, 1)
        phi = phi + d
        for i, q in enumerate(spec.q):
            rs = cb[i] * torch.exp(-(mu[i] + q * phi))
            rho[i] *= torch.exp((spec.lambda_rho * torch.log(rs / rho[i])).clamp(-0.2, 0.2))
    for _ in range(spec.max_iter):
        mu = F.mu(rho)
        if spec.screened_poisson:
            star = phi + newton(rho)
        else:
            star = _cg(one, one, one, lo, torch.zeros_like(phi), charge(rho)[0], phi)
        phi = spec.lambda_phi * star + (1 - spec.lambda_phi) * phi
        for i, q in enumerate(spec.q):
            D0 = 1.0 if spec.D is None else spec.D[i]
            D = D0 * torch.exp(-(q * phi + mu[i]))
            mean = lambda a, b: 2 * a * b / (a + b)  # noqa: E731
            Dlo, Dhi = (D0 * math.exp(-(q * v + mub[i])) for v in (spec.phi_lo, spec.phi_hi))
            cx, cy = mean(D, torch.roll(D, -1, 2)), mean(D, torch.roll(D, -1, 1))
            cz = torch.cat([mean(D[:-1], D[1:]), mean(D[-1:], Dhi)])
            clo = mean(D[0], Dlo)
            b = torch.zeros_like(phi)
            b[0] += clo * spec.rho_b[i] * math.exp(q * spec.phi_lo + mub[i])
            b[-1] += cz[-1] * spec.rho_b[i] * math.exp(q * spec.phi_hi + mub[i])
            x = _cg(cx, cy, cz, clo, torch.zeros_like(phi), b, rho[i] * torch.exp(q * phi + mu[i]))
            rs = x * torch.exp(-(q * phi + mu[i]))
            if spec.rho_mix == 3:
                t = torch.log(rs / rho[i])
                a = torch.where(t * prev[i] < 0, (0.5 * lam[i]).clamp(min=spec.lambda_rho / 1024),
                                (1.1 * lam[i]).clamp(max=spec.lambda_rho))
                lam[i], prev[i] = a, (a * t).clamp(-0.2, 0.2)
                rho[i] *= torch.exp(prev[i])
            else:
                t = spec.lambda_rho * torch.log(rs / rho[i])
                rho[i] *= torch.exp(t.clamp(-0.2, 0.2) if spec.rho_mix == 2 else t)
    return dict(phi=phi.cpu().numpy(), rho=rho.cpu().numpy(), iterations=None, status=None)


def exact(case, seed):
    if case["kind"] in ("mu", "mu_film"):
        spec, rho = _mu_inputs(case, seed)
        return _Fmt(spec).mu(torch.from_numpy(rho).cuda())
    if case["kind"] == "server":
        return [_exact_solve(spec) for spec in _requests(case, seed)]
    return _exact_solve(_solve_spec(case["kind"], case.get("n"), case["sweeps"], seed, case))
