"""The work whose speed counts: calls of this package's public entry points.

Each case is one call (or one forward and backward pass) as a lattice-QCD
program makes it: the operator alone, GMRES-DR, the deflated BiCGStab solves
in FP64 and in mixed precision, the twisted-mass shifts, the differentiable
solve and the tall-skinny product.  Gauge fields are random SU(3) links
exp(i eps H) and sources Gaussian or Z4 noise, made on the GPU from the seed.

Solves run to a true residual of 1e-12, where two solutions of one system
agree to about 1e-10 however the arithmetic of the iteration is arranged.
"""
import math

import torch

import paper_0710_1988_gb300 as wdl
from paper_0710_1988_gb300.autograd import wilson_solve

TOL = 1e-12
EPS = 0.5          # spread of the links, as in this repository's workloads (kappa_c ~ 0.1477)
DEV = "cuda"


def _apply(name, dims, nrhs, dagger=False, mu=0.0, even_odd=False):
    return {"name": name, "kind": "apply", "lx": dims[0], "ly": dims[1], "lz": dims[2], "lt": dims[3],
            "nrhs": nrhs, "kappa": 0.137, "mu": mu, "dagger": dagger, "even_odd": even_odd}


def _gmresdr(name, dims, m, k, cycles):
    return {"name": name, "kind": "gmresdr", "lx": dims[0], "ly": dims[1], "lz": dims[2], "lt": dims[3],
            "kappa": 0.146, "m": m, "k": k, "cycles": cycles}


def _solve(name, dims, nrhs, kappa, k=0, m=0, bits=64, delta=0.0, even_odd=False):
    return {"name": name, "kind": "solve", "lx": dims[0], "ly": dims[1], "lz": dims[2], "lt": dims[3],
            "nrhs": nrhs, "kappa": kappa, "m": m, "k": k, "bits": bits, "delta": delta,
            "even_odd": even_odd}


def listed():
    return [
        # one operator product on the smallest lattice: launch latency
        _apply("apply_4x4x4x4", (4, 4, 4, 4), 1),
        # A^dagger of a few twisted-mass spinors on a lattice of odd extents
        _apply("apply_dagger_ragged", (9, 7, 5, 11), 3, dagger=True, mu=0.05),
        # the operator on the right-hand sides of one batched solve
        _apply("apply_16x16x16x16_x10", (16, 16, 16, 16), 10),
        # one vector on the largest lattice
        _apply("apply_32x32x32x64", (32, 32, 32, 64), 1),
        # the even-odd Schur operator, a batch on a large lattice
        _apply("apply_even_odd_24x24x24x48", (24, 24, 24, 48), 4, mu=0.016, even_odd=True),
        # GMRES-DR(80,40) on the first source, a full cycle and a restarted one, and the
        # deflation space it leaves at work on the next source
        _gmresdr("gmresdr_16x16x16x16", (16, 16, 16, 16), 80, 40, 2),
        # a small deflated FP64 solve: every launch is short
        _solve("solve_fp64_4x4x4x4", (4, 4, 4, 4), 3, 0.13, k=6, m=20),
        # the deflated FP64 solve of ten sources
        _solve("solve_fp64_16x16x16x16", (16, 16, 16, 16), 10, 0.146, k=40, m=80),
        # the mixed-precision solve of twelve sources, restarted refinement
        _solve("solve_fp32_20x20x20x32", (20, 20, 20, 32), 12, 0.146, bits=32, delta=1e-3),
        # FP16 storage, reliable updates
        _solve("solve_fp16_16x16x16x32", (16, 16, 16, 32), 4, 0.145, bits=16),
        # twisted-mass shifts of four sources through the even-odd system, each
        # projected over the earlier solutions, mixed precision
        {"name": "shifts_16x16x16x32", "kind": "shifts", "lx": 16, "ly": 16, "lz": 16, "lt": 32,
         "nrhs": 4, "kappa": 0.146, "nshift": 3, "mu0": 0.064, "even_odd": True, "mixed": True},
        # forward and backward through one FP64 solve: gradients of source, kappa and links
        {"name": "gradient_8x8x8x16", "kind": "gradient", "lx": 8, "ly": 8, "lz": 8, "lt": 16,
         "kappa": 0.144, "mixed": False},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_dims(rng, vmin, vmax, even=False):
    """Extents whose product lies between vmin and vmax, log-uniformly."""
    target = math.exp(rng.uniform(math.log(vmin), math.log(vmax)))
    side = target ** 0.25
    dims = []
    for i in range(4):
        d = side * math.exp(rng.uniform(-0.35, 0.35)) if i < 3 else target / math.prod(dims)
        d = max(2, int(round(d)))
        dims.append(d + d % 2 if even else d)
    while math.prod(dims) > vmax and max(dims) > 2:
        i = dims.index(max(dims))
        dims[i] -= 2 if even else 1
    return tuple(dims)


def draw(rng):
    kind = rng.choice(["apply", "apply", "apply_eo", "gmresdr", "solve64", "solve64", "solve32",
                       "solve16", "shifts", "gradient"])
    if kind == "apply":
        dims = _draw_dims(rng, 256, 1.5e6)
        top = max(1, min(16, int(2.0e6 / math.prod(dims))))
        c = _apply("", dims, _log_int(rng, 1, top), dagger=rng.random() < 0.5,
                   mu=rng.choice([0.0, 0.0, 0.05, -0.3]))
    elif kind == "apply_eo":
        dims = _draw_dims(rng, 256, 6.0e5, even=True)
        top = max(1, min(16, int(2.4e6 / math.prod(dims))))
        c = _apply("", dims, _log_int(rng, 1, top), dagger=rng.random() < 0.5,
                   mu=rng.choice([0.0, 0.016, 0.064]), even_odd=True)
    elif kind == "gmresdr":
        m = rng.randint(12, 80)
        c = _gmresdr("", _draw_dims(rng, 1500, 6.0e4), m, rng.randint(4, max(4, 5 * m // 8)),
                     rng.randint(1, 2))
    elif kind in ("solve64", "solve32", "solve16"):
        bits = int(kind[5:])
        even = bits != 16 and rng.random() < 0.3
        dims = _draw_dims(rng, 256, 6.5e4 if bits == 64 else 1.3e5, even=even)
        top = max(1, min(12, int((4.0e5 if bits == 64 else 1.5e6) / math.prod(dims))))
        k = rng.choice([0, rng.randint(4, 24)]) if bits != 16 else 0
        c = _solve("", dims, _log_int(rng, 1, top), round(rng.uniform(0.125, 0.144), 4), k=k,
                   m=2 * k + 8 if k else 0, bits=bits,
                   delta=0.0 if bits == 64 else rng.choice([0.0, 1e-3]), even_odd=even)
    elif kind == "shifts":
        dims = _draw_dims(rng, 256, 1.3e5, even=True)
        top = max(1, min(6, int(5.0e5 / math.prod(dims))))
        c = {"kind": "shifts", "lx": dims[0], "ly": dims[1], "lz": dims[2], "lt": dims[3],
             "nrhs": _log_int(rng, 1, top), "kappa": round(rng.uniform(0.13, 0.146), 4),
             "nshift": rng.randint(2, 3), "mu0": rng.choice([0.064, 0.048, 0.1]),
             "even_odd": rng.random() < 0.6, "mixed": rng.random() < 0.6}
    else:
        dims = _draw_dims(rng, 256, 3.3e4)
        c = {"kind": "gradient", "lx": dims[0], "ly": dims[1], "lz": dims[2], "lt": dims[3],
             "kappa": round(rng.uniform(0.125, 0.144), 4), "mixed": rng.random() < 0.5}
    c.pop("name", None)
    return c


# ------------------------------------------------------------------ inputs

def _dims(c):
    return (c["lx"], c["ly"], c["lz"], c["lt"])


def _volume(c):
    return math.prod(_dims(c))


def _matmul(a, b):
    return (a.unsqueeze(-1) * b.unsqueeze(-3)).sum(-2)


def _gell_mann():
    l = torch.zeros(8, 3, 3, dtype=torch.complex128)
    l[0, 0, 1] = l[0, 1, 0] = l[1, 1, 0] = l[2, 0, 0] = 1
    l[1, 0, 1], l[1, 1, 0], l[2, 1, 1] = -1j, 1j, -1
    l[3, 0, 2] = l[3, 2, 0] = l[5, 1, 2] = l[5, 2, 1] = 1
    l[4, 0, 2], l[4, 2, 0], l[6, 1, 2], l[6, 2, 1] = -1j, 1j, -1j, 1j
    l[7, 0, 0] = l[7, 1, 1] = 1 / math.sqrt(3)
    l[7, 2, 2] = -2 / math.sqrt(3)
    return l.to(DEV)


def _links(volume, gen):
    """SU(3) links exp(i EPS sum_a h_a lambda_a / 2), h_a ~ N(0, 1): (V, 4, 3, 3)."""
    h = torch.randn(volume * 4, 8, dtype=torch.float64, device=DEV, generator=gen)
    x = (h.to(torch.complex128) @ _gell_mann().reshape(8, 9)).reshape(volume * 4, 3, 3) * (0.125j * EPS)
    u = term = torch.eye(3, dtype=torch.complex128, device=DEV).expand_as(x)
    for i in range(1, 9):                      # exp(x), squared twice
        term = _matmul(term, x) / i
        u = u + term
    u = _matmul(u, u)
    u = _matmul(u, u)
    r0 = u[:, 0] / torch.linalg.vector_norm(u[:, 0], dim=-1, keepdim=True)
    r1 = u[:, 1] - (r0.conj() * u[:, 1]).sum(-1, keepdim=True) * r0
    r1 = r1 / torch.linalg.vector_norm(r1, dim=-1, keepdim=True)
    r2 = torch.linalg.cross(r0, r1).conj()
    return torch.stack([r0, r1, r2], 1).reshape(volume, 4, 3, 3).contiguous()


def _gaussian(shape, gen):
    r = torch.randn(*shape, 2, dtype=torch.float64, device=DEV, generator=gen)
    return torch.view_as_complex(r)


def _z4(shape, gen):
    k = torch.randint(0, 4, shape, device=DEV, generator=gen)
    return torch.tensor([1, 1j, -1, -1j], dtype=torch.complex128, device=DEV)[k]


def _inputs(case, seed):
    """Links and sources of a case, from the seed alone."""
    gen = torch.Generator(device=DEV).manual_seed(int(seed))
    v = _volume(case)
    links = _links(v, gen)
    n = 12 * v // (2 if case["kind"] in ("apply", "solve") and case["even_odd"] else 1)
    nrhs = 2 if case["kind"] == "gmresdr" else case.get("nrhs", 1)
    if case["kind"] in ("gmresdr", "solve"):
        return links, _z4((nrhs, n), gen), gen
    return links, _gaussian((nrhs, n), gen), gen


def _mus(case):
    return [case["mu0"] / 2 ** i for i in range(case["nshift"])]


def prepare(case, seed):
    links, b, gen = _inputs(case, seed)
    kind = case["kind"]
    op = wdl.WilsonOperator(_dims(case), links, case["kappa"], case.get("mu", 0.0))
    s = {"case": case, "op": op, "b": b}
    if case.get("even_odd"):
        op.set_operator(True)
    if kind == "apply":
        s["out"] = torch.empty_like(b)
    elif kind == "gmresdr":
        s["x"] = torch.empty_like(b)
        s["V"] = torch.empty(case["k"], b.shape[1], dtype=torch.complex128, device=DEV)
    elif kind == "solve":
        s["x"] = torch.empty_like(b)
        if case["bits"] != 64:
            op.set_mixed_storage(case["bits"])
            op.set_mixed_restart(case["delta"])
        s["defl"] = None
        if case["k"]:                # the deflation space that a first solve left
            n = b.shape[1]
            b0, x0 = _z4((n,), gen), torch.zeros(n, dtype=torch.complex128, device=DEV)
            V = torch.empty(case["k"], n, dtype=torch.complex128, device=DEV)
            op.gmresdr(b0, x0, case["m"], case["k"], 1e-6, 2000, V_out=V)
            s["defl"] = op.deflation(V, case["k"])
    elif kind == "shifts":
        s["x"] = torch.empty(case["nshift"], *b.shape, dtype=torch.complex128, device=DEV)
    else:
        s["b"] = b.reshape(-1).requires_grad_()
        s["g"] = _gaussian((b.numel(),), gen)
        s["kappa"] = torch.tensor(case["kappa"], dtype=torch.float64, requires_grad=True)
        s["omega"] = torch.zeros(_volume(case), 4, 8, dtype=torch.float64, device=DEV,
                                 requires_grad=True)
    return s


# ------------------------------------------------------------------ one pass

def run(s):
    case, op, b = s["case"], s["op"], s["b"]
    kind = case["kind"]
    if kind == "apply":
        return op.apply(b, s["out"], dagger=case["dagger"])
    if kind == "gmresdr":
        s["x"].zero_()
        m, k = case["m"], case["k"]
        _, _, _, theta = op.gmresdr(b[0], s["x"][0], m, k, TOL, m + (m - k) * (case["cycles"] - 1),
                                    V_out=s["V"])
        # the basis itself is fixed only up to a rotation within its span, and
        # the projection that it is made for depends on the span alone
        op.dbicgstab(b[1], s["x"][1], op.deflation(s["V"], k), tol=TOL, max_iter=1)
        return {"x": s["x"][0], "theta": theta, "next": s["x"][1]}
    if kind == "solve":
        s["x"].zero_()
        call = op.dbicgstab if case["bits"] == 64 else op.dbicgstab_mixed
        rc, _ = call(b, s["x"], s["defl"], tol=TOL, max_iter=20000)
        if rc != 0:
            raise RuntimeError("the solve did not converge")
        return s["x"]
    if kind == "shifts":
        rc, _ = op.multishift(b, s["x"], _mus(case), tol=TOL, max_iter=20000, mixed=case["mixed"])
        if rc != 0:
            raise RuntimeError("a shift did not converge")
        return s["x"]
    x = wilson_solve(b, s["kappa"], s["omega"], op, tol=TOL, mixed=case["mixed"])
    gb, gk, gw = torch.autograd.grad(x, (b, s["kappa"], s["omega"]), s["g"])
    return {"x": x.detach(), "b": gb, "kappa": gk, "omega": gw}


# ------------------------------------------------------------------ what a pass cannot do without

def _iterations(kappa, even_odd=False, tol=TOL):
    """Typical BiCGStab iterations of one source on these fields, measured
    near kappa_c (about 330 at kappa = 0.146 to 1e-12), half on the Schur system."""
    n = 14.0 * -math.log10(tol) / 12 / (0.1477 / kappa - 1 + 0.03)
    return n / 2 if even_odd else n


def _product(v, nrhs, size=16, half=False):
    """Bytes and flops of one operator product: links once, vectors in and out."""
    return 36 * size * v + (12 if half else 24) * size * v * nrhs, 1368.0 * v * nrhs


def _bicgstab(v, nrhs, iters, size, even_odd):
    """Two products an iteration, and its three vector updates (r, p, v, s, t,
    x and the shadow residual: 14 vectors read or written, 30 flops a component)."""
    n = (6 if even_odd else 12) * v
    pb, pf = _product(v, nrhs, size, even_odd)
    return iters * (2 * pb + 14 * size * n * nrhs), iters * (2 * pf + 30.0 * n * nrhs)


def work(case):
    v, kind = _volume(case), case["kind"]
    eo = bool(case.get("even_odd"))
    if kind == "apply":
        b, f = _product(v, case["nrhs"], half=eo)
    elif kind == "gmresdr":
        n, m, k = 12 * v, case["m"], case["k"]
        b = f = 0.0
        for cyc in range(case["cycles"]):
            for j in range(k if cyc else 0, m):      # both Gram-Schmidt passes read the basis
                pb, pf = _product(v, 1)
                b += pb + 2 * 16.0 * n * (j + 1)
                f += pf + 32.0 * n * (j + 1)
            b += 16.0 * n * (m + 1 + k + 1 + m)      # restart product and x += V d
            f += 8.0 * n * ((m + 1) * (k + 1) + m)
        pb, pf = _product(v, k + 2)                  # W = A V, U^dagger W, the next source
        b, f = b + pb + 16.0 * n * 4 * k, f + pf + 8.0 * n * (k * k + 3 * k)
    elif kind == "solve":
        size = {64: 16, 32: 8, 16: 4}[case["bits"]]
        b, f = _bicgstab(v, case["nrhs"], _iterations(case["kappa"], eo), size, eo)
    elif kind == "shifts":
        b, f = _bicgstab(v, case["nrhs"], _iterations(case["kappa"], eo),
                         8 if case["mixed"] else 16, eo)
        b, f = b * case["nshift"], f * case["nshift"]
    else:
        b, f = _bicgstab(v, 1, 2 * _iterations(case["kappa"]), 8 if case["mixed"] else 16, False)
        b, f = b + v * (36 * 16 + 4 * 8 * 8 + 24 * 16), f + 4100.0 * v
    return {"bytes": float(b), "flops": float(f)}


# ------------------------------------------------------------------ plain torch in 64 bits

def _spin():
    """gamma matrices of the chiral basis, [[0, B], [B^dagger, 0]]."""
    s = torch.zeros(3, 2, 2, dtype=torch.complex128)
    s[0, 0, 1] = s[0, 1, 0] = s[2, 0, 0] = 1
    s[1, 0, 1], s[1, 1, 0], s[2, 1, 1] = -1j, 1j, -1
    g = torch.zeros(4, 4, 4, dtype=torch.complex128)
    for mu in range(4):
        blk = -1j * s[mu] if mu < 3 else torch.eye(2, dtype=torch.complex128)
        g[mu, :2, 2:], g[mu, 2:, :2] = blk, blk.conj().T
    return g.to(DEV)


class _Plain:
    """The Wilson operator with torch indexing; spinors (nrhs, V, 4, 3)."""

    def __init__(self, case, links):
        self.dims, self.links = _dims(case), links
        site = torch.arange(_volume(case), device=DEV).reshape(self.dims[::-1])
        self.up = [torch.roll(site, -1, 3 - mu).reshape(-1) for mu in range(4)]
        self.dn = [torch.roll(site, 1, 3 - mu).reshape(-1) for mu in range(4)]
        co = torch.meshgrid(*[torch.arange(d, device=DEV) for d in self.dims[::-1]], indexing="ij")
        self.parity = (sum(co) % 2).reshape(-1)
        self.gamma, self.one = _spin(), torch.eye(4, dtype=torch.complex128, device=DEV)
        self.g5 = torch.tensor([1.0, 1.0, -1.0, -1.0], device=DEV, dtype=torch.float64)[:, None]

    def hop(self, psi):
        out = torch.zeros_like(psi)
        for r in range(psi.shape[0]):
            for mu in range(4):
                u = self.links[:, mu]
                f = torch.einsum("st,vta->vsa", self.one - self.gamma[mu], psi[r][self.up[mu]])
                out[r] += torch.einsum("vab,vsb->vsa", u, f)
                w = torch.einsum("st,vta->vsa", self.one + self.gamma[mu], psi[r])
                w = torch.einsum("vba,vsb->vsa", u.conj(), w)
                out[r] += w[self.dn[mu]]
        return out

    def full(self, psi, kappa, mu=0.0):
        return psi - kappa * self.hop(psi) + 1j * mu * self.g5 * psi

    def schur(self, half, kappa, mu=0.0):
        psi = torch.zeros(half.shape[0], self.parity.numel(), 4, 3, dtype=half.dtype, device=DEV)
        even = self.parity == 0
        psi[:, even] = half
        odd = self.hop(psi) * (1 - 1j * mu * self.g5) / (1 + mu * mu)
        odd[:, even] = 0
        return (1 + 1j * mu * self.g5) * half - kappa * kappa * self.hop(odd)[:, even]

    def apply(self, psi, kappa, mu=0.0, dagger=False, even_odd=False):
        f = self.schur if even_odd else self.full
        return self.g5 * f(self.g5 * psi, kappa, -mu) if dagger else f(psi, kappa, mu)

    def solve(self, b, kappa, mu=0.0, dagger=False, even_odd=False):
        """BiCGStab to 1e-9, restarted from the true residual down to rounding."""
        A = lambda z: self.apply(z, kappa, mu, dagger, even_odd)
        dot = lambda p, q: (p.conj() * q).sum((1, 2, 3), keepdim=True)
        nrm = lambda p: dot(p, p).real.sqrt()
        x = torch.zeros_like(b)
        for _ in range(4):
            r = b - A(x)
            goal, d = 1e-5 * nrm(r), torch.zeros_like(r)
            r0, p, rho = r, r, dot(r, r)
            for it in range(3000):
                v = A(p)
                alpha = rho / dot(r0, v)
                s = r - alpha * v
                t = A(s)
                omega = dot(t, s) / dot(t, t)
                d = d + alpha * p + omega * s
                r = s - omega * t
                if it % 8 == 7 and bool((nrm(r) <= goal).all()):
                    break
                new = dot(r0, r)
                p = r + (new / rho) * (alpha / omega) * (p - omega * v)
                rho = new
            x = x + d
        return x


def _plain_gmresdr(case, A, g5, b):
    """GMRES-DR(m,k) with modified Gram-Schmidt applied twice, then the projection
    of the next source over the k vectors and one BiCGStab iteration."""
    m, k, n = case["m"], case["k"], b.shape[1]
    q = torch.zeros(m + 1, n, dtype=torch.complex128, device=DEV)
    h = torch.zeros(m + 1, m, dtype=torch.complex128, device=DEV)
    c = torch.zeros(m + 1, 1, dtype=torch.complex128, device=DEV)
    c[0] = torch.linalg.vector_norm(b[0])
    q[0], x, first = b[0] / c[0], torch.zeros_like(b[0]), 0
    for _ in range(case["cycles"]):
        for j in range(first, m):
            w = A(q[j])
            for _ in range(2):
                for i in range(j + 1):
                    d = torch.vdot(q[i], w)
                    h[i, j] += d
                    w = w - d * q[i]
            h[j + 1, j] = torch.linalg.vector_norm(w)
            q[j + 1] = w / h[j + 1, j]
        d = torch.linalg.lstsq(h, c).solution
        x = x + d[:, 0] @ q[:m]
        left = c - h @ d
        f = torch.linalg.solve(h[:m].conj().T, torch.eye(m, dtype=h.dtype, device=DEV)[:, m - 1])
        harm = h[:m].clone()
        harm[:, m - 1] += h[m, m - 1].abs() ** 2 * f
        theta, vec = torch.linalg.eig(harm)
        order = sorted(range(m), key=lambda i: (abs(theta[i].item()), theta[i].real.item()))[:k]
        theta = theta[order]
        p = torch.zeros(m + 1, k + 1, dtype=torch.complex128, device=DEV)
        p[:m, :k], p[:, k] = vec[:, order], left[:, 0]
        p = torch.linalg.qr(p).Q
        p = torch.linalg.qr(p).Q
        hk, c = p.conj().T @ h @ p[:m, :k], torch.cat([p.conj().T @ left, c.new_zeros(m - k, 1)])
        q[:k + 1] = p.T @ q
        h = torch.zeros_like(h)
        h[:k + 1, :k], first = hk, k
    v = q[:k]
    u = (v.reshape(k, -1, 4, 3) * g5).reshape(k, n)
    w = torch.stack([A(z) for z in v])
    y = torch.linalg.solve(u.conj() @ w.T, u.conj() @ b[1])
    x1, r = y @ v, b[1] - y @ w
    ar = A(r)
    alpha = torch.vdot(r, r) / torch.vdot(r, ar)
    s = r - alpha * ar
    t = A(s)
    return {"x": x, "theta": theta.cpu(),
            "next": x1 + alpha * r + torch.vdot(t, s) / torch.vdot(t, t) * s}


def exact(case, seed):
    kind, v, nrhs = case["kind"], _volume(case), case.get("nrhs", 1)
    if kind in ("solve", "shifts", "gradient"):
        # a plain solve of more than this takes too long
        if v * nrhs * case.get("nshift", 1) > 30000:
            return None
    elif kind == "gmresdr" and v > 140000:
        return None
    links, b, gen = _inputs(case, seed)
    plain = _Plain(case, links)
    kappa, eo = case["kappa"], bool(case.get("even_odd"))
    shape = (nrhs, -1, 4, 3)
    if kind == "apply":
        out = plain.apply(b.reshape(shape), kappa, case["mu"], case["dagger"], eo)
        return out.reshape(b.shape)
    if kind == "gmresdr":
        return _plain_gmresdr(case, lambda z: plain.full(z.reshape(1, -1, 4, 3), kappa).reshape(-1),
                              plain.g5, b)
    if kind == "solve":
        return plain.solve(b.reshape(shape), kappa, even_odd=eo).reshape(b.shape)
    if kind == "shifts":
        return torch.stack([plain.solve(b.reshape(shape), kappa, mu).reshape(b.shape)
                            for mu in _mus(case)])
    g = _gaussian((b.numel(),), gen)
    x = plain.solve(b.reshape(shape), kappa)
    lam = plain.solve(g.reshape(shape), kappa, dagger=True)
    # Re(g^dagger dx) = -Re(lam^dagger dA x): differentiate -Re(lam^dagger A x)
    k = torch.tensor(kappa, dtype=torch.float64, device=DEV, requires_grad=True)
    om = torch.zeros(v, 4, 8, dtype=torch.float64, device=DEV, requires_grad=True)
    turn = torch.einsum("vma,aij->vmij", om.to(torch.complex128), 0.5j * _gell_mann())
    plain.links = links + _matmul(turn, links)
    loss = -(lam.conj() * plain.full(x, k)).real.sum()
    gk, gw = torch.autograd.grad(loss, (k, om))
    return {"x": x.reshape(-1), "b": lam.reshape(-1), "kappa": gk.detach().cpu(), "omega": gw}
