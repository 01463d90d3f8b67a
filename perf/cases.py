"""Cases that time the library through its Python API.

Each case is one thing a user of the library does with it: apply the
operator to vectors that are on the GPU and take the result back as a
tensor, apply it to the twelve sources of a propagator, precondition, take
over a new gauge configuration, solve for one source or for twelve, compute
the pseudofermion force.  Sizes, links, couplings and solver settings are
those of the workloads in synth/ and bench.py.

exact() recomputes every result in complex128 with plain torch from the
definition of the operator (full 4x4 spin matrices, whole-lattice shifts)
and shares no code with the library.
"""
import math

import torch

import paper_1612_06556_gb300 as wc

DEV = "cuda"
C128 = torch.complex128
PREC = {"f64": wc.F64, "f32": wc.F32, "f16": wc.F16}


def _case(name, kind, dims, **kw):
    c = {"name": name, "kind": kind, "lx": dims[0], "ly": dims[1], "lz": dims[2], "lt": dims[3],
         "links": "exp", "eps": 0.3, "csw": 1.0, "kappa": 0.124}
    c.update(kw)
    return c


def listed():
    return [
        # The smallest operator call: a coarse lattice, where the launches
        # and the latency of one site's work count and bandwidth does not.
        _case("normal_f32_8x8x8x8", "normal", (8, 8, 8, 8), prec="f32", kappa=0.12),
        # M^+ M of one vector on the lattice the paper quotes its hopping
        # rate on: the inner loop of every solver that a user writes around
        # the operator.
        _case("normal_f32_24x24x24x32", "normal", (24, 24, 24, 32), prec="f32", links="haar", kappa=0.125),
        # The largest lattice of the workloads, with the binary16 storage it
        # prescribes.
        _case("normal_f16_32x32x32x64", "normal", (32, 32, 32, 64), prec="f16", eps=0.25, csw=1.6, kappa=0.128),
        # The double-precision operator, which every outer solver and every
        # residual check applies.
        _case("normal_f64_16x16x16x32", "normal", (16, 16, 16, 32), prec="f64", arith="f64"),
        # The twelve spin-colour sources of a propagator through the
        # operator in one call each way.
        _case("multi12_f32_24x24x24x32", "multi", (24, 24, 24, 32), prec="f32", rhs=12, links="haar", kappa=0.125),
        # The same on the even-odd operator that the propagator solves use.
        _case("schur12_f32_16x16x16x32", "schur_multi", (16, 16, 16, 32), prec="f32", rhs=12),
        # One application of the Schwarz preconditioner (4^4 blocks, overlap
        # 1, four MR steps) to a vector.
        _case("ras_f32_24x24x24x32", "ras", (24, 24, 24, 32), prec="f32", links="haar", kappa=0.125, schur=False,
              mr=4),
        # A new gauge configuration taken over: links, clover term, and its
        # inverse through the first even-odd application (each step of a
        # molecular-dynamics trajectory, each configuration of an ensemble).
        _case("configuration_16x16x16x32", "config", (16, 16, 16, 32), kappa=0.12),
        # Action and force of one molecular-dynamics step.
        _case("force_16x16x16x32", "force", (16, 16, 16, 32), kappa=0.12, tol=1e-12),
        # The double-precision point-source solve with the default settings.
        _case("solve_f64_8x8x8x8", "solve", (8, 8, 8, 8), kappa=0.12, tol=1e-12, solver="flexible", even_odd=False,
              arith="f64", krylov="f32", source="point"),
        # The mixed-precision solve of the paper's lattice with the settings
        # that are fastest on this card: even-odd, binary16 inner vectors,
        # double-FP32 refreshes.
        _case("solve_mixed_24x24x24x32", "solve", (24, 24, 24, 32), links="haar", kappa=0.125, tol=1e-10,
              solver="reliable", even_odd=True, arith="df32", krylov="f16", source="z2"),
        # A propagator: twelve point sources of one configuration in one
        # batched call; propagators are kept in single precision.
        _case("propagator_16x16x16x32", "batch", (16, 16, 16, 32), rhs=12, tol=1e-10, krylov="f32"),
    ]


def _extents(rng, lo, hi, step, least=2):
    """Four extents, multiples of step and at least `least`, whose volume is
    spread over [lo, hi] on the logarithm; t is the longest as a rule."""
    target = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    side = target ** 0.25
    while True:
        d = [max(least, step * max(1, round(side * math.exp(rng.uniform(-0.35, 0.35)) / step))) for _ in range(4)]
        if rng.random() < 0.7:
            d.sort()
        if 0.7 * lo <= d[0] * d[1] * d[2] * d[3] <= hi:
            return tuple(d)


def draw(rng):
    kind = rng.choice(["normal", "normal", "normal", "multi", "schur_multi", "ras", "config", "force", "solve",
                       "solve", "batch"])
    kw = {"links": rng.choice(["exp", "haar"]), "eps": round(rng.uniform(0.15, 0.4), 3),
          "csw": round(rng.uniform(0.8, 1.4), 3), "kappa": round(rng.uniform(0.110, 0.122), 4)}
    if kind == "normal":
        kw["prec"] = rng.choice(["f32", "f32", "f16", "f64"])
        if kw["prec"] == "f64":
            kw["arith"] = rng.choice(["f64", "df32"])
            dims = _extents(rng, 256, 200000, 1)
        else:
            dims = _extents(rng, 256, 1500000, 1)
    elif kind == "multi":
        kw.update(prec="f32", rhs=rng.randint(2, 16))
        dims = _extents(rng, 1000, 400000, 1)
    elif kind == "schur_multi":
        kw.update(prec=rng.choice(["f32", "f16"]), rhs=rng.randint(2, 16))
        dims = _extents(rng, 1000, 200000, 2)
    elif kind == "ras":
        kw.update(prec=rng.choice(["f32", "f16"]), schur=rng.random() < 0.4, mr=rng.randint(2, 5))
        dims = _extents(rng, 8192, 200000, 4, 8)
    elif kind == "config":
        dims = _extents(rng, 1000, 200000, 2)
    elif kind == "force":
        kw.update(tol=1e-12, kappa=round(rng.uniform(0.105, 0.115), 4))
        dims = _extents(rng, 1000, 40000, 2)
    elif kind == "solve":
        kw.update(tol=1e-11, kappa=round(rng.uniform(0.105, 0.115), 4), solver=rng.choice(["flexible", "reliable", "nested"]),
                  even_odd=rng.random() < 0.7, arith=rng.choice(["f64", "df32"]), krylov=rng.choice(["f32", "f16"]),
                  source=rng.choice(["point", "z2", "gaussian"]))
        dims = _extents(rng, 1000, 60000, 2)
    else:
        kw.update(tol=1e-10, kappa=round(rng.uniform(0.105, 0.115), 4), rhs=rng.randint(2, 14),
                  krylov=rng.choice(["f32", "f16"]))
        dims = _extents(rng, 1000, 40000, 2)
    c = _case("", kind, dims, **kw)
    del c["name"]
    return c


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _dims(case):
    return case["lx"], case["ly"], case["lz"], case["lt"]


def _volume(case):
    return case["lx"] * case["ly"] * case["lz"] * case["lt"]


def _normal(shape, gen):
    return torch.randn(shape, generator=gen, device=DEV, dtype=torch.float64)


def _mul3(a, b):
    return a[..., :, 0:1] * b[..., 0:1, :] + a[..., :, 1:2] * b[..., 1:2, :] + a[..., :, 2:3] * b[..., 2:3, :]


def _links(case, gen):
    """U[V,4,3,3]: exp(i eps H) with Gaussian traceless Hermitian H, or Haar
    (Gram-Schmidt of complex Gaussian rows)."""
    n = _volume(case) * 4
    if case["links"] == "haar":
        a = torch.complex(_normal((n, 2, 3), gen), _normal((n, 2, 3), gen))
        r0 = a[:, 0] / torch.linalg.vector_norm(a[:, 0], dim=-1, keepdim=True)
        r1 = a[:, 1] - (r0.conj() * a[:, 1]).sum(-1, keepdim=True) * r0
        r1 = r1 / torch.linalg.vector_norm(r1, dim=-1, keepdim=True)
        u = torch.stack([r0, r1, torch.linalg.cross(r0, r1).conj()], 1)
    else:
        w = _normal((n, 8), gen)
        z = torch.zeros_like(w[:, 0])
        s = w[:, 7] / math.sqrt(3)
        h = torch.stack([torch.complex(w[:, 2] + s, z), torch.complex(w[:, 0], -w[:, 1]),
                         torch.complex(w[:, 3], -w[:, 4]), torch.complex(w[:, 0], w[:, 1]),
                         torch.complex(s - w[:, 2], z), torch.complex(w[:, 5], -w[:, 6]),
                         torch.complex(w[:, 3], w[:, 4]), torch.complex(w[:, 5], w[:, 6]),
                         torch.complex(-2 * s, z)], -1).reshape(n, 3, 3)
        x = (0.5j * case["eps"] / 16) * h
        one = torch.eye(3, device=DEV, dtype=C128)
        u = one + x / 10
        for k in range(9, 0, -1):   # Horner form of the exponential series
            u = one + _mul3(x, u) / k
        for _ in range(4):          # exp(x)^16
            u = _mul3(u, u)
    return u.reshape(_volume(case), 4, 3, 3).contiguous()


def _source(case, gen, kind, which):
    v = _volume(case)
    if kind == "point":
        psi = torch.zeros((v, 4, 3), device=DEV, dtype=C128)
        at = int(torch.randint(v, (1,), generator=gen, device=DEV).item()) if which < 0 else 0
        psi.view(v, 12)[at, max(which, 0) % 12] = 1
        return psi
    if kind == "z2":
        return (2.0 * torch.randint(2, (v, 4, 3), generator=gen, device=DEV) - 1.0).to(C128)
    return torch.complex(_normal((v, 4, 3), gen), _normal((v, 4, 3), gen))


def _inputs(case, seed):
    """Links and sources, from the seed alone."""
    gen = torch.Generator(device=DEV)
    gen.manual_seed(seed)
    u = _links(case, gen)
    if case["kind"] == "solve":
        psi = [_source(case, gen, case["source"], -1)]
    elif case["kind"] == "batch":
        psi = [_source(case, gen, "point", r) for r in range(case["rhs"])]
    else:
        psi = [_source(case, gen, "gaussian", 0) for _ in range(case.get("rhs", 1))]
    return u, psi


def _field_prec(case):
    return PREC[case.get("prec", "f64")]


class _State:
    pass


def prepare(case, seed):
    s = _State()
    u, psi = _inputs(case, seed)
    kind, v = case["kind"], _volume(case)
    s.case = case
    s.lat = lat = wc.Lattice(_dims(case))
    lat.load_gauge(u).load_clover(case["csw"], case["kappa"])
    if case.get("arith") == "df32":
        lat.set_fp64_arith(wc.ARITH_DF32)
    prec = _field_prec(case)
    n = len(psi)
    s.ins = [lat.field(prec).load(p) for p in psi]
    s.outs = [lat.field(prec) for _ in range(n)]
    dtype = C128 if prec == wc.F64 and kind != "batch" else torch.complex64
    if kind in ("normal", "multi", "schur_multi"):
        s.mid = [lat.field(prec) for _ in range(n)]
    if kind == "config":
        s.u = u                    # the next configuration, in the caller's memory
    if kind == "force":
        s.force = torch.empty((v, 4, 3, 3), device=DEV, dtype=C128)
        s.params = wc.solve_params(tol=case["tol"], solver=wc.SOLVER_RELIABLE, even_odd=True)
    elif kind == "solve":
        s.params = wc.solve_params(
            tol=case["tol"], even_odd=case["even_odd"], krylov_prec=PREC[case["krylov"]],
            solver={"flexible": wc.SOLVER_FLEXIBLE, "reliable": wc.SOLVER_RELIABLE,
                    "nested": wc.SOLVER_NESTED}[case["solver"]])
    elif kind == "batch":
        s.params = wc.solve_params(tol=case["tol"], solver=wc.SOLVER_RELIABLE, even_odd=True,
                                   krylov_prec=PREC[case["krylov"]])
    if kind != "force":
        s.result = torch.empty((n, v, 4, 3), device=DEV, dtype=dtype)
    return s


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------

def run(s):
    case, lat, kind = s.case, s.lat, s.case["kind"]
    if kind == "normal":
        lat.apply_M(s.mid[0], s.ins[0])
        lat.apply_Mdag(s.outs[0], s.mid[0])
    elif kind == "multi":
        lat.apply_multi(s.mid, s.ins)
        lat.apply_multi(s.outs, s.mid, dagger=True)
    elif kind == "schur_multi":
        lat.apply_schur_multi(s.mid, s.ins)
        lat.apply_schur_multi(s.outs, s.mid, dagger=True)
    elif kind == "ras":
        if case["schur"]:
            lat.ras_schur(s.outs[0], s.ins[0], mr_iters=case["mr"])
        else:
            lat.ras(s.outs[0], s.ins[0], mr_iters=case["mr"])
    elif kind == "config":
        lat.load_gauge(s.u).load_clover(case["csw"], case["kappa"])
        lat.apply_schur(s.outs[0], s.ins[0])
    elif kind == "force":
        return {"S": lat.action_force(s.ins[0], s.force, s.params), "F": s.force}
    elif kind == "solve":
        s.outs[0].copy_from(s.ins[0], 0.0)      # start from zero
        lat.solve(s.outs[0], s.ins[0], s.params)
    else:
        for x, b in zip(s.outs, s.ins):
            x.copy_from(b, 0.0)
        wc.solve_batch([lat] * len(s.ins), s.outs, s.ins, s.params)
    for f, out in zip(s.outs, s.result):
        f.store_async(out)
    if case.get("prec") == "f16":
        # a program that stores its vectors in binary16 keeps the result so
        return torch.view_as_real(s.result).half()
    return s.result


def work(case):
    """Inputs read once, results written once; the links as two rows and the
    packed clover term in the operator's storage precision.  A solve is
    counted as the reading of its system and the writing of its solution, and
    one operator application."""
    kind, v, n = case["kind"], _volume(case), case.get("rhs", 1)
    width = {"f64": 8, "f32": 4, "f16": 2}[case.get("prec", "f64")]
    shared = (48 + 72) * width * v                     # 4 links of 12 reals, 72 clover reals
    spinor = 24 * width * v
    result = {"f64": 192, "f32": 96, "f16": 48}[case.get("prec", "f64")] * v
    flops = 1824 * v
    if kind in ("normal", "multi"):                    # two applications, then the export
        return {"bytes": 2 * (shared + 2 * n * spinor) + n * (spinor + result), "flops": 2 * n * flops}
    if kind == "schur_multi":                          # even sites only are vectors; the export is whole
        return {"bytes": 2 * (shared + n * spinor) + n * (spinor + result), "flops": 2 * n * flops}
    if kind == "ras":                                  # one pass over the blocks per MR step
        return {"bytes": shared + 3 * spinor + result, "flops": case["mr"] * flops}
    if kind == "config":
        # in: 4 links of 18 reals, a vector; out: links, clover and its inverse
        # in double precision, a vector; 6 planes with 4 leaves of 3x3 products
        return {"bytes": v * (576 + 384 + 2 * 576 + 192 + 192), "flops": v * (6 * 8 * 198 + 2 * 1824)}
    if kind == "force":
        return {"bytes": v * (192 + 576 + 576 + 576), "flops": 2 * flops + 4 * v * 48 * 198}
    return {"bytes": v * (384 + 576) + n * v * (192 + 192), "flops": 2 * n * flops}


# ---------------------------------------------------------------------------
# the same results in complex128 from the definition
# ---------------------------------------------------------------------------

_PLANES = ((0, 1), (0, 2), (0, 3), (1, 2), (1, 3), (2, 3))


def _gammas():
    s = [torch.tensor(m, dtype=C128, device=DEV) for m in
         ([[0, 1], [1, 0]], [[0, -1j], [1j, 0]], [[1, 0], [0, -1]], [[1, 0], [0, 1]])]
    g = []
    for k in range(4):
        m = torch.zeros((4, 4), dtype=C128, device=DEV)
        m[:2, 2:] = 1j * s[k] if k < 3 else s[k]
        m[2:, :2] = -1j * s[k] if k < 3 else s[k]
        g.append(m)
    return g


def _matvec(u, h):
    """u (3x3) times every colour vector of h[..., spin, 3]."""
    u = u.unsqueeze(-3)
    return u[..., 0] * h[..., 0:1] + u[..., 1] * h[..., 1:2] + u[..., 2] * h[..., 2:3]


def _dag(u):
    return u.conj().transpose(-1, -2)


def _spin(m, psi):
    return torch.einsum("st,...tc->...sc", m, psi)


class _Operator:
    """M, its parts and its adjoint on fields of shape grid + (4, 3); the
    grid is (t, z, y, x), with any number of leading batch dimensions where
    `open` drops the hops over the boundary (an isolated block)."""

    def __init__(self, u, csw, kappa, phase=None, fields=None, open=False):
        self.u, self.kappa, self.ck, self.open = u, kappa, csw * kappa, open
        self.gamma = _gammas()
        self.phase = phase      # of the forward hop in t, per site
        self.f = self._field_strengths() if fields is None else fields
        self.inverse = None

    def _shift(self, a, mu, d, inner):
        """a at x + d mu."""
        dim = a.dim() - inner - 1 - mu
        out = torch.roll(a, -d, dim)
        if self.open:
            out = out.clone()
            out.select(dim, a.shape[dim] - 1 if d > 0 else 0).zero_()
        return out

    def _field_strengths(self):
        out = []
        sh = lambda a, mu, d: self._shift(a, mu, d, 2)  # noqa: E731
        for mu, nu in _PLANES:
            um, un = self.u[..., mu, :, :], self.u[..., nu, :, :]
            # plaquette at x; the leaves at x of its three neighbours are
            # theirs carried to their corner x
            p = _mul3(_mul3(um, sh(un, mu, 1)), _mul3(_dag(sh(um, nu, 1)), _dag(un)))
            far = _mul3(un, sh(um, nu, 1))
            q = p + sh(_mul3(_mul3(_dag(um), p), um), mu, -1) + sh(_mul3(_mul3(_dag(un), p), un), nu, -1)
            q = q + sh(sh(_mul3(_mul3(_dag(far), p), far), mu, -1), nu, -1)
            anti = q - _dag(q)
            tr = anti.diagonal(dim1=-2, dim2=-1).sum(-1) / 3
            out.append((anti - tr[..., None, None] * torch.eye(3, device=DEV, dtype=C128)) / 8)
        return out

    def hop(self, psi, sign=1):
        """H psi (sign 1) or H^+ psi (sign -1)."""
        acc = torch.zeros_like(psi)
        one = torch.eye(4, device=DEV, dtype=C128)
        for mu in range(4):
            um = self.u[..., mu, :, :]
            if mu == 3 and self.phase is not None:
                um = um * self.phase[..., None, None]
            fwd = self._shift(psi, mu, 1, 2)
            acc = acc + _matvec(um, _spin(one - sign * self.gamma[mu], fwd))
            bwd = _matvec(_dag(um), _spin(one + sign * self.gamma[mu], psi))
            acc = acc + self._shift(bwd, mu, -1, 2)
        return acc

    def _sigma(self, p):
        mu, nu = _PLANES[p]
        g = self.gamma
        return 0.5j * (g[mu] @ g[nu] - g[nu] @ g[mu])

    def clover(self, psi):
        """(1 + T) psi."""
        acc = psi
        for p in range(6):
            acc = acc + 1j * self.ck * _spin(self._sigma(p), _matvec(self.f[p], psi))
        return acc

    def clover_inverse(self, psi):
        if self.inverse is None:
            grid = self.f[0].shape[:-2]
            a = torch.zeros(grid + (4, 3, 4, 3), device=DEV, dtype=C128)
            for p in range(6):
                a += 1j * self.ck * torch.einsum("st,...ab->...satb", self._sigma(p), self.f[p])
            a = a.reshape(grid + (12, 12)) + torch.eye(12, device=DEV, dtype=C128)
            self.inverse = torch.linalg.inv(a)
        return (self.inverse @ psi.reshape(psi.shape[:-2] + (12, 1))).reshape(psi.shape)

    def m(self, psi, sign=1):
        return self.clover(psi) - self.kappa * self.hop(psi, sign)

    def schur(self, psi, even, sign=1):
        """The Schur complement on the even sites (even: mask)."""
        x = psi * even
        t = self.clover_inverse(self.hop(x, sign)) * ~even
        return (self.clover(x) - self.kappa ** 2 * self.hop(t, sign)) * even


def _grid(case):
    return (case["lt"], case["lz"], case["ly"], case["lx"])


def _even(case):
    g = _grid(case)
    c = sum(torch.arange(n, device=DEV).reshape([-1 if k == d else 1 for k in range(4)]) for d, n in enumerate(g))
    return ((c % 2) == 0)[..., None, None]


def _operator(case, u):
    g = _grid(case)
    phase = torch.ones(g, device=DEV, dtype=torch.float64)
    phase[-1] = -1.0                      # antiperiodic in time
    return _Operator(u.reshape(g + (4, 3, 3)), case["csw"], case["kappa"], phase)


def _vdot(a, b):
    return torch.vdot(a.reshape(-1), b.reshape(-1))


def _bicgstab(op, b, tol=3e-15):
    """Solution of op x = b, refined from the true residual until it does not
    get smaller."""
    x, best = torch.zeros_like(b), math.inf
    scale = torch.linalg.vector_norm(b).item()
    for _ in range(6):
        r = b - op(x)
        now = torch.linalg.vector_norm(r).item() / scale
        if now < tol or now > 0.5 * best:
            break
        best = now
        d, shadow, p = torch.zeros_like(b), r.clone(), r.clone()
        rho = _vdot(shadow, r)
        for _ in range(3000):
            v = op(p)
            alpha = rho / _vdot(shadow, v)
            q = r - alpha * v
            t = op(q)
            omega = _vdot(t, q) / _vdot(t, t)
            d = d + alpha * p + omega * q
            r = q - omega * t
            size = torch.linalg.vector_norm(r).item() / scale
            if not size > max(1e-8 * now, 0.3 * tol):
                break
            new = _vdot(shadow, r)
            p = r + (new / rho) * (alpha / omega) * (p - omega * v)
            rho = new
        x = x + d
    return x


def _exact_ras(case, op, psi):
    """MR from zero on every extended block (core 4^4, one site per face),
    hops that leave the block dropped; the cores of the block solutions."""
    b, o = 4, 1
    g = _grid(case)
    e = b + 2 * o
    v = _volume(case)
    start = torch.cartesian_prod(*[torch.arange(0, n, b, device=DEV) for n in g])      # [B, 4], t z y x
    local = torch.cartesian_prod(*[torch.arange(e, device=DEV) for _ in range(4)])
    size = torch.tensor(g, device=DEV)
    even = _even(case).reshape(-1)
    flat = lambda a, inner: a.reshape((v,) + a.shape[a.dim() - inner:])  # noqa: E731
    u, f = flat(op.u, 3), [flat(a, 2) for a in op.f]
    phase, src = op.phase.reshape(-1), psi.reshape(v, 4, 3)
    out = torch.zeros_like(src)
    core = ((local >= o) & (local < o + b)).all(-1)
    for k in range(0, len(start), 256):
        c = (start[k:k + 256, None] + local[None] - o) % size
        at = ((c[..., 0] * g[1] + c[..., 1]) * g[2] + c[..., 2]) * g[3] + c[..., 3]       # [B, e^4]
        shape = (at.shape[0], e, e, e, e)
        blk = _Operator(u[at].reshape(shape + (4, 3, 3)), case["csw"], case["kappa"], phase[at].reshape(shape),
                        [a[at].reshape(shape + (3, 3)) for a in f], open=True)
        r = src[at].reshape(shape + (4, 3))
        mask = even[at].reshape(shape)[..., None, None]
        if case["schur"]:
            r = r * mask
        x = torch.zeros_like(r)
        for _ in range(case["mr"]):
            q = blk.schur(r, mask) if case["schur"] else blk.m(r)
            dims = (1, 2, 3, 4, 5, 6)
            qq = (q.abs() ** 2).sum(dims, keepdim=True)
            alpha = (q.conj() * r).sum(dims, keepdim=True) / qq
            x = x + alpha * r
            r = r - alpha * q
        sel = core.expand(at.shape[0], -1)
        out[at[sel]] = x.reshape(at.shape + (4, 3))[sel]
    return out


def _exact_force(case, u, phi):
    op = _operator(case, u)
    y = _bicgstab(lambda a: op.m(a, -1), phi)
    x = _bicgstab(op.m, y)
    leaf = u.detach().clone().requires_grad_(True)
    var = _operator(case, leaf)
    (-2 * _vdot(y, var.m(x)).real).backward()
    g = _mul3(u, _dag(leaf.grad))
    anti = (g - _dag(g)) / 2
    tr = anti.diagonal(dim1=-2, dim2=-1).sum(-1) / 3
    return {"S": float(_vdot(y, y).real), "F": anti - tr[..., None, None] * torch.eye(3, device=DEV, dtype=C128)}


def exact(case, seed):
    u, psi = _inputs(case, seed)
    g, kind = _grid(case), case["kind"]
    psi = [p.reshape(g + (4, 3)) for p in psi]
    if kind == "force":
        return _exact_force(case, u, psi[0])
    op = _operator(case, u)
    if kind in ("normal", "multi"):
        res = [op.m(op.m(p), -1) for p in psi]
    elif kind == "schur_multi":
        even = _even(case)
        res = [op.schur(op.schur(p, even), even, -1) for p in psi]
    elif kind == "config":
        res = [op.schur(psi[0], _even(case))]
    elif kind == "ras":
        res = [_exact_ras(case, op, psi[0])]
    else:
        res = [_bicgstab(op.m, p) for p in psi]
    out = torch.stack([r.reshape(_volume(case), 4, 3) for r in res])
    return torch.view_as_real(out) if case.get("prec") == "f16" else out
