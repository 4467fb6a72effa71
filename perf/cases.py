"""What the Wilson-Dirac library is timed on.

A user loads one gauge field and then applies the operator (dslash, M, M_hat,
also to many sources in one launch) or solves M_kappa x = b on it: one source,
many sources, several masses, from device or from host fields.  The cases are
those calls in every storage precision, link storage and gauge option that the
solvers and the benchmark use, from 8^3x16 (a call is launch latency) to
64^3x128 (fields far beyond L2).

Every case has a "kind":
  dslash       out = D in, one parity to the other
  apply        out = M_hat in (which = 1, even sites) or M in (which = 0, both parities)
  dslash_batch D on many sources in one launch
  solve        device-resident M_kappa x = b, BiCGstab or CGNR, any inner precision
  solve_host   the same from page-locked host arrays in the host layout
  batch        the spin-colour point sources of a propagator, solved together
  multishift   one source, several kappa
16-bit results come back as the stored numbers and the site norms; Q16, whose
stored numbers are integers, is measured inside the solves that use it.
"""
import math

import torch

import paper_0911_3191_gb300 as wd

F64, F32, Q16, H16N, B16N = wd.F64, wd.F32, wd.Q16, wd.H16N, wd.B16N
EPS = 0.3  # link disorder of the benchmark's fields
TOL = 1e-12  # true residual of every solve
LINK_BYTES = {F32: 48, Q16: 24, H16N: 24, B16N: 24}
SPINOR_BYTES = {F64: 192, F32: 96, Q16: 52, H16N: 52, B16N: 52}


def _case(kind, dims, prec, **kw):
    x, y, z, t = dims
    c = {"kind": kind, "x": x, "y": y, "z": z, "t": t, "prec": prec, "recon": 18, "temporal": True, "anti": False,
         "dagger": False}
    c.update(kw)
    return c


def listed():
    general = {"temporal": False}
    cases = {
        # a call on the smallest lattice of the tests and examples: launch latency and the host path
        "dslash_f64_8x16": _case("dslash", (8, 8, 8, 16), F64, **general),
        # the reliable update's matrix product at the benchmark's lattice and link format
        "dslash_f64_24x64": _case("dslash", (24, 24, 24, 64), F64),
        # FP64 M_hat^dag on an uneven lattice, compressed general links, antiperiodic time
        "mhat_dag_f64_ragged": _case("apply", (20, 14, 22, 38), F64, which=1, dagger=True, recon=12, anti=True,
                                     **general),
        # FP32 operator at the serving engine's largest lattice
        "dslash_f32_48x96": _case("dslash", (48, 48, 48, 96), F32, recon=12, **general),
        # 16-bit operator on the largest lattice of the bandwidth sweep
        "dslash_b16n_64x128": _case("dslash", (64, 64, 64, 128), B16N, recon=12, **general),
        # the twelve sources of a propagator through one 16-bit launch
        "dslash_batch_h16n_24x64": _case("dslash_batch", (24, 24, 24, 64), H16N, nrhs=12),
        # a small solve, as in tuning runs and unit tests: one iteration is a few launches
        "solve_q16_8x16": _case("solve", (8, 8, 8, 16), Q16, kappa=0.12, solver=0),
        # the benchmark's solve: 16-bit inner BiCGstab with FP64 reliable updates
        "solve_q16_24x64": _case("solve", (24, 24, 24, 64), Q16, kappa=0.124, solver=0),
        # the pure FP64 solve that the mixed one is measured against
        "solve_f64_24x64": _case("solve", (24, 24, 24, 64), F64, kappa=0.124, solver=0),
        # host arrays in and out, normal equations, FP32 inner, general links, uneven lattice
        "solve_host_cgnr_f32_ragged": _case("solve_host", (16, 12, 20, 36), F32, kappa=0.12, solver=1, recon=12,
                                            **general),
        # a propagator: twelve point sources on one gauge field
        "batch_q16_16x32": _case("batch", (16, 16, 16, 32), Q16, kappa=0.12, nrhs=12),
        # several masses for one source
        "multishift_q16_24x32": _case("multishift", (24, 24, 24, 32), Q16, kappa=0.122, nkappa=3),
    }
    return [dict(c, name=name) for name, c in cases.items()]


def _draw_dims(rng, lo, hi):
    """Even, mostly unequal extents with lo <= volume <= hi, the volume spread over its logarithm."""
    while True:
        v = math.exp(rng.uniform(math.log(lo), math.log(hi)))
        side = v ** 0.25
        x, y, z = (2 * max(1, round(0.5 * side * math.exp(rng.uniform(-0.45, 0.3)))) for _ in range(3))
        t = 2 * max(1, round(0.5 * v / (x * y * z)))
        if t <= 128 and lo <= x * y * z * t <= hi:
            return x, y, z, t


def draw(rng):
    kind = rng.choice(["dslash", "dslash", "apply", "dslash_batch", "solve", "solve", "solve_host", "batch",
                       "multishift"])
    kw = {"recon": rng.choice([12, 18]), "temporal": rng.random() < 0.5, "anti": rng.random() < 0.3}
    if kind in ("dslash", "apply"):
        prec = rng.choice([F64, F64, F32, H16N, B16N])
        dims = _draw_dims(rng, 2048, 1 << 20 if prec == F64 else 1 << 23)
        kw["dagger"] = rng.random() < 0.5
        if kind == "apply":
            kw["which"] = rng.choice([0, 1])
        return _case(kind, dims, prec, **kw)
    if kind == "dslash_batch":
        return _case(kind, _draw_dims(rng, 2048, 1 << 19), rng.choice([F32, H16N, B16N]), nrhs=rng.choice([2, 5, 12]),
                     **kw)
    kw["kappa"] = round(rng.uniform(0.105, 0.122), 4)
    if kind == "batch":
        return _case(kind, _draw_dims(rng, 2048, 1 << 17), rng.choice([Q16, F32, B16N]), nrhs=rng.choice([3, 7, 12]),
                     **kw)
    if kind == "multishift":
        return _case(kind, _draw_dims(rng, 2048, 1 << 18), rng.choice([Q16, F32]), nkappa=rng.choice([2, 3, 4]), **kw)
    kw["solver"] = rng.choice([0, 0, 1])
    return _case(kind, _draw_dims(rng, 2048, 1 << 19), rng.choice([F64, F32, Q16, Q16, H16N, B16N]), **kw)


# ------------------------------------------------------------------ inputs
def _dims(case):
    return case["x"], case["y"], case["z"], case["t"]


def _volume(case):
    return math.prod(_dims(case))


def _generator(seed, stream):
    g = torch.Generator(device="cuda")
    g.manual_seed(1_000_003 * int(seed) + stream)
    return g


def _links(case, seed):
    """Random SU(3) links near the unit matrix, (V, 4, 3, 3, 2) float64: rows a, b of 1 + i EPS H made
    orthonormal, row c = (a x b)^*."""
    v = _volume(case)
    out = torch.empty((v, 4, 3, 3), dtype=torch.complex128, device="cuda")
    gen = _generator(seed, 1)
    step = 1 << 20
    for s in range(0, v, step):
        n = min(step, v - s)
        w = (0.5 * EPS) * torch.randn((8, n, 4), generator=gen, dtype=torch.float64, device="cuda")
        d = w[7] / math.sqrt(3.0)
        one = torch.ones_like(d)
        h01, h02, h12 = torch.complex(w[0], -w[1]), torch.complex(w[3], -w[4]), torch.complex(w[5], -w[6])
        a = torch.stack([torch.complex(one, w[2] + d), 1j * h01, 1j * h02], -1)
        b = torch.stack([1j * h01.conj(), torch.complex(one, d - w[2]), 1j * h12], -1)
        a = a / a.abs().square().sum(-1, keepdim=True).sqrt()
        b = b - (a.conj() * b).sum(-1, keepdim=True) * a
        b = b / b.abs().square().sum(-1, keepdim=True).sqrt()
        o = out[s: s + n]
        o[:, :, 0], o[:, :, 1] = a, b
        for i in range(3):
            j, k = (i + 1) % 3, (i + 2) % 3
            o[:, :, 2, i] = (a[..., j] * b[..., k] - a[..., k] * b[..., j]).conj()
    return torch.view_as_real(out)


def _spinor(case, seed, stream=2):
    """Complex Gaussian source, (V, 4, 3) complex128."""
    g = _generator(seed, stream)
    return torch.view_as_complex(torch.randn((_volume(case), 4, 3, 2), generator=g, dtype=torch.float64,
                                             device="cuda"))


def _sources(case, seed):
    """The right-hand sides of a case, as (V, 4, 3) fields in the host layout."""
    if case["kind"] == "batch":  # point sources at the origin, one per spin and colour
        out = []
        for r in range(case["nrhs"]):
            b = torch.zeros((_volume(case), 4, 3), dtype=torch.complex128, device="cuda")
            b[0, r // 3, r % 3] = 1.0
            out.append(b)
        return out
    n = case["nrhs"] if case["kind"] == "dslash_batch" else 1
    return [_spinor(case, seed, 2 + r) for r in range(n)]


def _kappas(case):
    """Several masses: kappa and lighter hopping, as in a mass scan."""
    return [case["kappa"] - 0.004 * k for k in range(case["nkappa"])]


def _views(buf, ctx, prec, nfields):
    """Stored numbers of `nfields` single-parity fields as tensors: [field, array, site, value], norms [field, site]."""
    vh = ctx.volume // 2
    stride = (vh + 31) // 32 * 32
    fields = buf.view(nfields, ctx.field_bytes(prec))
    if prec in (F64, F32):
        dtype, arrays, values = (torch.float64, 12, 2) if prec == F64 else (torch.float32, 6, 4)
        return fields.view(dtype)[:, : stride * arrays * values].view(nfields, arrays, stride, values)[:, :, :vh]
    codes = fields[:, : 48 * stride].view(torch.float16 if prec == H16N else torch.bfloat16)
    off = (48 * stride + 255) // 256 * 256
    norms = fields[:, off: off + 4 * stride].view(torch.float32)
    return {"numbers": codes.view(nfields, 3, stride, 8)[:, :, :vh], "norms": norms[:, :vh]}


def _field(ctx, prec, nfields):
    return torch.zeros(nfields * ctx.field_bytes(prec), dtype=torch.uint8, device="cuda")


def prepare(case, seed):
    ctx = wd.WilsonDirac(_dims(case), t_antiperiodic=case["anti"])
    ctx.load_gauge(_links(case, seed), recon=case["recon"], temporal_gauge=case["temporal"])
    kind, prec = case["kind"], case["prec"]
    s = {"case": case, "ctx": ctx, "kind": kind, "prec": prec, "dagger": case["dagger"]}
    src = _sources(case, seed)
    if kind in ("dslash", "dslash_batch"):
        fb = ctx.field_bytes(prec)
        s["in"], s["out"] = _field(ctx, prec, len(src)), _field(ctx, prec, len(src))
        for r, b in enumerate(src):
            ctx.field_import(s["in"][r * fb: (r + 1) * fb], b, wd.ODD, prec)
        s["result"] = _views(s["out"], ctx, prec, len(src))
    elif kind == "apply":
        n, fb = (1, 2)[case["which"] == 0], ctx.field_bytes(prec)
        s["in"], s["out"] = _field(ctx, prec, n), _field(ctx, prec, n)
        for p in range(n):
            ctx.field_import(s["in"][p * fb: (p + 1) * fb], src[0], p, prec)
        s["which"], s["kappa"] = (wd.M_FULL, wd.M_SCHUR_EVEN)[case["which"]], 0.12
        s["result"] = _views(s["out"], ctx, prec, n)
    elif kind == "solve_host":
        s["b"] = torch.empty(src[0].shape, dtype=src[0].dtype, pin_memory=True)
        s["b"].copy_(src[0])
        s["x"] = torch.zeros(src[0].shape, dtype=src[0].dtype, pin_memory=True)
        s["result"] = s["x"]
    else:
        fb, n = ctx.field_bytes(F64), len(_kappas(case)) if kind == "multishift" else len(src)
        s["b"], s["x"] = _field(ctx, F64, 2 * len(src)), _field(ctx, F64, 2 * n)
        for r, b in enumerate(src):
            for p in range(2):
                ctx.field_import(s["b"][(2 * r + p) * fb: (2 * r + p + 1) * fb], b, p, F64)
        s["kappas"] = _kappas(case) if kind == "multishift" else [case["kappa"]] * n
        s["result"] = _views(s["x"], ctx, F64, 2 * n)
    torch.cuda.synchronize()
    return s


def run(s):
    ctx, kind = s["ctx"], s["kind"]
    if kind == "dslash":
        ctx.dslash(s["out"], s["in"], wd.EVEN, s["dagger"], s["prec"])
    elif kind == "apply":
        ctx.apply_M(s["out"], s["in"], s["kappa"], s["which"], s["dagger"], s["prec"])
    elif kind == "dslash_batch":
        ctx.dslash_batch(s["out"], s["in"], s["case"]["nrhs"], wd.EVEN, s["dagger"], s["prec"])
    elif kind == "batch":
        ctx.solve_batch_device(s["x"], s["b"], s["kappas"], tol=TOL, inner_precision=s["prec"], check=False)
    elif kind == "multishift":
        ctx.solve_multishift_device(s["x"], s["b"], s["kappas"], tol=TOL, inner_precision=s["prec"], check=False)
    else:
        f = ctx.solve if kind == "solve_host" else ctx.solve_device
        f(s["x"], s["b"], s["case"]["kappa"], tol=TOL, solver=s["case"]["solver"], inner_precision=s["prec"],
          check=False)
    return s["result"]


# -------------------------------------------------------------------- work
def _link_bytes(case, prec):
    """Bytes of the links of one parity's output sites, each link once: 8 a site, or 6 in the temporal gauge."""
    per = 8 * case["recon"] if prec == F64 else LINK_BYTES[prec]
    return (6 if case["temporal"] else 8) * per * (_volume(case) // 2)


def _dslash_flops(case):
    """1320 a site (Sec. 4.3 of the paper), less the two temporal SU(3) products in the temporal gauge."""
    return (1056 if case["temporal"] else 1320) * (_volume(case) // 2)


def _iterations(case, kappa):
    """BiCGstab iterations to 1e-12 on these fields (37 at kappa 0.12, 51 at 0.124); CGNR takes about twice as many."""
    n = 4.31 / (1.0 - 8.0 * kappa + 0.0766)
    return (2 if case.get("solver") == 1 else 1) * n


def work(case):
    kind, prec = case["kind"], case["prec"]
    vh = _volume(case) // 2
    links, flops = _link_bytes(case, prec), _dslash_flops(case)
    if kind in ("dslash", "dslash_batch"):
        n = case.get("nrhs", 1)
        return {"bytes": links + n * 2 * SPINOR_BYTES[prec] * vh, "flops": n * flops}
    if kind == "apply":  # the links of both parities are the same 8 a site
        n = 2 if case["which"] == 0 else 1
        return {"bytes": links + n * 2 * SPINOR_BYTES[prec] * vh, "flops": 2 * (flops + 48 * vh)}
    # solves: four inner dslashes an iteration; the systems of a batch share the links, the masses of a
    # multi-shift solve the whole iteration
    n = case["nrhs"] if kind == "batch" else 1
    its = _iterations(case, case["kappa"])
    return {"bytes": its * 4 * (links + n * 2 * SPINOR_BYTES[prec] * vh), "flops": its * 4 * n * flops}


# ------------------------------------------------------------------- exact
# The same in complex128 torch, in the basis with diagonal gamma_4 that device fields hold: psi = S psi_host.
_S = [[0, 1, 0, 1], [-1, 0, -1, 0], [0, 1, 0, -1], [-1, 0, 1, 0]]
_GAMMA = [  # gamma_mu psi, by row: (column, factor)
    [(3, 1j), (2, 1j), (1, -1j), (0, -1j)],
    [(3, 1), (2, -1), (1, -1), (0, 1)],
    [(2, 1j), (3, -1j), (0, -1j), (1, 1j)],
    [(0, 1), (1, 1), (2, -1), (3, -1)],
]


def _rotate(m, psi):
    """m psi over colour: (..., 3, 3) on (..., spin, 3)."""
    return (m.unsqueeze(-3) * psi.unsqueeze(-2)).sum(-1)


class _Lattice:
    def __init__(self, case, seed):
        x, y, z, t = _dims(case)
        self.grid, self.anti = (t, z, y, x), case["anti"]
        self.U = torch.view_as_complex(_links(case, seed)).view(*self.grid, 4, 3, 3)
        self.S = torch.tensor(_S, dtype=torch.complex128, device="cuda") * math.sqrt(0.5)
        self.G = None
        if case["temporal"]:  # device fields hold G psi, G(x, t) = U_4(x, 0) ... U_4(x, t-1)
            self.G = torch.zeros((*self.grid, 3, 3), dtype=torch.complex128, device="cuda")
            self.G[0] = torch.eye(3, dtype=torch.complex128, device="cuda")
            for k in range(1, t):
                self.G[k] = self.G[k - 1] @ self.U[k - 1, :, :, :, 3]
        c = [torch.arange(n, device="cuda") for n in self.grid]
        par = (c[0][:, None, None, None] + c[1][:, None, None] + c[2][:, None] + c[3]) % 2
        self.sites = [torch.nonzero(par.reshape(-1) == p)[:, 0] for p in range(2)]
        self.even = (par == 0)[..., None, None]

    def internal(self, b):
        return torch.einsum("ab,vbc->vac", self.S, b).view(*self.grid, 4, 3)

    def hop(self, psi, mu, forward, sign):
        """(1 + sign gamma_mu) U psi(x + mu), or U^dag psi(x - mu): two spin rows through the link."""
        axis = 3 - mu
        U = self.U[..., mu, :, :]
        if mu == 3:
            keep = 0 if sign > 0 else 2
            h = 2 * psi[..., keep: keep + 2, :]
        else:
            h = torch.stack([psi[..., r, :] + sign * f * psi[..., c, :] for r, (c, f) in
                             enumerate(_GAMMA[mu][:2])], -2)
        if forward:
            h = torch.roll(h, -1, axis)
            edge = -1
        else:
            h = torch.roll(_rotate(U.mH, h), 1, axis)
            edge = 0
        if mu == 3 and self.anti:
            h[edge] = -h[edge]
        if forward:
            h = _rotate(U, h)
        full = torch.zeros_like(psi)
        if mu == 3:
            full[..., keep: keep + 2, :] = h
            return full
        full[..., :2, :] = h
        for r in (2, 3):  # P = 1 + sign gamma: its lower rows are sign gamma times the upper ones
            c, f = _GAMMA[mu][r]
            full[..., r, :] = sign * f * h[..., c, :]
        return full

    def D(self, psi, dagger=False):
        out = torch.zeros_like(psi)
        for mu in range(4):
            for forward in (True, False):
                out += self.hop(psi, mu, forward, -1 if forward != dagger else 1)
        return out

    def solve(self, b, kappa):
        """M_kappa x = b by BiCGstab on the Schur system, restarted from its own residual until nothing is gained."""
        even = self.even.to(b.dtype)

        def schur(v):
            return v - kappa ** 2 * even * self.D(self.D(v))

        bh = even * (b + kappa * self.D((1 - even) * b))
        x, stop = torch.zeros_like(b), 1e-15 * torch.linalg.vector_norm(b)
        for _ in range(3):
            r = bh - schur(x)
            if torch.linalg.vector_norm(r) <= stop:
                break
            goal = torch.maximum(stop, 1e-9 * torch.linalg.vector_norm(r))
            y, r0, p, rho = torch.zeros_like(b), r.clone(), r.clone(), None
            rho = torch.sum(r0.conj() * r)
            for _ in range(400):
                v = schur(p)
                alpha = rho / torch.sum(r0.conj() * v)
                r = r - alpha * v
                q = schur(r)
                omega = torch.sum(q.conj() * r) / torch.sum(q.conj() * q)
                y += alpha * p + omega * r
                r = r - omega * q
                if torch.linalg.vector_norm(r) <= goal:
                    break
                new = torch.sum(r0.conj() * r)
                p = r + (new / rho) * (alpha / omega) * (p - omega * v)
                rho = new
            x = x + y
        return x + (1 - even) * (b + kappa * self.D(x))

    def stored(self, psi, parity, prec):
        """A field as _views gives it for one parity."""
        if self.G is not None:
            psi = _rotate(self.G, psi)
        v = torch.view_as_real(psi.reshape(-1, 12)[self.sites[parity]]).reshape(-1, 24)
        if prec in (F64, F32):
            return v.view(v.shape[0], -1, 2 if prec == F64 else 4).transpose(0, 1)
        norm = v.abs().amax(1)
        return {"numbers": (v / norm[:, None]).view(-1, 3, 8).transpose(0, 1), "norms": norm}


def _stack(fields):
    if isinstance(fields[0], dict):
        return {k: torch.stack([f[k] for f in fields]) for k in fields[0]}
    return torch.stack(fields)


def exact(case, seed):
    lat, kind, prec = _Lattice(case, seed), case["kind"], case["prec"]
    src = [lat.internal(b) for b in _sources(case, seed)]
    if kind in ("dslash", "dslash_batch"):  # from the odd sites to the even ones
        return _stack([lat.stored(lat.D(b, case["dagger"]), 0, prec) for b in src])
    if kind == "apply":
        kappa, b = 0.12, src[0]
        if case["which"] == 0:
            out = b - kappa * lat.D(b, case["dagger"])
            return _stack([lat.stored(out, p, prec) for p in range(2)])
        out = b - kappa ** 2 * lat.D(lat.D(b * lat.even, case["dagger"]), case["dagger"])
        return _stack([lat.stored(out, 0, prec)])
    if kind == "solve_host":
        x = lat.solve(src[0], case["kappa"])
        return torch.einsum("ba,vbc->vac", lat.S, x.reshape(-1, 4, 3)).cpu()
    if kind == "multishift":
        xs = [lat.solve(src[0], k) for k in _kappas(case)]
    else:
        xs = [lat.solve(b, case["kappa"]) for b in src]
    return _stack([lat.stored(x, p, F64) for x in xs for p in range(2)])
