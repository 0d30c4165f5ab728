"""Performance cases of the staggered-fermion library: what a program that uses it has it do.

A case names one public operation (`op`), the lattice (`dims`, "LxxLyxLzxLt"), the precision and
the options that the operation takes.  The operations are the single steps of an RHMC run (the
Dirac operator in its storage kinds, the multi-shift solver, the fermion force, stout smearing and
its chain rule, the gauge force and action) and, as whole calls, a multi-shift solve and one
molecular-dynamics force evaluation.

Inputs: links exp(0.3 i H) with Gaussian traceless Hermitian H (the "expih" links of the
synthetic inputs), Gaussian sources, log-spaced poles from 1e-5 to 10 and residues U(0.1, 1); the
molecular-dynamics cases use the stored 10-pole approximation of x^(-1/4) for m = 0.3.
`exact` is the same arithmetic in plain torch complex128 (gradients by autograd).
"""
import math

import torch

import paper_1801_01473_gb300 as stg
from paper_1801_01473_gb300.rational import load_table

RHO = 0.15    # stout parameter, two steps
STEPS = 2
BETA = 5.6
MD_EPS = 5e-4   # momentum step of a fine inner level of a nested integrator


# ------------------------------------------------------------------ the cases

def listed():
    return [
        # the smallest call: one operator application on canonical fields of the 4^4 check lattice
        {"name": "dslash f64 4^4", "op": "dslash", "dims": "4x4x4x4", "prec": "f64", "recon": 18},
        # the solver's operator in single precision on the 32^4 benchmark lattice, <p, A p> included
        {"name": "normal op f32-12 32^4", "op": "normal_op", "dims": "32x32x32x32", "prec": "f32", "recon": 12, "mass": 0.01},
        # the same in double precision, as pure FP64 solves and residual checks use it
        {"name": "normal op f64-18 24^4", "op": "normal_op", "dims": "24x24x24x24", "prec": "f64", "recon": 18, "mass": 0.02},
        # several pseudofermions at once on 16-bit links, the flat lattice of the uneven batch
        {"name": "dslash 4 rhs bf16 24^3x8", "op": "dslash_multi", "dims": "24x24x24x8", "prec": "bf16", "recon": 12, "nrhs": 4},
        # the benchmark's multi-shift solve: mixed precision, 16 poles, light mass
        {"name": "mscg mixed 32^4", "op": "mscg", "dims": "32x32x32x32", "inner": "f32", "mass": 0.01, "poles": 16},
        # a Metropolis / heatbath solve in pure double precision (the library's default)
        {"name": "mscg f64 16^4", "op": "mscg", "dims": "16x16x16x16", "inner": "", "mass": 0.05, "poles": 12},
        # the fermion force of a 12-pole approximation in double precision
        {"name": "fermion force f64 24^3x32", "op": "fermion_force", "dims": "24x24x24x32", "prec": "f64", "poles": 12, "kind": 0},
        # stout smearing in double precision: the links of every Hamiltonian and heatbath
        {"name": "stout smear f64 16^3x32", "op": "stout_smear", "dims": "16x16x16x32", "prec": "f64"},
        # its chain rule in double-precision molecular dynamics, extents all different
        {"name": "stout chain f64 20x12x28x16", "op": "stout_force", "dims": "20x12x28x16", "prec": "f64", "kind": 0},
        # the gauge force of double-precision molecular dynamics, ragged extents
        {"name": "gauge force f64 18x22x14x26", "op": "gauge_force", "dims": "18x22x14x26", "prec": "f64", "kind": 0},
        # one force evaluation of single-precision molecular dynamics: what a trajectory repeats
        {"name": "md force 32^4", "op": "md_force", "dims": "32x32x32x32", "prec": "f32"},
        # the same on the small lattice that thermalisation runs use
        {"name": "md force 8^4", "op": "md_force", "dims": "8x8x8x8", "prec": "f32"},
    ]


def _dims(rng, lo, hi):
    """Four even extents around one size drawn evenly in its logarithm."""
    base = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    ext = [min(hi, max(4, 2 * round(base * rng.uniform(0.75, 1.33) / 2))) for _ in range(4)]
    return "x".join(str(e) for e in ext)


def draw(rng):
    op = rng.choice(["dslash", "normal_op", "normal_op", "dslash_multi", "mscg", "fermion_force", "stout_smear",
                     "stout_force", "gauge_force", "gauge_action", "md_force"])
    if op == "dslash":
        prec = rng.choice(["f64", "f64", "f32", "ds"])
        return {"op": op, "dims": _dims(rng, 4, 32), "prec": prec, "recon": 18 if prec != "f32" else rng.choice([12, 18])}
    if op == "normal_op":
        prec, recon = rng.choice([("f32", 12), ("f32", 18), ("f64", 18), ("f64", 12), ("f16", 12), ("ds", 18)])
        return {"op": op, "dims": _dims(rng, 6, 32), "prec": prec, "recon": recon, "mass": round(rng.uniform(0.01, 0.3), 3)}
    if op == "dslash_multi":
        prec = rng.choice(["f32", "f32", "bf16", "f16", "f64"])
        return {"op": op, "dims": _dims(rng, 6, 28), "prec": prec, "recon": 18 if prec == "f64" else 12, "nrhs": rng.randint(2, 12)}
    if op == "mscg":
        return {"op": op, "dims": _dims(rng, 6, 20), "inner": rng.choice(["", "f32", "f32", "f16"]),
                "mass": round(math.exp(rng.uniform(math.log(0.03), math.log(0.3))), 3), "poles": rng.randint(4, 16)}
    if op == "fermion_force":
        return {"op": op, "dims": _dims(rng, 6, 28), "prec": rng.choice(["f64", "f32"]), "poles": rng.randint(4, 16), "kind": rng.randint(0, 1)}
    if op in ("stout_smear", "stout_force", "gauge_force"):
        prec = rng.choice(["f64", "f32"])
        c = {"op": op, "dims": _dims(rng, 4, 20 if prec == "f64" else 32), "prec": prec}
        return c if op == "stout_smear" else dict(c, kind=rng.randint(0, 1))
    if op == "gauge_action":
        return {"op": op, "dims": _dims(rng, 4, 26)}
    return {"op": op, "dims": _dims(rng, 6, 24), "prec": rng.choice(["f32", "f32", "f64"])}


# ------------------------------------------------------------------ inputs

def _ext(case):
    return tuple(int(v) for v in case["dims"].split("x"))


def _volume(case):
    return math.prod(_ext(case))


def _mm(a, b):
    """Product of 3x3 matrices over leading axes, entry by entry."""
    return (a[..., :, :, None] * b[..., None, :, :]).sum(-2)


def _dag(a):
    return a.conj().transpose(-1, -2)


def _exp(a, terms):
    """Taylor series of exp(a) by Horner's rule."""
    one = torch.eye(3, dtype=a.dtype, device=a.device)
    e = one + a / terms
    for n in range(terms - 1, 0, -1):
        e = one + _mm(a, e) / n
    return e


def _normal(gen, *shape):
    return torch.randn(shape, dtype=torch.float64, device="cuda", generator=gen)


def _complex(gen, *shape):
    return torch.view_as_complex(_normal(gen, *shape, 2)) * math.sqrt(0.5)


def _links(case, gen):
    v = _volume(case)
    u = torch.empty((4, v, 3, 3), dtype=torch.complex128, device="cuda")
    for mu in range(4):
        g = _complex(gen, v, 3, 3)
        h = 0.5 * (g + _dag(g))
        h = h - torch.diagonal(h, dim1=-2, dim2=-1).sum(-1).real[..., None, None] / 3 * torch.eye(3, device="cuda")
        u[mu] = _exp(0.3j * h, 22)
    return u


def _poles(n):
    return [10.0 ** (-5 + 6 * i / (n - 1)) for i in range(n)]


def _inputs(case, seed):
    """The arrays a program has in hand, in double precision."""
    gen = torch.Generator(device="cuda").manual_seed(int(seed))
    v, op = _volume(case), case["op"]
    s = {"links": _links(case, gen)}
    if op in ("dslash", "normal_op"):
        s["psi"] = _complex(gen, v // 2, 3)
    elif op == "dslash_multi":
        s["psi"] = _complex(gen, case["nrhs"], v // 2, 3)
    elif op == "mscg":
        s["b"], s["poles"] = _complex(gen, v // 2, 3), _poles(case["poles"])
    elif op == "fermion_force":
        # solutions shrink with their pole as those of the solver do
        scale = torch.tensor([1.0 / (0.05 + p) for p in _poles(case["poles"])], device="cuda", dtype=torch.float64)
        s["x"] = _complex(gen, case["poles"], v // 2, 3) * scale[:, None, None]
        s["residues"] = (0.1 + 0.9 * torch.rand(case["poles"], dtype=torch.float64, device="cuda", generator=gen)).tolist()
    elif op == "stout_force":
        s["grad"] = _complex(gen, 4, v, 3, 3)
    elif op == "md_force":
        s["b"], s["xi"] = _complex(gen, v // 2, 3), _normal(gen, 4, v, 8)
    return s


def prepare(case, seed):
    s = _inputs(case, seed)
    op, lat = case["op"], stg.Lattice(_ext(case))
    s.update(case=case, lat=lat)
    if op in ("dslash", "normal_op", "dslash_multi"):
        s["gauge"] = g = stg.Gauge(lat, s["links"], case["prec"], case["recon"])
        if op == "normal_op":
            s["in"] = stg.pack(lat, s["psi"], g.vec_prec)
            s["out"], s["tmp"] = g.new_field(), g.new_field()
            s["pq"] = torch.empty(1, dtype=torch.float64, device="cuda")
        elif op == "dslash_multi":
            s["in"] = torch.stack([stg.pack(lat, p, g.vec_prec) for p in s["psi"]])
            s["out"] = torch.empty_like(s["in"])
    elif op == "mscg":
        s["gauge"] = stg.Gauge(lat, s["links"], "f64", 18)
        s["inner"] = stg.Gauge(lat, s["links"], case["inner"], 12) if case["inner"] else None
    elif op == "fermion_force":
        s["gauge"] = stg.Gauge(lat, s["links"], "f64", 18)
    elif op in ("stout_smear", "stout_force", "gauge_force"):
        dt = torch.complex128 if case["prec"] == "f64" else torch.complex64
        s["links"] = s["links"].to(dt)
        if op == "stout_force":
            s["grad"] = s["grad"].to(dt)
            s["levels"] = stg.stout_smear(lat, s["links"], RHO, STEPS)
    elif op == "md_force":
        tab = load_table()["action"]
        f32 = case["prec"] == "f32"
        pf = stg.md.Pseudofermion(s["b"], list(tab.poles), list(tab.residues), float(tab.alpha0))
        s["action"] = stg.md.Action(lat, BETA, mass=0.3, pseudofermions=[pf], stout_rho=RHO, stout_steps=STEPS, tol=1e-10,
                                    md_tol=1e-7 if f32 else None, inner="f32" if f32 else None, precision=case["prec"])
        s["mom"] = stg.md_momenta(lat, s["xi"])
    return s


def run(s):
    case, lat = s["case"], s["lat"]
    op = case["op"]
    if op == "dslash":
        return stg.dslash(s["gauge"], 0, s["psi"])
    if op == "normal_op":
        stg.normal_op_(s["gauge"], case["mass"], 0.0, s["out"], s["in"], s["tmp"], s["pq"])
        return s["out"], s["pq"]
    if op == "dslash_multi":
        return stg.dslash_multi_(s["gauge"], 0, s["out"], s["in"])
    if op == "mscg":
        x, _ = stg.mscg(s["gauge"], s["b"], s["poles"], case["mass"], tol=1e-10, g_inner=s["inner"])
        return x
    if op == "fermion_force":
        return stg.fermion_force(s["gauge"], s["residues"], s["x"], kind=case["kind"], prec=case["prec"])
    if op == "stout_smear":
        return stg.stout_smear(lat, s["links"], RHO, STEPS)
    if op == "stout_force":
        return stg.stout_force(lat, s["links"], s["levels"], RHO, s["grad"], kind=case["kind"])
    if op == "gauge_force":
        return stg.gauge_force(lat, s["links"], BETA, kind=case["kind"])
    if op == "gauge_action":
        r = stg.gauge_action(lat, s["links"], BETA)
        return r["action"], r["plaquette_sum"], r["rectangle_sum"]
    mom = s["mom"].clone()  # every pass starts from the momenta of one heatbath
    s["action"].apply_force(s["links"], mom, MD_EPS)
    return mom


# ------------------------------------------------------------------ what a pass cannot do without

_LINK = {("f64", 18): 144, ("f64", 12): 96, ("f32", 18): 72, ("f32", 12): 48, ("bf16", 12): 24, ("f16", 12): 24, ("ds", 18): 144}
_VEC = {"f64": 48, "ds": 48}


def _solve(v, mass, smallest, tol, link, vec, poles):
    """Bytes and flops of a conjugate-gradient solve at the iteration count of its condition number
    (lowest eigenvalue of -D D near 0.045 for these links): the links twice and five vectors per
    iteration, and the solutions written once."""
    its = math.log(2 / tol) / (2 * math.sqrt((mass * mass + smallest + 0.045) / 16))
    return {"bytes": its * (8 * v * link + 5 * v / 2 * vec) + poles * v / 2 * 48, "flops": its * v * (570 + 18 + 12 * poles)}


def work(case):
    v, op = _volume(case), case["op"]
    if op in ("dslash", "normal_op", "dslash_multi"):
        link, n = _LINK[(case["prec"], case["recon"])], case.get("nrhs", 1)
        vec = 48 if op == "dslash" else _VEC.get(case["prec"], 24)
        d = 2 if op == "normal_op" else 1
        # links once per application, each field read and written once; rows 1 and 2 rebuild row 3
        return {"bytes": d * 4 * v * link + n * v * vec, "flops": d * v / 2 * (n * 570 + (336 if case["recon"] == 12 else 0))}
    if op == "mscg":
        return _solve(v, case["mass"], 1e-5, 1e-10, 48 if case["inner"] else 144, 24 if case["inner"] else 48, case["poles"])
    c = 16 if case.get("prec", "f64") == "f64" else 8
    m = 4 * v * 9 * c  # bytes of one set of links
    prod = 4 * v * 216  # flops of one 3x3 complex product per link
    if op == "fermion_force":
        n = case["poles"]  # the solutions, the links, the force; D and nine complex products per pole and link
        return {"bytes": n * v / 2 * 48 + 4 * v * 144 + m, "flops": n * (v / 2 * 570 + 4 * v * 72) + prod}
    if op == "stout_smear":
        # two products a staple side and plane, the six of Q, Q^2, exp(iQ) and U'
        return {"bytes": m * (1 + STEPS), "flops": STEPS * prod * (12 + 4)}
    if op == "stout_force":
        return {"bytes": m * (STEPS + 2), "flops": STEPS * prod * (12 + 10 + 24)}
    if op == "gauge_force":
        return {"bytes": 2 * m, "flops": prod * 34}
    if op == "gauge_action":
        return {"bytes": m, "flops": v * 216 * 6 * 8}
    w = _solve(v, 0.3, 6e-3, 1e-7 if c == 8 else 1e-10, 48 if c == 8 else 144, 24 if c == 8 else 48, 10)
    link_part = m * (2 + 1 + STEPS + STEPS + 2) + 3 * 4 * v * 144
    return {"bytes": w["bytes"] + link_part, "flops": w["flops"] + prod * (34 + STEPS * 62) + 10 * 4 * v * 72}


# ------------------------------------------------------------------ the same in plain torch, 64 bits

def _at(f, dims, mu, step):
    """f(x + step mu) of an array over sites [V, ...]."""
    g = f.reshape(*dims[::-1], *f.shape[1:])
    return torch.roll(g, -step, dims=3 - mu).reshape(f.shape)


def _coords(dims):
    i = torch.arange(math.prod(dims), device="cuda")
    out = []
    for e in dims:
        out.append(i % e)
        i = i // e
    return out


class _Dirac:
    def __init__(self, dims, links):
        x = _coords(dims)
        self.dims, self.v = dims, math.prod(dims)
        par = (x[0] + x[1] + x[2] + x[3]) % 2
        self.sites = [torch.nonzero(par == p).reshape(-1) for p in (0, 1)]
        self.phase = []
        for mu in range(4):
            s = 1.0 - 2.0 * ((sum(x[:mu]) if mu else 0 * x[0]) % 2).double()
            if mu == 3:
                s = torch.where(x[3] == dims[3] - 1, -s, s)
            self.phase.append(s)
        self.fwd = [self.phase[mu][:, None, None] * links[mu] for mu in range(4)]
        self.bwd = [_dag(_at(self.fwd[mu], dims, mu, -1)).resolve_conj().contiguous() for mu in range(4)]

    def to(self, par, psi):
        """Rows of parity `par` from a field on the other parity."""
        full = torch.zeros((self.v, 3), dtype=psi.dtype, device="cuda")
        full[self.sites[1 - par]] = psi
        at, out = self.sites[par], torch.zeros_like(psi)
        for mu in range(4):
            out += (self.fwd[mu][at] * _at(full, self.dims, mu, 1)[at][:, None, :]).sum(-1)
            out -= (self.bwd[mu][at] * _at(full, self.dims, mu, -1)[at][:, None, :]).sum(-1)
        return 0.5 * out

    def normal(self, mass, psi):
        return mass * mass * psi - self.to(0, self.to(1, psi))

    def solve(self, b, mass, poles):
        """Multi-shift conjugate gradient to the end of double precision."""
        n = len(poles)
        base = min(range(n), key=lambda i: poles[i])
        extra = torch.tensor([p - poles[base] for p in poles], dtype=torch.float64, device="cuda")
        x = torch.zeros((n, *b.shape), dtype=b.dtype, device="cuda")
        p = b.repeat(n, 1, 1)
        r = b.clone()
        z0, z1 = torch.ones_like(extra), torch.ones_like(extra)
        rr = torch.vdot(r.reshape(-1), r.reshape(-1)).real
        stop, alpha0, beta0 = float(rr) * 1e-31, torch.ones_like(rr), torch.zeros_like(rr)
        for k in range(5000):
            q = self.normal(mass, p[base]) + poles[base] * p[base]
            alpha = rr / torch.vdot(p[base].reshape(-1), q.reshape(-1)).real
            # zeta_{k+1} of each shift from zeta_k, zeta_{k-1}
            z2 = z1 * z0 * alpha0 / (alpha * beta0 * (z0 - z1) + z0 * alpha0 * (1 + extra * alpha))
            x += (alpha * z2 / z1)[:, None, None] * p
            r -= alpha * q
            new = torch.vdot(r.reshape(-1), r.reshape(-1)).real
            beta = new / rr
            p *= (beta * (z2 / z1) ** 2)[:, None, None]
            p += z2[:, None, None] * r
            live = z2.abs() > 1e-30
            z0, z1 = torch.where(live, z1, z0), torch.where(live, z2, z1)
            alpha0, beta0, rr = alpha, beta, new
            if k % 8 == 7 and float(rr) < stop:
                break
        return x


def _ta(z):
    a = 0.5 * (z - _dag(z))
    return a - torch.diagonal(a, dim1=-2, dim2=-1).sum(-1)[..., None, None] / 3 * torch.eye(3, device="cuda")


def _stout_step(dims, u):
    out = []
    for mu in range(4):
        c = 0
        for nu in range(4):
            if nu == mu:
                continue
            c = c + _mm(_mm(u[nu], _at(u[mu], dims, nu, 1)), _dag(_at(u[nu], dims, mu, 1)))
            low = _mm(_mm(_dag(u[nu]), u[mu]), _at(u[nu], dims, mu, 1))
            c = c + _at(low, dims, nu, -1)
        out.append(_mm(_exp(_ta(_mm(RHO * c, _dag(u[mu]))), 24), u[mu]))
    return torch.stack(out)


def _loops(dims, u):
    """Sums of Re tr over plaquettes and over 2x1 rectangles, each once."""
    plaq = rect = 0.0
    for mu in range(4):
        for nu in range(4):
            if nu == mu:
                continue
            corner = _mm(u[mu], _at(u[nu], dims, mu, 1))      # x -> x + mu -> x + mu + nu
            other = _mm(u[nu], _at(u[mu], dims, nu, 1))       # x -> x + nu -> x + mu + nu
            if mu < nu:
                plaq = plaq + (corner * other.conj()).sum().real
            long_low = _mm(u[mu], _at(corner, dims, mu, 1))   # two steps mu, one nu
            long_up = _mm(other, _at(_at(u[mu], dims, nu, 1), dims, mu, 1))
            rect = rect + (long_low * long_up.conj()).sum().real
    return plaq, rect


def _action(dims, u):
    plaq, rect = _loops(dims, u)
    return -BETA / 3 * (2 * 5 / 6 * plaq - rect / 12), plaq, rect


def _gauge_gradient(dims, links):
    u = links.clone().requires_grad_(True)
    _action(dims, u)[0].backward()
    return u.grad


def _stout_gradient(dims, links, grad):
    u = links.clone().requires_grad_(True)
    v = u
    for _ in range(STEPS):
        v = _stout_step(dims, v)
    v.backward(gradient=grad)
    return u.grad


def _fermion_w(dims, links, x, residues):
    """W of dS = Re tr(dU W) for S = sum_i r_i Re(b^dag x_i)."""
    d = _Dirac(dims, links)
    w = torch.zeros_like(links)
    for xi, r in zip(x, residues):
        full_x = torch.zeros((d.v, 3), dtype=links.dtype, device="cuda")
        full_y = torch.zeros_like(full_x)
        full_x[d.sites[0]] = xi
        full_y[d.sites[1]] = d.to(1, xi)
        for mu in range(4):
            u = r * d.phase[mu]
            w[mu] += u[:, None, None] * (_at(full_y, dims, mu, 1)[:, :, None] * full_x.conj()[:, None, :]
                                         - _at(full_x, dims, mu, 1)[:, :, None] * full_y.conj()[:, None, :])
    return w


def _internal(case, f):
    """Canonical fields [..., Vh, 3] in the layout that the library's operators return, as doubles."""
    r = torch.view_as_real(f.resolve_conj())
    if case["prec"] == "f64":
        return r.transpose(-3, -2).flatten(-3)
    return torch.cat([r[..., :2, :].flatten(-3), r[..., 2, :].flatten(-2)], -1)


def exact(case, seed):
    s, op, dims = _inputs(case, seed), case["op"], _ext(case)
    links = s["links"]
    if op == "dslash":
        return _Dirac(dims, links).to(0, s["psi"])
    if op == "normal_op":
        q = _Dirac(dims, links).normal(case["mass"], s["psi"])
        return (None if case["prec"] == "ds" else _internal(case, q)), (s["psi"].conj() * q).sum().real.reshape(1)
    if op == "dslash_multi":
        d = _Dirac(dims, links)
        return _internal(case, torch.stack([d.to(0, p) for p in s["psi"]]))
    if op == "mscg":
        return _Dirac(dims, links).solve(s["b"], case["mass"], s["poles"])
    if op == "fermion_force":
        w = _fermion_w(dims, links, s["x"], s["residues"])
        return _ta(_mm(links, w)) if case["kind"] == 0 else _dag(w).resolve_conj()
    if op == "stout_smear":
        one = _stout_step(dims, links)
        return torch.stack([one, _stout_step(dims, one)])
    if op == "stout_force":
        g = _stout_gradient(dims, links, s["grad"])
        return _ta(_mm(links, _dag(g))) if case["kind"] == 0 else g
    if op == "gauge_force":
        g = _gauge_gradient(dims, links)
        return _ta(_mm(links, _dag(g))) if case["kind"] == 0 else g
    if op == "gauge_action":
        return tuple(float(t) for t in _action(dims, links))
    tab = load_table()["action"]
    smeared = links
    for _ in range(STEPS):
        smeared = _stout_step(dims, smeared)
    x = _Dirac(dims, smeared).solve(s["b"], 0.3, list(tab.poles))
    w = _fermion_w(dims, smeared, x, list(tab.residues))
    g = _stout_gradient(dims, links, _dag(w).resolve_conj()) + _gauge_gradient(dims, links)
    xi = s["xi"]
    h = torch.zeros((4, _volume(case), 3, 3), dtype=torch.complex128, device="cuda")
    r3 = 1 / math.sqrt(3)
    h[..., 0, 0], h[..., 1, 1], h[..., 2, 2] = xi[..., 2] + r3 * xi[..., 7], -xi[..., 2] + r3 * xi[..., 7], -2 * r3 * xi[..., 7]
    for (r, c), k in (((0, 1), 0), ((0, 2), 3), ((1, 2), 5)):
        h[..., r, c] = torch.complex(xi[..., k], -xi[..., k + 1])
        h[..., c, r] = torch.complex(xi[..., k], xi[..., k + 1])
    return math.sqrt(0.5) * h - MD_EPS * 1j * _ta(_mm(links, _dag(g)))
