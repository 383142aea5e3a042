"""The cases that the performance of this package is measured on.

A case is one call, or one short chain of calls, that an analysis makes through the package's
public functions: pair masses and boosts of large arrays of 4-vectors in both precisions and both
layouts, their gradients through autograd, jagged events with their gradients and the fused
selection, and vectors in the other coordinate systems.  Sizes and distributions are those of the
benchmark and the tests (gvx_synth describes the distributions; here the same ones are drawn on
the GPU): 65,536 pairs for a small call, 2^24 for gradients, 2^26 for whole samples, 2^20 events.
"""
import math

import torch

import paper_2312_02756_gb300 as gvx

F64, F32 = "float64", "float32"
Z_MASS = 91.1876


def listed():
    return [
        # one block of events read from a file: 65,536 pairs, where the call itself counts
        dict(name="mass_64k", op="mass", n=65536, dtype=F64, layout="soa", layout_b="soa", light=False),
        # the pair masses of a whole sample held as columns
        dict(name="mass_64m", op="mass", n=1 << 26, dtype=F64, layout="soa", layout_b="soa", light=False),
        # the same in single precision, half of the particles light and hard
        dict(name="mass_f32_64m", op="mass", n=1 << 26, dtype=F32, layout="soa", layout_b="soa", light=True),
        # every vector of a sample into its own frame
        dict(name="boost_64m", op="boost", n=1 << 26, dtype=F64, layout="soa", layout_beta="soa",
             shared=False, beta_max=0.99),
        # a differentiable fit: masses and their gradients with respect to both legs, vectors as rows
        dict(name="mass_grad_16m", op="mass_grad", n=1 << 24, dtype=F64, layout="aos", layout_b="aos",
             light=False),
        # the same for boosts: gradients with respect to vectors and velocities
        dict(name="boost_grad_16m", op="boost_grad", n=1 << 24, dtype=F64, layout="soa",
             layout_beta="soa", shared=False, beta_max=0.99),
        # all pairs and the summed vector of each of 2^20 events
        dict(name="jagged_1m", op="jagged", events=1 << 20, mean=8, layout="aos", graph=False),
        # their gradients in a fit, on a ragged number of events held as columns
        dict(name="jagged_grad_300k", op="jagged_grad", events=300007, mean=8, layout="soa"),
        # dilepton-style selection: cuts, histogram and best candidate in one pass
        dict(name="select_1m", op="select", events=1 << 20, mean=8, layout="aos", pt_min=20.0,
             eta_max=2.5, bins=200, hi=400.0),
        # pair masses of Cartesian vectors as rows, a ragged number of them
        dict(name="mass_pxpypze_10m", op="mass_cart", n=10000019, dtype=F64, layout="aos",
             coords="pxpypze"),
        # the same with the mass stored in place of the energy, as columns
        dict(name="mass_pxpypzm_10m", op="mass_cart", n=10000019, dtype=F64, layout="soa",
             coords="pxpypzm"),
        # detector coordinates to Cartesian, then one Lorentz transformation for all vectors
        dict(name="transform_10m", op="transform", n=10000019, dtype=F64, layout="soa",
             coords="ptetaphim", per_vector=False),
    ]


def _log_int(rng, lo, hi):
    """A whole number, log-uniform in [lo, hi]."""
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    op = rng.choice(["mass", "mass", "mass_grad", "boost", "boost_grad", "jagged", "jagged_grad",
                     "select", "mass_cart", "transform"])
    layout, other = rng.choice(["soa", "aos"]), rng.choice(["soa", "aos"])
    dtype = rng.choice([F64, F64, F32])
    if op in ("jagged", "jagged_grad", "select"):
        mean = rng.randint(4, 12)  # the pairs grow with its square: fewer events of larger ones
        most = int((1 << 20) * min(1.0, (8.0 / mean) ** 2))
        case = dict(op=op, mean=mean, layout=layout,
                    events=_log_int(rng, 200, most // 3 if op == "jagged_grad" else most))
        if op == "jagged":
            case["graph"] = rng.random() < 0.5
        if op == "select":
            case.update(pt_min=rng.choice([0.0, 10.0, 20.0, 30.0]), eta_max=rng.choice([2.1, 2.5, 5.0]),
                        bins=rng.randint(20, 400), hi=rng.choice([200.0, 400.0, 1000.0]))
        return case
    grad = op.endswith("_grad")
    if op == "mass_cart":
        return dict(op=op, n=_log_int(rng, 1000, 10000019), dtype=dtype, layout=layout,
                    coords=rng.choice(["pxpypze", "pxpypzm", "ptetaphie"]))
    if op == "transform":
        return dict(op=op, n=_log_int(rng, 1000, 10000019), dtype=dtype, layout=layout,
                    coords=rng.choice(["ptetaphim", "ptetaphie", "pxpypzm"]),
                    per_vector=rng.random() < 0.25)
    n = _log_int(rng, 1000, 1 << 24 if grad else 1 << 26)
    if op.startswith("mass"):
        return dict(op=op, n=n, dtype=dtype, layout=layout, layout_b=other, light=rng.random() < 0.3)
    return dict(op=op, n=n, dtype=dtype, layout=layout, layout_beta=other,
                shared=rng.random() < 0.25, beta_max=0.999999 if dtype == F32 else 0.99)


# ------------------------------------------------------------------------------------- inputs

class _Draws:
    """Seeded draws on the GPU, in FP64."""

    def __init__(self, seed):
        self.g = torch.Generator(device="cuda")
        self.g.manual_seed(int(seed))

    def uniform(self, lo, hi, *shape):
        return torch.rand(*shape, dtype=torch.float64, device="cuda", generator=self.g) * (hi - lo) + lo

    def log_uniform(self, lo, hi, *shape):
        return self.uniform(math.log(lo), math.log(hi), *shape).exp_()

    def directions(self, n):
        d = torch.randn(3, n, dtype=torch.float64, device="cuda", generator=self.g)
        return d / d.square().sum(0).sqrt_().clamp_(min=1e-30)

    def ptetaphim(self, n, light=False):
        """(4, n): pt log-uniform in [1, 1000], eta in [-4, 4], phi in [-pi, pi), m in [0, 10];
        light: half of them with pt log-uniform in [100, 5000] and m in [0, 1e-3]."""
        v = torch.stack([self.log_uniform(1.0, 1000.0, n), self.uniform(-4.0, 4.0, n),
                         self.uniform(-math.pi, math.pi, n), self.uniform(0.0, 10.0, n)])
        if light:
            hard = self.uniform(0.0, 1.0, n) < 0.5
            v[0] = torch.where(hard, self.log_uniform(100.0, 5000.0, n), v[0])
            v[3] = torch.where(hard, self.uniform(0.0, 1e-3, n), v[3])
        return v

    def pxpypze(self, n):
        """(4, n): isotropic, |p| log-uniform in [1, 3e4], on shell with m in [0, 10]."""
        p, m = self.log_uniform(1.0, 3.0e4, n), self.uniform(0.0, 10.0, n)
        return torch.cat([self.directions(n) * p, (p * p + m * m).sqrt_()[None]])

    def velocities(self, n, beta_max):
        return self.directions(n) * self.uniform(0.0, beta_max, n)

    def in_coords(self, n, coords):
        v = self.ptetaphim(n)
        pt, eta, phi, m = v
        if coords == "ptetaphim":
            return v
        energy = ((pt * eta.cosh()).square() + m * m).sqrt()
        if coords == "ptetaphie":
            return torch.stack([pt, eta, phi, energy])
        return torch.stack([pt * phi.cos(), pt * phi.sin(), pt * eta.sinh(),
                            energy if coords == "pxpypze" else m])


def _laid_out(v, layout, dtype=F64):
    """Components by rows (k, n) as the given layout and type."""
    v = v.to(getattr(torch, dtype))
    return (v.t() if layout == "aos" else v).contiguous()


def _inputs(case, seed):
    """The tensors of a case by name."""
    d, op = _Draws(seed), case["op"]
    if op in ("jagged", "jagged_grad", "select"):
        # Poisson multiplicities up to 64, the same ones in another order for each seed, so that the
        # number of particles and pairs belongs to the case
        counts = torch.poisson(torch.full((case["events"],), float(case["mean"]), device="cuda"),
                               generator=_Draws(1).g).clamp_(max=64).long()
        counts = counts[torch.randperm(case["events"], device="cuda", generator=d.g)]
        off = torch.zeros(case["events"] + 1, dtype=torch.int64, device="cuda")
        torch.cumsum(counts, 0, out=off[1:])
        s = {"offsets": off, "particles": _laid_out(d.ptetaphim(int(off[-1])), case["layout"])}
        s["n_pairs"] = int((counts * (counts - 1) // 2).sum())
        if op == "jagged_grad":
            s["gm"] = d.uniform(-1.0, 1.0, s["n_pairs"])
            s["gs"] = d.uniform(-1.0, 1.0, case["events"], 4)
        return s
    n, dtype, layout = case["n"], case["dtype"], case["layout"]
    if op in ("mass", "mass_grad"):
        s = {"a": _laid_out(d.ptetaphim(n, case["light"]), layout, dtype),
             "b": _laid_out(d.ptetaphim(n, case["light"]), case["layout_b"], dtype)}
        if op == "mass_grad":
            s["g"] = d.uniform(-1.0, 1.0, n).to(getattr(torch, dtype))
    elif op in ("boost", "boost_grad"):
        beta = d.velocities(1 if case["shared"] else n, case["beta_max"])
        s = {"v": _laid_out(d.pxpypze(n), layout, dtype),
             "beta": _laid_out(beta, case["layout_beta"], dtype)}
        if case["shared"]:
            s["beta"] = s["beta"].reshape(3)
        if op == "boost_grad":
            s["g"] = _laid_out(d.uniform(-1.0, 1.0, 4, n), layout, dtype)
    elif op == "mass_cart":
        s = {"a": _laid_out(d.in_coords(n, case["coords"]), layout, dtype),
             "b": _laid_out(d.in_coords(n, case["coords"]), layout, dtype)}
    else:
        matrix = _boost_matrix(d.velocities(n if case["per_vector"] else 1, 0.9))
        s = {"v": _laid_out(d.in_coords(n, case["coords"]), layout, dtype),
             "L": (matrix if case["per_vector"] else matrix[0]).to(getattr(torch, dtype)).contiguous()}
    return s


def _boost_matrix(beta):
    """(n, 4, 4) boosts of (px, py, pz, E) by the columns of beta."""
    n = beta.shape[1]
    gamma = (1.0 - beta.square().sum(0)).rsqrt()
    m = torch.zeros(n, 4, 4, dtype=torch.float64, device="cuda")
    m[:, :3, :3] = (torch.eye(3, dtype=torch.float64, device="cuda")
                    + (gamma * gamma / (1.0 + gamma))[:, None, None] * (beta.t()[:, :, None] * beta.t()[:, None, :]))
    m[:, :3, 3] = m[:, 3, :3] = (gamma * beta).t()
    m[:, 3, 3] = gamma
    return m


def prepare(case, seed):
    s = _inputs(case, seed)
    s["case"] = case
    for name in {"mass_grad": ("a", "b"), "boost_grad": ("v", "beta"),
                 "jagged_grad": ("particles",)}.get(case["op"], ()):
        s[name].requires_grad_(True)
    if case.get("graph"):
        s["replay"] = gvx.EventPairMassesGraph(s["particles"], s["offsets"], s["n_pairs"],
                                               layout=case["layout"])
    return s


def run(s):
    case = s["case"]
    op = case["op"]
    if op in ("mass", "mass_grad"):
        m = gvx.invariant_mass(s["a"], s["b"], case["layout"], case["layout_b"])
        return m if op == "mass" else (m, *torch.autograd.grad(m, (s["a"], s["b"]), s["g"]))
    if op in ("boost", "boost_grad"):
        out = gvx.boost(s["v"], s["beta"], case["layout"], None if case["shared"] else case["layout_beta"])
        return out if op == "boost" else (out, *torch.autograd.grad(out, (s["v"], s["beta"]), s["g"]))
    if op == "mass_cart":
        return gvx.invariant_mass_cart(s["a"], s["b"], case["coords"], case["layout"], case["layout"])
    if op == "transform":
        cart = gvx.to_pxpypze(s["v"], case["coords"], case["layout"])
        return cart, gvx.lorentz_apply(s["L"], cart, case["layout"])
    if op == "select":
        return gvx.event_pair_select(s["particles"], s["offsets"], case["pt_min"], case["eta_max"], 0.0,
                                     case["hi"], case["bins"], Z_MASS, layout=case["layout"])
    if case.get("graph"):
        s["replay"].launch()
        return s["replay"].pair_offsets, s["replay"].pair_m, s["replay"].sums
    off, m, sums = gvx.event_pair_masses(s["particles"], s["offsets"], s["n_pairs"], case["layout"])
    if op == "jagged":
        return off, m, sums
    return off, m, sums, *torch.autograd.grad((m, sums), s["particles"], (s["gm"], s["gs"]))


# --------------------------------------------------------------------------------------- work

def work(case):
    """Bytes: each input read once, each output written once.  Operations: those of the plain
    formulas, an elementary function counted as one."""
    op = case["op"]
    if op in ("jagged", "jagged_grad", "select"):
        e, p = case["events"], case["events"] * case["mean"]
        q = case["events"] * case["mean"] ** 2 / 2
        if op == "select":
            return {"bytes": 32 * p + 24 * e, "flops": 2 * p}
        out = {"bytes": 32 * p + 8 * q + 48 * e, "flops": 12 * p + 16 * q}
        if op == "jagged_grad":
            out = {"bytes": out["bytes"] + 32 * p + 8 * q + 32 * e, "flops": out["flops"] + 30 * p + 40 * q}
        return out
    n, w = case["n"], 8 if case["dtype"] == F64 else 4
    beta = 0 if case.get("shared") else 3
    values, flops = {
        "mass": (9, 28), "mass_grad": (9 + 9, 80), "mass_cart": (9, 28),
        "boost": (8 + beta, 24), "boost_grad": (16 + 2 * beta, 70),
        "transform": (4 + 4 + 4 + (16 if case.get("per_vector") else 0), 40),
    }[op]
    return {"bytes": values * n * w, "flops": flops * n}


# -------------------------------------------------------------------------------------- exact

def _rows(v, layout):
    v = v.detach().double()
    return v.t().contiguous() if layout == "aos" else v


def _like(v, layout):
    return v.t().contiguous() if layout == "aos" else v


def _half_dphi(p1, p2):
    d = p1 - p2
    wrapped = (math.pi - p1.abs()) + (math.pi - p2.abs()) + 2.4492935982947064e-16
    far = (d.abs() > math.pi) & (p1.abs() <= math.pi) & (p2.abs() <= math.pi)
    return 0.5 * torch.where(far, -wrapped * d.sign(), d)


def _mass(a, b):
    """Pair masses of (pt, eta, phi, m) rows, as a sum of non-negative terms."""
    q1, q2 = a[3].square(), b[3].square()
    p1, p2 = a[0] * a[1].cosh(), b[0] * b[1].cosh()
    e1, e2 = (p1.square() + q1).sqrt(), (p2.square() + q2).sqrt()
    t = 2.0 * (q1 * p2.square() + q2 * p1.square() + q1 * q2) / (e1 * e2 + p1 * p2)
    s = (0.5 * (a[1] - b[1])).sinh().square() + _half_dphi(a[2], b[2]).sin().square()
    return (q1 + q2 + t + 4.0 * a[0] * b[0] * s).sqrt()


def _mass_cart(a, b, coords):
    if coords == "ptetaphie":
        p1, p2 = a[0] * a[1].cosh(), b[0] * b[1].cosh()
        s = (0.5 * (a[1] - b[1])).sinh().square() + _half_dphi(a[2], b[2]).sin().square()
        m2 = (a[3] - p1 + b[3] - p2) * (a[3] + p1 + b[3] + p2) + 4.0 * a[0] * b[0] * s
    else:
        if coords == "pxpypzm":
            q1, q2 = a[3].square(), b[3].square()
            e1, e2 = (a[:3].square().sum(0) + q1).sqrt(), (b[:3].square().sum(0) + q2).sqrt()
        else:
            e1, e2 = a[3], b[3]
            p1, p2 = a[:3].square().sum(0).sqrt(), b[:3].square().sum(0).sqrt()
            q1, q2 = (e1 - p1) * (e1 + p1), (e2 - p2) * (e2 + p2)
        m2 = q1 + q2 + 2.0 * (e1 * e2 - (a[:3] * b[:3]).sum(0))
    return m2.abs().sqrt() * m2.sign()


def _boost(v, beta):
    beta = beta.reshape(3, -1)
    gamma = (1.0 - beta.square().sum(0)).rsqrt()
    bp = (beta * v[:3]).sum(0)
    energy = gamma * (v[3] + bp)
    f = gamma * gamma / (1.0 + gamma) * bp + gamma * v[3]
    return torch.cat([v[:3] + f * beta, energy[None]])


def _pairs(off):
    """Indices (i, j), i < j, of every in-event pair in row-major order, and each particle's event."""
    counts = off[1:] - off[:-1]
    event = torch.repeat_interleave(torch.arange(len(counts), device=off.device), counts)
    k = torch.arange(int(off[-1]), device=off.device)
    after = off[1:][event] - 1 - k  # partners that follow a particle in its event
    i = torch.repeat_interleave(k, after)
    first = torch.cumsum(after, 0) - after
    return i, i + 1 + torch.arange(len(i), device=off.device) - first[i], event


def _sums(p, event, n_events):
    pt, eta, phi, m = p
    cart = torch.stack([pt * phi.cos(), pt * phi.sin(), pt * eta.sinh(),
                        ((pt * eta.cosh()).square() + m * m).sqrt()], 1)
    return torch.zeros(n_events, 4, dtype=torch.float64, device=p.device).index_add(0, event, cart)


def exact(case, seed):
    s, op = _inputs(case, seed), case["op"]
    if op in ("mass", "mass_grad"):
        a, b = _rows(s["a"], case["layout"]), _rows(s["b"], case["layout_b"])
        if op == "mass":
            return _mass(a, b)
        a, b = a.clone().requires_grad_(True), b.clone().requires_grad_(True)
        m = _mass(a, b)
        ga, gb = torch.autograd.grad(m, (a, b), s["g"].double())
        return m.detach(), _like(ga, case["layout"]), _like(gb, case["layout_b"])
    if op in ("boost", "boost_grad"):
        v = _rows(s["v"], case["layout"])
        beta = s["beta"].double() if case["shared"] else _rows(s["beta"], case["layout_beta"])
        if op == "boost":
            return _like(_boost(v, beta), case["layout"])
        v, beta = v.clone().requires_grad_(True), beta.clone().requires_grad_(True)
        out = _boost(v, beta)
        gv, gbeta = torch.autograd.grad(out, (v, beta), _rows(s["g"], case["layout"]))
        return (_like(out.detach(), case["layout"]), _like(gv, case["layout"]),
                gbeta if case["shared"] else _like(gbeta, case["layout_beta"]))
    if op == "mass_cart":
        return _mass_cart(_rows(s["a"], case["layout"]), _rows(s["b"], case["layout"]), case["coords"])
    if op == "transform":
        x, w = _rows(s["v"], case["layout"]), case["coords"]
        if w == "pxpypzm":
            cart = torch.cat([x[:3], x.square().sum(0).sqrt()[None]])
        else:
            energy = x[3] if w == "ptetaphie" else ((x[0] * x[1].cosh()).square() + x[3].square()).sqrt()
            cart = torch.stack([x[0] * x[2].cos(), x[0] * x[2].sin(), x[0] * x[1].sinh(), energy])
        moved = torch.einsum("nij,jn->in" if case["per_vector"] else "ij,jn->in", s["L"].double(), cart)
        return _like(cart, case["layout"]), _like(moved, case["layout"])
    off, p = s["offsets"], _rows(s["particles"], case["layout"])
    if op == "select":
        i, j, event = _pairs(off)
        ok = (p[0] >= case["pt_min"]) & (p[1].abs() <= case["eta_max"])
        both = ok[i] & ok[j]
        i, j = i[both], j[both]
        m = _mass(p[:, i], p[:, j])
        d, e = (m - Z_MASS).abs(), event[i]
        nearest = torch.full((case["events"],), math.inf, dtype=torch.float64, device="cuda")
        nearest.scatter_reduce_(0, e, d, "amin")
        best = torch.full((case["events"],), math.nan, dtype=torch.float64, device="cuda")
        chosen = d == nearest[e]
        best[e[chosen]] = m[chosen]
        return None, None, best
    i, j, event = _pairs(off)
    if op == "jagged":
        return None, _mass(p[:, i], p[:, j]), _sums(p, event, case["events"])
    p = p.clone().requires_grad_(True)
    m, sums = _mass(p[:, i], p[:, j]), _sums(p, event, case["events"])
    gp, = torch.autograd.grad((m, sums), p, (s["gm"], s["gs"]))
    return None, m.detach(), sums.detach(), _like(gp, case["layout"])
