"""The calls whose speed is measured, with their inputs and their values in 64 bits.

A case is one pass through the package's public entry points (paper_2210_00947_gb300.mgar, .batch, .autograd) as a
topology-optimisation program makes it: a design cycle, a whole run from host memory, an MGCG or MGAR solve, the
design update around a solver of the user's own, the differentiable compliance, the batched design cycle, the boundary
post-processing.  Grids and settings are those of the package's workloads (paper_2210_00947_gb300.workloads).

The mixed-precision cases solve to 1e-10 (the compliance checks' tolerance; the gradient case to 1e-11, as the
differentiation workload), the FP64 ones to the default 1e-8.  Temperatures start from zero in every pass, so that each
pass does the same work.
"""
import itertools
import math

import numpy as np
import torch
import torch.nn.functional as F

from paper_2210_00947_gb300 import autograd, batch, mgar, workloads

LOAD = 0.01          # uniform nodal load of the heat-sink workloads
ALPHA, LP = 1.4 / 50, 250  # continuous filter (the paper's defaults for 300 cycles)


def _case(kind, nx, ny, nz=0, precision="mixed", **more):
    c = dict(kind=kind, nx=nx, ny=ny, nz=nz, precision=precision, volfrac=0.3 if nz else 0.4, rmin=1.5,
             eps2=1e-10 if precision == "mixed" else 1e-8)
    c.update(more)
    return c


def listed():
    return [
        # the smallest whole problem: a design cycle on the 100 x 100 plate with the default (FP64) precision,
        # latency and launches
        dict(_case("step", 100, 100, precision="fp64"), name="step_2d_100_fp64"),
        # one analysis of the paper's Model 1 (361^2 nodes) in FP64
        dict(_case("solve", 360, 360, precision="fp64", volfrac=0.5, rmin=3.0), name="solve_2d_360_fp64"),
        # a design cycle of the large 2D workload
        dict(_case("step", 1024, 1024), name="step_2d_1024"),
        # a design cycle of the headline workload
        dict(_case("step", 128, 128, 128), name="step_3d_128"),
        # an analysis on a small ragged block
        dict(_case("solve", 75, 53, 41), name="solve_3d_ragged"),
        # the FP64 analysis of the headline workload (what the mixed path is measured against)
        dict(_case("solve", 128, 128, 128, precision="fp64"), name="solve_3d_128_fp64"),
        # one reanalysis (two basis vectors) of the paper's Model 2 on the last factorised matrix
        dict(_case("mgar", 720, 720, precision="fp64", volfrac=0.5, rmin=3.0), name="mgar_2d_720_fp64"),
        # the first design cycles of the paper's 3D model with the continuous filter, from host memory
        dict(_case("run", 224, 112, 112, rmin=3.0, cycles=2), name="run_3d_quarter"),
        # the design half of a cycle around a solver of the user's own: the paper's Model 4 (2041^2 nodes)
        dict(_case("update", 2040, 2040, volfrac=0.5, rmin=3.0), name="update_2d_2040"),
        # 64 uneven designs, one cycle of all
        dict(kind="batch", count=64, design_seed=2210, eps2=1e-10, name="batch_64"),
        # forward and backward of the differentiable compliance on 256^3 independent random densities
        dict(_case("grad", 256, 256, 256, eps2=1e-11), name="grad_3d_256"),
        # post-processing of a finished headline design
        dict(_case("post", 128, 128, 128), name="post_3d_128"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("step", "step", "solve", "solve", "mgar", "run", "update", "batch", "grad", "post"))
    if kind == "batch":
        return dict(kind="batch", count=_log(rng, 4, 64), design_seed=rng.randrange(1 << 20), eps2=1e-10)
    three = kind != "update" and rng.random() < 0.5
    precision = "fp64" if kind == "mgar" or (kind in ("step", "solve") and rng.random() < 0.4) else "mixed"
    top = 128 if three else {"step": 1024, "solve": 1024, "mgar": 1024, "run": 720, "grad": 1024}.get(kind, 2040)
    if precision == "fp64":
        top = min(top, 96 if three else 720)
    low = 24 if three else 64
    a = _log(rng, low, top)
    b = min(top, max(low, _log(rng, a / 2, a * 2)))
    c = min(top, max(low, _log(rng, a / 2, a * 2))) if three else 0
    rmin = rng.choice((1.5, 1.5, 2.0, 3.0)) if not three else rng.choice((1.5, 1.5, 2.0))
    case = _case(kind, a, b, c, precision, rmin=rmin, volfrac=round(rng.uniform(0.2, 0.5), 2))
    if kind == "run":
        case.update(rmin=3.0, cycles=rng.choice((1, 2, 3)))
    return case


# ---------------------------------------------------------------- inputs
def _dev():
    return torch.device("cuda", torch.cuda.current_device())


def _gen(seed, salt=0):
    g = torch.Generator(device=_dev())
    g.manual_seed(1000003 * int(seed) + salt)
    return g


def _smooth(shape, cell, g):
    """Uniform random values on a grid of `cell` spacing, interpolated to `shape`."""
    coarse = [n // cell + 2 for n in shape]
    v = torch.rand([1, 1] + coarse, generator=g, device=_dev(), dtype=torch.float64)
    return F.interpolate(v, size=shape, mode="bilinear" if len(shape) == 2 else "trilinear", align_corners=True)[0, 0]


def _eshape(c):
    return (c["ny"], c["nx"]) if not c["nz"] else (c["nz"], c["ny"], c["nx"])


def _density(c, seed, salt=0):
    """A design in mid-optimisation, mean about volfrac: a stem from the sink (the middle of x = 0) and grey regions
    of some elements' width; independent uniform values for the gradient case."""
    g = _gen(seed, 1)
    shape = _eshape(c)
    if c["kind"] == "grad":
        return 0.05 + 0.95 * torch.rand(shape, generator=g, device=_dev(), dtype=torch.float64).reshape(-1)
    v = 0.9 * (_smooth(shape, 10, g) - 0.5) + 0.1 * torch.rand(shape, generator=g, device=_dev(), dtype=torch.float64)
    if salt:  # the same design some cycles later
        v = v + 0.1 * (_smooth(shape, 12, _gen(seed, 1 + salt)) - 0.5)
    off = [((torch.arange(n, device=_dev(), dtype=torch.float64) + 0.5) / n - 0.5) / 0.06 for n in shape[:-1]]
    off = off[0][:, None] if len(off) == 1 else torch.sqrt(off[0][:, None] ** 2 + off[1][None, :] ** 2)[..., None]
    v = (v + 0.6 * torch.exp(-off * off)).reshape(-1)
    return (v - v[:: max(1, v.numel() // 1000000)].mean() + c["volfrac"]).clamp(0.02, 1.0)


def _temperature(c, seed):
    """Temperatures rising away from the sink, with the design's unevenness; zero on the sink."""
    g = _gen(seed, 7)
    shape = tuple(n + 1 for n in _eshape(c))
    x = torch.linspace(0.0, 1.0, shape[-1], device=_dev(), dtype=torch.float64)
    t = 20.0 * (1.0 - torch.exp(-3.0 * x)).expand(shape) + 3.0 * _smooth(shape, 24, g) + 0.3 * _smooth(shape, 6, g)
    return t.reshape(-1) * (1 - torch.as_tensor(_fixed(c), device=_dev()).double())


def _fixed(c):
    if c["kind"] == "run" and c["nz"]:  # the quarter model's corner sink, an eighth of the face's side
        return workloads.quarter_sink_mask(c["nx"], c["ny"], c["nz"], max(2, c["ny"] // 8))
    return workloads.heat_sink_mask(c["nx"], c["ny"], c["nz"])


def _levels(c):
    return workloads.levels_for_direct_coarsest(c["nx"], c["ny"], c["nz"], max_nodes=300)


def _solver(c):
    fixed = _fixed(c)
    more = {}
    if c["kind"] == "run":
        more = dict(filter_alpha=ALPHA, filter_lp=LP)
    if c["kind"] == "mgar":
        more = dict(m=2, basis_guess=mgar.MGAR_GUESS_ZERO)
    p = mgar.default_params(nx=c["nx"], ny=c["ny"], nz=c["nz"], nl=_levels(c), rmin=c["rmin"], eps2=c["eps2"],
                            volfrac=c["volfrac"], n_on=1000,
                            precision=mgar.MGAR_MIXED if c["precision"] == "mixed" else mgar.MGAR_FP64, **more)
    return mgar.Solver(p, fixed, workloads.nodal_load(fixed, LOAD))


def _flat_views(sizes):
    """One buffer holding every design's vector (each on a 256-byte boundary) and the views of it."""
    at = [0]
    for n in sizes:
        at.append(at[-1] + (n + 31) // 32 * 32)
    flat = torch.zeros(at[-1], dtype=torch.float64, device=_dev())
    return flat, [flat[a: a + n] for a, n in zip(at, sizes)]


def prepare(case, seed):
    c, s = case, {"case": case}
    if c["kind"] == "batch":
        designs = [batch.Design(**d) for d in workloads.batched_designs(c["count"], c["design_seed"])]
        s["solvers"] = [mgar.Solver(d.params(30, mgar.MGAR_MIXED, n_on=1000, eps2=c["eps2"]), d.fixed(), d.q())
                        for d in designs]
        s["volfracs"] = [d.volfrac for d in designs]
        s["rho"], s["rhos"] = _flat_views([d.nx * d.ny for d in designs])
        s["T"], s["Ts"] = _flat_views([(d.nx + 1) * (d.ny + 1) for d in designs])
        for k, (d, r) in enumerate(zip(designs, s["rhos"])):
            r.copy_(_density(dict(kind="batch", nx=d.nx, ny=d.ny, nz=0, volfrac=d.volfrac), seed * 64 + k))
        s["rho0"] = s["rho"].clone()
        s["batch"] = mgar.BatchSolver(s["solvers"])
        return s
    s["solver"] = sv = _solver(c)
    s["rho0"] = _density(c, seed)
    if c["kind"] in ("step", "solve", "mgar", "grad"):
        s["T"] = torch.zeros(sv.n_nodes, dtype=torch.float64, device=_dev())
    if c["kind"] in ("step", "update"):
        s["rho"] = s["rho0"].clone()
    if c["kind"] == "mgar":
        sv.set_density(s["rho0"])
        sv.build_hierarchy()  # the reference matrix K0
        s["rho"] = _density(c, seed, salt=2)
        s["T_prev"] = _temperature(c, seed)
    if c["kind"] == "run":
        s["rho_host"] = s["rho0"].cpu().pin_memory()
        s["rho_out"] = torch.empty_like(s["rho_host"]).pin_memory()
    if c["kind"] in ("update", "post"):
        s["T"] = _temperature(c, seed)
    if c["kind"] == "update":
        s["dc"], s["dv"] = torch.empty_like(s["rho0"]), torch.empty_like(s["rho0"])
    if c["kind"] == "post":
        s["out"] = torch.empty_like(s["rho0"])
    if c["kind"] == "grad":
        s["rho"] = s["rho0"].clone().requires_grad_(True)
    return s


def run(state):
    s, c = state, state["case"]
    kind = c["kind"]
    if kind == "batch":
        s["rho"].copy_(s["rho0"])
        s["T"].zero_()
        info = s["batch"].cycle(s["rhos"], s["Ts"], s["volfracs"], 0.2)
        return {"rho": s["rho"], "T": s["T"], "compliance": np.array([i["compliance"] for i in info]),
                "lam": np.array([i["lam"] for i in info])}
    sv = s["solver"]
    if kind == "step":
        s["rho"].copy_(s["rho0"])
        s["T"].zero_()
        info = sv.step(s["rho"], s["T"], 1)
        return {"rho": s["rho"], "T": s["T"], "scalars": np.array([info["compliance"], info["lam"]])}
    if kind == "solve":
        sv.set_density(s["rho0"])
        s["T"].zero_()
        _, _, ok = sv.solve_mgcg(s["T"])
        return {"T": s["T"], "converged": ok}
    if kind == "mgar":
        sv.set_density(s["rho"])
        res, accepted = sv.solve_mgar(s["T_prev"], s["T"])
        return {"T": s["T"], "scalars": np.array([res]), "accepted": accepted}
    if kind == "run":
        info = sv.run(s["rho_host"], c["cycles"], s["rho_out"])
        return {"rho": s["rho_out"], "compliance": np.array([i["compliance"] for i in info]),
                "lam": np.array([i["lam"] for i in info])}
    if kind == "update":
        s["rho"].copy_(s["rho0"])
        sv.set_density(s["rho"])
        comp = sv.sensitivity(s["T"], s["dc"], s["dv"])
        lam, change = sv.oc_update(s["rho"], s["dc"], c["volfrac"], 0.2)
        return {"dc": s["dc"], "dv": s["dv"], "rho": s["rho"], "scalars": np.array([comp, lam, change])}
    if kind == "grad":
        s["T"].zero_()
        s["rho"].grad = None
        comp = autograd.ComplianceFunction.apply(s["rho"], sv, s["T"])
        comp.backward()
        return {"compliance": comp.detach(), "grad": s["rho"].grad}
    level, volume = sv.postprocess(s["rho0"], s["T"], c["volfrac"], s["out"])
    return {"rho": s["out"], "scalars": np.array([level, volume])}


def work(case):
    """Inputs once, outputs once; operations of the solve from a nominal count of iterations (15, or 20 to 1e-10),
    each one V-cycle (three finest-level stencil passes, the coarse levels a sixth more) and one product."""
    c = case
    if c["kind"] == "batch":
        nodes = elems = 0
        for d in workloads.batched_designs(c["count"], c["design_seed"]):
            nodes += (d["nx"] + 1) * (d["ny"] + 1)
            elems += d["nx"] * d["ny"]
        return {"bytes": 17.0 * nodes + 16.0 * elems, "flops": 20 * 4.5 * 18.0 * nodes + 200.0 * elems}
    n, e = workloads.num_nodes(c["nx"], c["ny"], c["nz"]), workloads.num_elements(c["nx"], c["ny"], c["nz"])
    row = 64.0 if c["nz"] else 18.0
    its = 15 if c["precision"] == "fp64" else 20
    r = ALPHA * max(c["nx"], c["ny"], c["nz"]) if c["kind"] == "run" else c["rmin"]
    r = max(r, c["rmin"])
    taps = 4.19 * r ** 3 if c["nz"] else 3.14 * r * r
    filt, oc, solve = 2.0 * taps * e, 40.0 * e, its * (4.5 * row + 10.0) * n
    kind = c["kind"]
    if kind == "step":
        return {"bytes": 17.0 * n + 16.0 * e, "flops": solve + 2 * filt + oc}
    if kind == "solve":
        return {"bytes": 17.0 * n + 8.0 * e, "flops": solve + filt}
    if kind == "mgar":
        return {"bytes": 25.0 * n + 16.0 * e, "flops": (7.5 * row + 20.0) * n + filt}
    if kind == "run":
        return {"bytes": 9.0 * n + 16.0 * e, "flops": c["cycles"] * (solve + 2 * filt + oc)}
    if kind == "update":
        return {"bytes": 16.0 * n + 32.0 * e, "flops": 2 * filt + oc}
    if kind == "grad":
        return {"bytes": 9.0 * n + 24.0 * e, "flops": 26 * (4.5 * row + 10.0) * n + 2 * filt}
    points = 125 if c["nz"] else 25
    return {"bytes": 8.0 * n + 16.0 * e, "flops": filt * 2 + 2.0 * points * e}


# ------------------------------------------------- the same in 64 bits, plain torch
class _Ref:
    """The discrete problem in torch, FP64: arrays shaped (nz,) ny, nx, x fastest."""

    def __init__(self, c):
        self.c, self.eshape, self.d = c, _eshape(c), 3 if c["nz"] else 2
        self.nshape = tuple(n + 1 for n in self.eshape)
        self.free = 1.0 - torch.as_tensor(_fixed(c), device=_dev()).double().reshape(self.nshape)
        self.q = LOAD * self.free
        self.corners = list(itertools.product((0, 1), repeat=self.d))
        if self.d == 2:  # weights -k0_ab of the pairs
            w = {1: 1 / 6, 2: 2 / 6}
        else:
            w = {2: 1 / 12, 3: 1 / 12}
        self.pairs = [(a, b, w[h]) for a, b in itertools.combinations(range(len(self.corners)), 2)
                      if (h := sum(x != y for x, y in zip(self.corners[a], self.corners[b]))) in w]
        self.diag = 4 / 6 if self.d == 2 else 4 / 12

    def at(self, x, a):
        return x[tuple(slice(o, o + n) for o, n in zip(self.corners[a], self.eshape))]

    def k_apply(self, k, x):
        y = torch.zeros_like(x)
        for a, b, w in self.pairs:
            t = (self.at(x, a) - self.at(x, b)) * k * w
            self.at(y, a).add_(t)
            self.at(y, b).sub_(t)
        return y

    def a_apply(self, k, x):  # Z K Z + (I - Z)
        return self.free * self.k_apply(k, self.free * x) + (1 - self.free) * x

    def a_diag(self, k):
        dg = torch.zeros(self.nshape, dtype=torch.float64, device=_dev())
        for a in range(len(self.corners)):
            self.at(dg, a).add_(k * self.diag)
        return dg * self.free + (1 - self.free)

    def filter(self, x, r, transpose=False):
        reach = int(math.ceil(r))
        offs = [(o, r - math.sqrt(sum(v * v for v in o)))
                for o in itertools.product(range(-reach, reach + 1), repeat=self.d)]
        offs = [(o, w) for o, w in offs if w > 0]
        pad = [reach] * (2 * self.d)

        def acc(v):
            v, out = F.pad(v, pad), torch.zeros(self.eshape, dtype=torch.float64, device=_dev())
            for o, w in offs:
                out.add_(v[tuple(slice(reach + i, reach + i + n) for i, n in zip(o, self.eshape))], alpha=w)
            return out

        hs = acc(torch.ones(self.eshape, dtype=torch.float64, device=_dev()))
        return acc(x / hs) if transpose else acc(x) / hs

    def simp(self, rho_t):
        return 1e-3 + (1.0 - 1e-3) * rho_t ** 3

    def solve(self, k):
        dinv = self.free / self.a_diag(k)
        x = torch.zeros_like(self.q)
        r = self.q.clone()
        z = dinv * r
        p, rz, q2 = z.clone(), (r * z).sum(), (r * r).sum()
        for it in range(20000):
            ap = self.free * self.k_apply(k, p)
            alpha = rz / (p * ap).sum()
            x += alpha * p
            r -= alpha * ap
            z = dinv * r
            new = (r * z).sum()
            p = z + (new / rz) * p
            rz = new
            if it % 100 == 99 and float((r * r).sum() / q2) < 1e-27:
                break
        return x

    def sens(self, rho_t, t):
        e = torch.zeros(self.eshape, dtype=torch.float64, device=_dev())
        for a, b, w in self.pairs:
            e += w * (self.at(t, a) - self.at(t, b)) ** 2
        return -3.0 * (1.0 - 1e-3) * rho_t ** 2 * e

    def oc(self, rho, dc, dv, volfrac, move=0.2):
        s = rho * torch.sqrt(torch.clamp(-dc, min=0.0) / dv)
        lo, hi = torch.clamp(rho - move, min=0.0), torch.clamp(rho + move, max=1.0)
        a, b = -47.0, 47.0  # ln mu
        for _ in range(120):
            m = 0.5 * (a + b)
            if float((dv * torch.minimum(torch.maximum(s * math.exp(m), lo), hi)).sum()) >= volfrac:
                b = m
            else:
                a = m
        mu = math.exp(0.5 * (a + b))
        new = torch.minimum(torch.maximum(s * mu, lo), hi)
        return new, 1.0 / (mu * mu), float((new - rho).abs().max())

    def dv(self, r):
        return self.filter(torch.full(self.eshape, 1.0 / math.prod(self.eshape), dtype=torch.float64, device=_dev()), r, True)

    def cycle(self, rho, r):
        rt = self.filter(rho, r)
        t = self.solve(self.simp(rt))
        dc = self.filter(self.sens(rt, t), r, True)
        new, lam, _ = self.oc(rho, dc, self.dv(r), self.c["volfrac"])
        return new, t, float((self.q * t).sum()), lam, dc


def _p1(nf):
    """Interpolation from the nodes min(2I, nf) onto nodes 0..nf of one axis."""
    nc = (nf + 1) // 2
    p = torch.zeros(nf + 1, nc + 1, dtype=torch.float64, device=_dev())
    for i in range(nf + 1):
        if i % 2 == 0:
            p[i, i // 2] = 1.0
        elif i < nf:
            p[i, i // 2] = p[i, i // 2 + 1] = 0.5
        else:
            p[i, i // 2 + 1] = 1.0
    return p


def _along(ms, x):
    for ax, m in enumerate(ms):
        x = torch.movedim(torch.tensordot(m, x, dims=([1], [ax])), 0, ax)
    return x


class _Vcycle:
    """One V-cycle (damped Jacobi 0.9, one sweep each way, zero guess) with Galerkin operators found by probing."""

    def __init__(self, ref, k, nl):
        self.ref, self.k = ref, k
        self.apply, self.dinv, self.ps = [lambda x: ref.a_apply(k, x)], [1.0 / ref.a_diag(k)], []
        n = ref.eshape
        for level in range(1, nl):
            self.ps.append([_p1(m) for m in n])
            n = tuple((m + 1) // 2 for m in n)
            shape = tuple(m + 1 for m in n)
            idx = torch.meshgrid(*[torch.arange(m, device=_dev()) for m in shape], indexing="ij")
            offs = list(itertools.product((-1, 0, 1), repeat=ref.d))
            st = [torch.zeros(shape, dtype=torch.float64, device=_dev()) for _ in offs]
            for colour in itertools.product((0, 1, 2), repeat=ref.d):
                probe = torch.ones(shape, dtype=torch.float64, device=_dev())
                for i, cc in zip(idx, colour):
                    probe *= (i % 3 == cc)
                y = self.restrict(level - 1, self.apply[level - 1](self.prolong(level - 1, probe)))
                for s, o in zip(st, offs):
                    hit = torch.ones(shape, dtype=torch.bool, device=_dev())
                    for i, oo, cc, m in zip(idx, o, colour, shape):
                        hit &= ((i + oo) % 3 == cc) & (i + oo >= 0) & (i + oo < m)
                    s.copy_(torch.where(hit, y, s))

            def stencil(x, st=st, offs=offs, shape=shape):
                xp = F.pad(x, [1] * (2 * len(shape)))
                out = torch.zeros_like(x)
                for s, o in zip(st, offs):
                    out += s * xp[tuple(slice(1 + oo, 1 + oo + m) for oo, m in zip(o, shape))]
                return out

            self.apply.append(stencil)
            self.dinv.append(1.0 / st[len(offs) // 2])
        count = math.prod(shape)
        eye = torch.eye(count, dtype=torch.float64, device=_dev())
        self.dense = torch.stack([stencil(eye[i].reshape(shape)).reshape(-1) for i in range(count)], 1)

    def prolong(self, level, x):
        x = _along(self.ps[level], x)
        return self.ref.free * x if level == 0 else x

    def restrict(self, level, x):
        x = self.ref.free * x if level == 0 else x
        return _along([p.T for p in self.ps[level]], x)

    def __call__(self, b, level=0):
        if level == len(self.ps):
            return torch.linalg.solve(self.dense, b.reshape(-1)).reshape(b.shape)
        w = 0.9 * self.dinv[level]
        x = w * b
        x = x + self.prolong(level, self(self.restrict(level, b - self.apply[level](x)), level + 1))
        return x + w * (b - self.apply[level](x))


def exact(case, seed):
    c = case
    if c["kind"] == "batch" or (c["nz"] and c["nx"] * c["ny"] * c["nz"] > 3000000 and c["kind"] != "post"):
        return None  # minutes of unpreconditioned iterations
    ref = _Ref(c)
    rho = _density(c, seed).reshape(ref.eshape)
    kind = c["kind"]
    if kind in ("step", "solve", "grad"):
        if kind == "solve":
            return {"T": ref.solve(ref.simp(ref.filter(rho, c["rmin"]))).reshape(-1), "converged": None}
        new, t, comp, lam, dc = ref.cycle(rho, c["rmin"])
        if kind == "grad":
            return {"compliance": torch.tensor(comp, dtype=torch.float64), "grad": dc.reshape(-1)}
        return {"rho": new.reshape(-1), "T": t.reshape(-1), "scalars": np.array([comp, lam])}
    if kind == "run":
        r = ALPHA * max(c["nx"], c["ny"], c["nz"])
        grow = r > c["rmin"]
        eta = math.exp((math.log(c["rmin"]) - math.log(r)) / LP) if grow else 1.0
        comps, lams = [], []
        for _ in range(c["cycles"]):
            r = max(c["rmin"], eta * r) if grow else c["rmin"]
            rho, _, comp, lam, _ = ref.cycle(rho, r)
            comps.append(comp)
            lams.append(lam)
        return {"rho": rho.reshape(-1), "compliance": np.array(comps), "lam": np.array(lams)}
    if kind == "mgar":
        k0 = ref.simp(ref.filter(rho, c["rmin"]))
        k = ref.simp(ref.filter(_density(c, seed, salt=2).reshape(ref.eshape), c["rmin"]))
        t = _temperature(c, seed).reshape(ref.nshape)
        b = -ref.free * ref.k_apply(k - k0, ref.free * t)
        basis = torch.stack([t.reshape(-1), _Vcycle(ref, k0, _levels(c))(b).reshape(-1)], 1)
        basis = torch.linalg.qr(basis).Q
        w = torch.stack([ref.a_apply(k, basis[:, i].reshape(ref.nshape)).reshape(-1) for i in range(2)], 1)
        y = torch.linalg.solve(basis.T @ w, basis.T @ ref.q.reshape(-1))
        res = float(torch.linalg.norm(w @ y - ref.q.reshape(-1)) / torch.linalg.norm(ref.q))
        return {"T": basis @ y, "scalars": np.array([res]), "accepted": None}
    rt = ref.filter(rho, c["rmin"])
    t = _temperature(c, seed).reshape(ref.nshape)
    dcp = ref.sens(rt, t)
    if kind == "update":
        dc, dv = ref.filter(dcp, c["rmin"], True), ref.dv(c["rmin"])
        new, lam, change = ref.oc(rho, dc, dv, c["volfrac"])
        return {"dc": dc.reshape(-1), "dv": dv.reshape(-1), "rho": new.reshape(-1),
                "scalars": np.array([float((ref.q * t).sum()), lam, change])}
    # post-processing: nodal projection of -dcp, then the share of lattice points above the level
    r, reach = c["rmin"], int(math.ceil(c["rmin"] + 0.5))
    num, den = (torch.zeros(ref.nshape, dtype=torch.float64, device=_dev()) for _ in range(2))
    one = F.pad(torch.ones_like(dcp), [reach] * (2 * ref.d))
    val = F.pad(-dcp, [reach] * (2 * ref.d))
    for o in itertools.product(range(-reach, reach), repeat=ref.d):
        w = r - math.sqrt(sum((v + 0.5) ** 2 for v in o))
        if w > 0:
            sl = tuple(slice(reach + v, reach + v + n) for v, n in zip(o, ref.nshape))
            num.add_(val[sl], alpha=w)
            den.add_(one[sl], alpha=w)
    ns = num / den
    points = []
    for p in itertools.product((0.0, 0.25, 0.5, 0.75, 1.0), repeat=ref.d):
        s = torch.zeros(ref.eshape, dtype=torch.float64, device=_dev())
        for a, corner in enumerate(ref.corners):
            w = math.prod(x if o else 1 - x for x, o in zip(p, corner))
            if w:
                s.add_(ref.at(ns, a), alpha=w)
        points.append(s)
    lo, hi = -1.0, float(ns.max())
    total = len(points) * rho.numel()
    while lo < (mid := 0.5 * (lo + hi)) < hi:
        if sum(int((s > mid).sum()) for s in points) > c["volfrac"] * total:
            lo = mid
        else:
            hi = mid
    out = sum((s > hi).double() for s in points) / len(points)
    return {"rho": out.reshape(-1), "scalars": np.array([hi, float(out.mean())])}
