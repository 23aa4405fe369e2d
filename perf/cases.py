"""What is timed of this library: the calls that a simulation makes, on inputs shaped like its workloads.

Every case is one pass through the public entry points (``Grid``, ``Ensemble``, ``Mesh``, ``residual``)
with the handles and output buffers that a program keeps between calls.  The operations:

  jacobian  bind the iterate, assemble R and J in one fused pass: once per Newton iteration
  residual  bind the iterate, assemble R alone: line searches, explicit checks, the repeated application
  ensemble  R and J of many models of uneven sizes in one launch: uncertainty sweeps
  gradient  R(p, ln k) forward and its adjoint backward through autograd: inversion for the permeability
  jvp       J w without J: the operator of a matrix-free Krylov solver
  newton    one implicit Newton step (assembly, preconditioned BiCGStab, update)
  mesh      R and J on a faulted mesh given as connections

Sizes are the benchmark's and the tests' configurations, or of the same ranges with odd and ragged
extents.  Inputs follow ``paper_2304_11274_gb300/synth.py``'s distributions, drawn on the GPU.
"""
import math

import torch

from paper_2304_11274_gb300 import api

PHYSICS = dict(rho_ref=1000.0, p_ref=1.0e7, c_f=4.5e-10, mu=1.0e-3, g=9.81, dt=86400.0, c_r=0.0,
               dx=10.0, dy=10.0, dz=2.0)


def _case(op, nx, ny, nz, precision, connectivity=10, **more):
    return dict(op=op, nx=nx, ny=ny, nz=nz, precision=precision, connectivity=connectivity, **more)


def listed():
    return [
        # the smallest grid of the benchmark: latency, FP64 throughout, faces only
        dict(_case("jacobian", 32, 32, 32, "fp64", 6), name="jacobian_fp64_32cube"),
        # an ordinary model with odd extents and a compressible rock, faces only
        dict(_case("jacobian", 201, 117, 75, "mixed", 6, c_r=1e-9), name="jacobian_mixed_ragged"),
        # the benchmark's single grid, ten connections, mixed precision
        dict(_case("jacobian", 512, 512, 256, "mixed"), name="jacobian_mixed_512"),
        # the high-contrast layered medium in full FP64 (the reference run of a precision study)
        dict(_case("jacobian", 256, 256, 256, "fp64", layered=True), name="jacobian_fp64_layered"),
        # the paper's own grid, residual only (its repeated application of Algorithm 1)
        dict(_case("residual", 750, 994, 246, "mixed"), name="residual_mixed_750"),
        # twenty models of uneven sizes in one launch
        dict(op="ensemble", models=20, connectivity=10, precision="mixed", shapes=11, name="ensemble_mixed_20"),
        # gradient of a misfit with respect to pressure and log-permeability
        dict(_case("gradient", 128, 128, 128, "mixed"), name="gradient_mixed_128"),
        # the same in FP64 on a smaller model with odd extents (gradient checks, small inversions)
        dict(_case("gradient", 97, 83, 50, "fp64", c_r=1e-9), name="gradient_fp64_ragged"),
        # matrix-free operator application on the benchmark's grid
        dict(_case("jvp", 512, 512, 256, "mixed"), name="jvp_mixed_512"),
        # and in FP64 on an ordinary model, faces only
        dict(_case("jvp", 161, 119, 67, "fp64", 6), name="jvp_fp64_ragged"),
        # one implicit step, the whole call
        dict(_case("newton", 128, 128, 128, "mixed", rtol=1e-10), name="newton_mixed_128"),
        # a mesh with a fault and pinched-out cells
        dict(_case("mesh", 96, 96, 48, "mixed"), name="mesh_mixed_faulted"),
    ]


def _extent(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["jacobian", "jacobian", "residual", "ensemble", "gradient", "jvp", "newton", "mesh"])
    precision = rng.choice(["mixed", "mixed", "fp64"])
    conn = rng.choice([6, 10])
    c_r = rng.choice([0.0, 0.0, 1e-9])
    if op == "ensemble":
        return dict(op=op, models=rng.randint(2, 20), connectivity=conn, precision="mixed", shapes=rng.randint(0, 9999), c_r=c_r)
    # (fewest cells, most cells): a drawn case costs no more than the largest listed one
    few, most = {"jacobian": (5e3, 6e7), "residual": (5e3, 1.5e8), "gradient": (5e3, 2e6), "jvp": (5e3, 6e7),
                 "newton": (4e3, 8e5), "mesh": (4e3, 3e5)}[op]
    if precision == "fp64":
        most = {"jacobian": 1.2e7, "residual": 1.6e7, "jvp": 8e6, "gradient": 5e5, "newton": 1.5e5}.get(op, most)
    cells = _extent(rng, few, most)
    # extents around the cube root, the z extent the smallest as a rule
    side = cells ** (1.0 / 3.0)
    nx = max(8, _extent(rng, side, 2.5 * side))
    ny = max(6, _extent(rng, 0.7 * side, 1.6 * side))
    nz = max(3, min(256, cells // (nx * ny)))
    if op == "newton":  # well-conditioned steps, solved to the tests' tolerance
        return _case(op, nx, ny, nz, precision, conn, c_r=1e-8, dt=3600.0, rtol=1e-10)
    if op == "mesh":
        return _case(op, nx, ny, nz, precision, conn)
    c = _case(op, nx, ny, nz, precision, conn, c_r=c_r)
    if op == "jacobian" and rng.random() < 0.25:
        c["layered"] = True
    return c


# ---------------------------------------------------------------- inputs


def _phys(case):
    return dict(PHYSICS, c_r=case.get("c_r", 0.0) or 0.0, dt=case.get("dt", PHYSICS["dt"]), connectivity=case["connectivity"])


def _fields(case, seed):
    """Permeability, porosity, depth (FP64) and p, p^n in the path's type, on the GPU, from the seed."""
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    gen = torch.Generator(device="cuda").manual_seed(int(seed))
    ph = _phys(case)
    n = nx * ny * nz

    def uniform(count, lo, hi):
        return torch.rand(count, generator=gen, device="cuda", dtype=torch.float64).mul_(hi - lo).add_(lo)

    layer = torch.arange(nz, device="cuda", dtype=torch.float64)

    def spread(x):
        return x.view(nz, 1).expand(nz, nx * ny).reshape(-1)

    if case.get("layered"):
        lk = spread(uniform(nz, -18.0, -12.0))
        base = spread(5.0e6 + 2.5e7 * layer / max(nz - 1, 1))
    else:
        lk = torch.randn(n, generator=gen, device="cuda", dtype=torch.float64).mul_(0.5).sub_(13.0)
        base = spread(1.0e7 + ph["rho_ref"] * ph["g"] * layer * ph["dz"])
    log_k = lk * math.log(10.0)
    del lk
    poro = uniform(n, 0.1, 0.3)
    depth = spread((layer + 0.5) * ph["dz"])
    dt = torch.float32 if case["precision"] == "mixed" else torch.float64
    p = uniform(n, -1.0e5, 1.0e5).add_(base)
    if case.get("layered"):
        p.clamp_(5.0e6, 3.0e7)
    return dict(log_k=log_k, poro=poro, depth=depth, p=p.to(dt), pn=base.to(dt))


def _direction(n, seed):
    gen = torch.Generator(device="cuda").manual_seed(int(seed) * 7919 + 17)
    return torch.randn(n, generator=gen, device="cuda", dtype=torch.float64)


def _model_cases(case):
    """The ensemble's models: nx, ny ~ U{64..256}, nz ~ U{32..128}, as the benchmark draws them."""
    import random
    rng = random.Random(case["shapes"])
    return [_case("jacobian", rng.randint(64, 256), rng.randint(64, 256), rng.randint(32, 128), "mixed", case["connectivity"],
                  c_r=case.get("c_r", 0.0)) for _ in range(case["models"])]


def _links(nx, ny, nz, connectivity):
    """Cell pairs of the structured links, each once, on the GPU."""
    lin = torch.arange(nx * ny * nz, device="cuda").view(nz, ny, nx)
    pairs = [(lin[:, :, :-1], lin[:, :, 1:]), (lin[:, :-1], lin[:, 1:]), (lin[:-1], lin[1:])]
    if connectivity == 10:
        pairs += [(lin[:, :-1, :-1], lin[:, 1:, 1:]), (lin[:, :-1, 1:], lin[:, 1:, :-1])]
    return torch.cat([a.reshape(-1) for a, _ in pairs]), torch.cat([b.reshape(-1) for _, b in pairs])


def _mesh(case, seed):
    """A corner-point-like mesh: the block x >= nx/2 thrown down by half a layer, 5 % of the cells pinched out."""
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    ph = _phys(case)
    gen = torch.Generator(device="cuda").manual_seed(int(seed))

    def rand(count):
        return torch.rand(count, generator=gen, device="cuda", dtype=torch.float64)

    n0, xf, dz = nx * ny * nz, nx // 2, ph["dz"]
    lin = torch.arange(n0, device="cuda")
    i, k = lin % nx, lin // (nx * ny)
    depth = (k + 0.5) * dz + torch.where(i >= xf, 0.5 * dz, 0.0)
    a, b = _links(nx, ny, nz, case["connectivity"])
    ia, ib = a % nx, b % nx
    keep = ~((torch.minimum(ia, ib) < xf) & (torch.maximum(ia, ib) >= xf))
    left = lin[i == xf - 1]
    up = left[k[left] >= 1]
    a = torch.cat([a[keep], left, up])
    b = torch.cat([b[keep], left + 1, up + 1 - nx * ny])
    # which cells are pinched out belongs to the mesh, as its extents do: the values on it come from the seed
    holes = torch.Generator(device="cuda").manual_seed(1000003 * nx + 1009 * ny + nz)
    active = torch.rand(n0, generator=holes, device="cuda") >= 0.05
    active[0] = True
    keep = active[a] & active[b]
    idx = torch.cumsum(active, 0) - 1
    ci, cj = idx[a[keep]], idx[b[keep]]
    n = int(active.sum())
    T = torch.pow(10.0, torch.randn(ci.numel(), generator=gen, device="cuda", dtype=torch.float64) * 0.5 - 12.7)
    V = ph["dx"] * ph["dy"] * dz * (0.8 + 0.4 * rand(n))
    poro = 0.1 + 0.2 * rand(n)
    depth = depth[active]
    base = 1.0e7 + ph["rho_ref"] * ph["g"] * (depth - 0.5 * dz)
    p = base + 1.0e5 * (2.0 * rand(n) - 1.0)
    dt = torch.float32 if case["precision"] == "mixed" else torch.float64
    return dict(n=n, ci=ci, cj=cj, T=T, V=V, poro=poro, depth=depth, p=p.to(dt), pn=base.to(dt))


# ---------------------------------------------------------------- a program's state and one pass


def _grid(case, f):
    g = api.Grid(case["nx"], case["ny"], case["nz"], _phys(case), case["precision"], torch.exp(f["log_k"]), f["poro"], f["depth"])
    g.set_state(f["p"], f["pn"])
    return g


def prepare(case, seed):
    op = case["op"]
    if op == "ensemble":
        grids = [_grid(c, _fields(c, seed * 1000 + m)) for m, c in enumerate(_model_cases(case))]
        ens = api.Ensemble(grids)
        return dict(op=op, grids=grids, ens=ens, outs=ens.allocate_outputs())
    if op == "mesh":
        m = _mesh(case, seed)
        mesh = api.Mesh(m["n"], m["ci"].cpu().numpy(), m["cj"].cpu().numpy(), m["T"], m["V"], m["poro"], m["depth"],
                        _phys(case), case["precision"])
        mesh.set_state(m["p"], m["pn"])
        return dict(op=op, mesh=mesh, p=m["p"], outs=mesh.empty_outputs())
    f = _fields(case, seed)
    g = _grid(case, f)
    s = dict(op=op, grid=g, p=f["p"])
    if op == "jacobian":
        s["outs"] = g.empty_outputs()
    elif op == "residual":
        s["R"] = torch.empty(g.n, dtype=torch.float64, device="cuda")
    elif op == "gradient":
        s["p"] = f["p"].requires_grad_(True)
        s["log_k"] = f["log_k"].requires_grad_(True)
        s["v"] = _direction(g.n, seed)
    elif op == "jvp":
        s["w"] = _direction(g.n, seed)
        s["Jw"] = torch.empty(g.n, dtype=torch.float64, device="cuda")
    elif op == "newton":
        s["iterate"] = torch.empty_like(f["p"])
        s["rtol"] = case["rtol"]
    return s


def run(state):
    op = state["op"]
    if op == "ensemble":
        state["ens"].assemble()
        return state["outs"]
    if op == "mesh":
        state["mesh"].set_pressure(state["p"])
        return state["mesh"].assemble(*state["outs"])
    g = state["grid"]
    if op == "jacobian":
        g.set_pressure(state["p"])
        return g.assemble_jacobian(*state["outs"])
    if op == "residual":
        g.set_pressure(state["p"])
        return g.assemble_residual(state["R"])
    if op == "gradient":
        R = api.residual(g, state["p"], state["log_k"])
        g_p, g_lnk = torch.autograd.grad(R, (state["p"], state["log_k"]), state["v"])
        return R.detach(), g_p, g_lnk
    if op == "jvp":
        g.set_pressure(state["p"])
        return g.jvp(state["w"], out=state["Jw"])[0]
    p = state["iterate"]  # newton: the step updates its iterate in place
    p.copy_(state["p"])
    _, R, _ = g.newton_step(p, rtol=state["rtol"], want_residual=True)
    return p, R


# ---------------------------------------------------------------- what a pass cannot do without


def _owned_links(nx, ny, nz, connectivity):
    m = (nx - 1) * ny * nz + nx * (ny - 1) * nz + nx * ny * (nz - 1)
    return m + (2 * (nx - 1) * (ny - 1) * nz if connectivity == 10 else 0)


def work(case):
    """Bytes: the fields a pass reads and the results it writes, each once.  Flops: density 12 and accumulation 16 per
    cell; per link 20 for the flux and its derivatives (8 for the flux alone) and 2 or 4 additions at its ends."""
    op = case["op"]
    if op == "ensemble":
        parts = [work(c) for c in _model_cases(case)]
        return {k: sum(w[k] for w in parts) for k in ("bytes", "flops")}
    n, m = case["nx"] * case["ny"] * case["nz"], _owned_links(case["nx"], case["ny"], case["nz"], case["connectivity"])
    r = 4 if case["precision"] == "mixed" else 8
    mixed = case["precision"] == "mixed"
    fields = n * (3 * r + 8 + (r if case.get("c_r") else 0)) + m * r  # p, p^n, z, m^n, phi0; owned T
    jac = r * (n + 2 * m) + (8 * n if mixed else 0)
    cell, flux, link = 28 * n, 10 * m, 24 * m
    if op == "mesh":  # columns and T per entry
        return {"bytes": 0.95 * (n * (3 * r + 16 + 8) + (n + 2 * m) * 4 + m * r + jac), "flops": 0.95 * (cell + link)}
    if op == "jacobian":
        return {"bytes": fields + 8 * n + jac, "flops": cell + link}
    if op == "residual":
        return {"bytes": fields + 8 * n, "flops": cell + flux}
    if op == "jvp":
        return {"bytes": fields + 16 * n, "flops": cell + link + 4 * m}
    if op == "gradient":  # p, p^n, z, m^n, phi0, ln k, v in; R, g_p, g_lnk out
        return {"bytes": n * (3 * r + 8 + (r if case.get("c_r") else 0) + 16 + 16 + r), "flops": 2 * (cell + 10 * m) + link}
    # newton: the assembly, and J read twice for one Krylov iteration at least
    return {"bytes": fields + 8 * n + 3 * jac + r * n, "flops": cell + link + 8 * m}


# ---------------------------------------------------------------- the same in 64 bits


class _Exact:
    """Eq. vk on a set of links in plain FP64 torch, each link seen from both of its ends."""

    def __init__(self, ph, f, dtype, V):
        d = torch.float64
        self.ph, self.p, self.pn = ph, f["p"].detach().to(d), f["pn"].to(d)
        self.z = f["depth"].to(dtype).to(d)  # the mixed path holds depth in FP32
        self.rho = ph["rho_ref"] * torch.exp(ph["c_f"] * (self.p - ph["p_ref"]))
        phi0, vdt, c_r, c_f = f["poro"], V / ph["dt"], ph["c_r"], ph["c_f"]
        rel = 1.0 + c_r * (self.p - ph["p_ref"])
        rho_n = ph["rho_ref"] * torch.exp(c_f * (self.pn - ph["p_ref"]))
        mass_n = vdt * phi0 * (1.0 + c_r * (self.pn - ph["p_ref"])) * rho_n
        dp = self.p - self.pn
        self.A = vdt * phi0 * c_r * dp * self.rho + mass_n * torch.expm1(c_f * dp)
        self.dA = vdt * phi0 * self.rho * (c_r + rel * c_f)

    def flux(self, T, a, b):
        """F from a to b, and dphi; a, b index (or slice) the flat or shaped fields."""
        pa, pb, ra, rb = self.p[a], self.p[b], self.rho[a], self.rho[b]
        hg = 0.5 * self.ph["g"] * (self.z[a] - self.z[b])
        dphi = (pa - pb) - (ra + rb) * hg
        Tm = T / self.ph["mu"]
        return Tm * torch.where(dphi > 0, ra, rb) * dphi, dphi, Tm, hg

    def both(self, T, a, b):
        """F_ab; dF_ab/dp_a, dF_ab/dp_b by a's upwind rule; the same flux's two by b's rule (they differ at a tie)."""
        F, dphi, Tm, hg = self.flux(T, a, b)
        ra, rb, cf = self.rho[a], self.rho[b], self.ph["c_f"]
        out = [F]
        for up in (dphi > 0, dphi >= 0):
            r = torch.where(up, ra, rb)
            out.append(Tm * (r * (1.0 - cf * ra * hg) + torch.where(up, cf * ra, 0.0) * dphi))
            out.append(Tm * (r * (-1.0 - cf * rb * hg) + torch.where(up, 0.0, cf * rb) * dphi))
        return out


def _structured(case, f):
    """The exact fields shaped (nz, ny, nx) and the links as (slices a, slices b, T, slot of b in a's row, slot of a in b's row)."""
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    ph = _phys(case)
    shaped = {k: v.detach().view(nz, ny, nx) for k, v in f.items()}
    e = _Exact(ph, shaped, torch.float32 if case["precision"] == "mixed" else torch.float64, ph["dx"] * ph["dy"] * ph["dz"])
    k = torch.exp(shaped["log_k"])
    dx, dy, dz = ph["dx"], ph["dy"], ph["dz"]
    lo, hi, al = slice(None, -1), slice(1, None), slice(None)
    geo = [((al, al, lo), (al, al, hi), dy * dz / dx, 6, 4), ((al, lo, al), (al, hi, al), dx * dz / dy, 8, 2),
           ((lo, al, al), (hi, al, al), dx * dy / dz, 10, 0)]
    if case["connectivity"] == 10:
        d = dz * dx * dy / (dx * dx + dy * dy)
        geo += [((al, lo, lo), (al, hi, hi), d, 9, 1), ((al, lo, hi), (al, hi, lo), d, 7, 3)]

    def links():
        for a, b, s, sa, sb in geo:
            yield a, b, 2.0 * k[a] * k[b] / (k[a] + k[b]) * s, sa, sb

    return e, k, links


_OFF = {0: (-1, 0, 0), 1: (0, -1, -1), 2: (0, -1, 0), 3: (0, -1, 1), 4: (0, 0, -1), 5: (0, 0, 0), 6: (0, 0, 1), 7: (0, 1, -1),
        8: (0, 1, 0), 9: (0, 1, 1), 10: (1, 0, 0)}


def _exact_rows(case, f):
    """R, the eleven slots of every row (nz, ny, nx, 11) and which of them exist."""
    e, _, links = _structured(case, f)
    shape = e.p.shape
    slots = torch.zeros(*shape, 11, device="cuda", dtype=torch.float64)
    there = torch.zeros(*shape, 11, device="cuda", dtype=torch.bool)
    there[..., 5] = True
    R, diag = e.A.clone(), e.dA.clone()
    for a, b, T, sa, sb in links():
        F, aa, ab, ba, bb = e.both(T, a, b)
        R[a] += F
        R[b] -= F
        diag[a] += aa
        diag[b] -= bb
        slots[a + (sa,)] = ab
        slots[b + (sb,)] = -ba
        there[a + (sa,)] = True
        there[b + (sb,)] = True
    slots[..., 5] = diag
    return R, slots, there


def _exact_jacobian(case, f):
    R, slots, there = _exact_rows(case, f)
    diag = slots[..., 5].reshape(-1).clone()
    vals = torch.masked_select(slots, there)
    return R.reshape(-1), vals, diag if case["precision"] == "mixed" else None


def _exact_newton(case, f):
    """p + delta with J delta = -R solved far below the case's tolerance (BiCGStab, scaled by the diagonal)."""
    R, slots, there = _exact_rows(case, f)
    nz, ny, nx = R.shape
    dinv = 1.0 / slots[..., 5]
    used = [(s, slots[..., s].contiguous(), _OFF[s]) for s in range(11) if bool(there[..., s].any())]
    del slots, there

    def mul(x):
        xp = torch.nn.functional.pad(x, (1, 1, 1, 1, 1, 1))
        y = torch.zeros_like(x)
        for _, c, (oz, oy, ox) in used:
            y.addcmul_(c, xp[1 + oz:1 + oz + nz, 1 + oy:1 + oy + ny, 1 + ox:1 + ox + nx])
        return y

    def dot(a, b):
        return (a * b).sum()

    b = -R
    x, r = torch.zeros_like(b), b.clone()
    rh, p = r.clone(), r.clone()
    rho, stop = dot(rh, r), 1e-13 * float(b.norm())
    for it in range(4000):
        v = mul(dinv * p)
        alpha = rho / dot(rh, v)
        s = r - alpha * v
        t = mul(dinv * s)
        omega = dot(t, s) / dot(t, t)
        x = x + dinv * (alpha * p + omega * s)
        r = s - omega * t
        if it % 8 == 0 and not float(r.norm()) > stop:
            break
        new = dot(rh, r)
        p = r + (new / rho) * (alpha / omega) * (p - omega * v)
        rho = new
    if not float((b - mul(x)).norm()) <= 1e-11 * float(b.norm()):
        return None
    return (f["p"].double().view(nz, ny, nx) + x).reshape(-1), R.reshape(-1)


def _exact_mesh(case, seed):
    f = _mesh(case, seed)
    e = _Exact(_phys(case), f, torch.float32 if case["precision"] == "mixed" else torch.float64, f["V"])
    a, b, n = f["ci"], f["cj"], f["n"]
    F, aa, ab, ba, bb = e.both(f["T"], a, b)
    R, diag = e.A.clone(), e.dA.clone()
    R.index_add_(0, a, F)
    R.index_add_(0, b, F, alpha=-1)
    diag.index_add_(0, a, aa)
    diag.index_add_(0, b, bb, alpha=-1)
    own = torch.arange(n, device="cuda")
    key = torch.cat([a * n + b, b * n + a, own * n + own])
    vals = torch.cat([ab, -ba, diag])[torch.argsort(key)]
    return R, vals, diag if case["precision"] == "mixed" else None


def exact(case, seed):
    op = case["op"]
    if op == "ensemble":
        return [_exact_jacobian(c, _fields(c, seed * 1000 + m)) for m, c in enumerate(_model_cases(case))]
    if op == "mesh":
        return _exact_mesh(case, seed)
    f = _fields(case, seed)
    if op == "jacobian":
        return _exact_jacobian(case, f)
    if op == "newton":
        return _exact_newton(case, f)
    e, k, links = _structured(case, f)
    if op == "residual":
        R = e.A
        for a, b, T, _, _ in links():
            F = e.flux(T, a, b)[0]
            R[a] += F
            R[b] -= F
        return R.reshape(-1)
    v = _direction(e.p.numel(), seed).view(e.p.shape)
    if op == "jvp":
        out = e.dA * v
        for a, b, T, _, _ in links():
            _, aa, ab, ba, bb = e.both(T, a, b)
            out[a] += aa * v[a] + ab * v[b]
            out[b] -= ba * v[a] + bb * v[b]
        return out.reshape(-1)
    R, g_p, g_lnk = e.A.clone(), e.dA * v, torch.zeros_like(v)
    for a, b, T, _, _ in links():
        F, aa, ab, ba, bb = e.both(T, a, b)
        R[a] += F
        R[b] -= F
        g_p[a] += v[a] * aa - v[b] * ba
        g_p[b] += v[a] * ab - v[b] * bb
        w = (v[a] - v[b]) * F / (k[a] + k[b])
        g_lnk[a] += w * k[b]
        g_lnk[b] += w * k[a]
    return R.reshape(-1), g_p.reshape(-1), g_lnk.reshape(-1)
