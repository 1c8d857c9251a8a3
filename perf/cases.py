"""The work a user has this solver do, as cases that can be timed and checked.

A case names a grid, the options and what is called on it:

  "rhs"    a program with its own time integrator: hand over a new state (set_state), take
           its right-hand side (rhs), all on the device
  "step"   a run: load a state, advance it some steps at the CFL time step (step), fetch it
  "c2p"    the primitives of a loaded state (con2prim), for output or analysis
  "batch"  a parameter study: many uneven instances loaded, advanced together and fetched

`prepare` builds the states (a Kerr-Schild slice in BSSN variables with seeded magnetised gas)
and the context; `run` is one pass through the public calls; `exact` evaluates the same
equations in plain torch in 64 bits, without the package.
"""
import math
import random
from types import SimpleNamespace

import numpy as np
import torch

import paper_2508_18221_gb300 as pkg

GAMMA = 4.0 / 3.0
RHO_ATM, EPS_ATM = 1e-12, 1e-10          # the floors of the options' defaults
BAND = (math.pi / 8, 7 * math.pi / 8)


# ------------------------------------------------------------------------------- cases
def _single(name, do, shape, r, **kw):
    c = dict(name=name, do=do, n_elem=shape[0], n_r=shape[1], n_theta=shape[2], n_phi=shape[3], r_min=r[0],
             r_max=r[1], spin=0.5, profile="powerlaw", theta_basis=0, precision=0, integrator=0, glm=0,
             contraction=0, cfl=0.3, steps=0)
    c.update(kw)
    return c


def listed():
    torus = dict(spin=0.9, profile="torus")
    return [
        # the 4,608-node instance: the smallest grid of the shipped workloads, where one call's
        # launches and the fixed start of each kernel count
        _single("rhs_small", "rhs", (2, 12, 12, 16), (1.8, 20.0)),
        _single("step_small", "step", (2, 12, 12, 16), (1.8, 20.0), steps=20),
        # odd node counts that fill no tile
        _single("rhs_ragged", "rhs", (5, 21, 27, 40), (1.8, 40.0), spin=0.7),
        # the other integrator with divergence cleaning, medium grid
        _single("step_rk4_glm", "step", (3, 18, 20, 32), (1.8, 30.0), integrator=1, glm=1, steps=5),
        # the 393,216-node torus: one right-hand side, a run in FP64 and in mixed precision, the
        # primitives of a loaded state
        _single("rhs_torus", "rhs", (8, 24, 32, 64), (1.5, 100.0), **torus),
        _single("step_torus", "step", (8, 24, 32, 64), (1.5, 100.0), steps=3, **torus),
        _single("step_torus_mixed", "step", (8, 24, 32, 64), (1.5, 100.0), precision=1, steps=3, **torus),
        _single("c2p_torus", "c2p", (8, 24, 32, 64), (1.5, 100.0), **torus),
        # the whole sphere on the Fourier theta basis (near the axis the metric fields are not
        # smooth there: small time steps)
        _single("step_sphere", "step", (8, 24, 32, 64), (1.5, 100.0), theta_basis=1, cfl=3e-4, steps=3, **torus),
        # the largest instance, 4.2 M nodes, mixed precision
        _single("step_large_mixed", "step", (16, 32, 64, 128), (1.3, 500.0), spin=0.94, profile="torus", precision=1,
                steps=2),
        # uneven batches (orders 8 .. 32, 2 .. 8 elements, 16 .. 64 azimuthal nodes), both precisions
        dict(name="batch", do="batch", instances=32, mix=1004, precision=0, steps=2),
        dict(name="batch_mixed", do="batch", instances=32, mix=2004, precision=1, steps=2),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    do = rng.choice(["rhs", "rhs", "step", "step", "step", "step", "c2p", "batch"])
    if do == "batch":
        return dict(do="batch", instances=_log_int(rng, 3, 32), mix=rng.randrange(1 << 20), precision=rng.randrange(2),
                    steps=rng.choice([1, 2]))
    precision = rng.randrange(2) if do == "step" else 0     # mixed precision is for runs
    fourier = int(rng.random() < 0.2)
    most = 4.0e6 if precision else 6.0e5
    while True:
        shape = (_log_int(rng, 1, 16), _log_int(rng, 6, 40), _log_int(rng, 6, 96), 2 * _log_int(rng, 4, 64))
        if 1.5e3 <= math.prod(shape) <= most:
            break
    r_min = rng.uniform(1.5, 1.9)
    c = _single("", do, shape, (r_min, r_min * rng.uniform(1.5, 2.2) ** min(shape[0], 7)), spin=rng.uniform(0.0, 0.95),
                theta_basis=fourier, precision=precision, integrator=int(rng.random() < 0.2),
                glm=int(rng.random() < 0.2), contraction=int(rng.random() < 0.1), cfl=3e-4 if fourier else 0.1)
    if do == "step":
        c["steps"] = 1 if math.prod(shape) > 3e5 else _log_int(rng, 1, 8)
    del c["name"]
    return c


def _instances(case):
    """The single-instance cases that a case is made of."""
    if case["do"] != "batch":
        return [case]
    rng = random.Random(case["mix"])
    out = []
    for _ in range(case["instances"]):
        n, spin = rng.choice([8, 12, 16, 24, 32]), rng.uniform(0.0, 0.99)
        r_h = 1.0 + math.sqrt(1.0 - spin * spin)
        out.append(_single("", "step", (rng.randint(2, 8), n, n, rng.choice([16, 32, 64])), (0.9 * r_h, 50.0), spin=spin,
                           precision=case["precision"], steps=case["steps"], cfl=0.1, rho0=rng.uniform(5e-3, 2e-2)))
    return out


def _nodes(c):
    return c["n_elem"] * c["n_r"] * c["n_theta"] * c["n_phi"]


def work(case):
    nbytes = flops = 0.0
    for c in _instances(case):
        p, nv = _nodes(c), 32 + c["glm"]
        if c["do"] == "c2p":
            nbytes += 8.0 * p * (15 + 7)          # metric and conserved variables in, primitives out
            flops += 300.0 * p
            continue
        nbytes += 8.0 * p * 2 * nv
        n = (c["n_r"], c["n_theta"], c["n_phi"])
        # the reflection symmetry of every operator halves the products: n per value and pass
        derivs = sum(k * m for k, m in zip((29 + 33, 29 + 22, 29 + 11), n))
        evals = 1 if c["do"] == "rhs" else c["steps"] * (4 if c["integrator"] else 3)
        # about 2,000 for the pointwise terms: curvature, gauge, sources, fluxes, recovery
        flops += p * (evals * (derivs + 2000.0) + c["steps"] * (nv * n[0] + 8 * n[1] + nv * n[2]))
    return {"bytes": nbytes, "flops": flops}


# ------------------------------------------------------------- grid and spectral operators
def _bary_diff(x):
    """Differentiation matrix on the nodes x (extended precision), barycentric form."""
    d = x[:, None] - x[None, :]
    np.fill_diagonal(d, 1)
    w = 1 / np.prod(2 * d, axis=1)
    m = (w[None, :] / w[:, None]) / d
    np.fill_diagonal(m, 0)
    np.fill_diagonal(m, -m.sum(axis=1))
    return m


def _sigma(k, kmax):
    return np.exp(-36.0 * (k / kmax) ** 8)


def _cheb_filter(n, lobatto):
    if lobatto:
        j = np.arange(n)
        T = np.cos(np.pi * np.outer(j, j) / (n - 1))                   # T_k at cos(j pi / (n - 1))
        c = np.where((j == 0) | (j == n - 1), 2.0, 1.0)
        C = 2.0 / (n - 1) * T / c[:, None] / c[None, :]                # [k, j]
        return (T.T * _sigma(j, n - 1)[None, :]) @ C
    k, j = np.arange(n), np.arange(n)
    T = np.cos(np.pi * np.outer(k, 2 * j + 1) / (2 * n))               # [k, j]
    C = np.where(k == 0, 1.0, 2.0)[:, None] / n * T
    return (T.T * _sigma(k, n - 1)[None, :]) @ C


def _fourier(n):
    """(derivative matrix, filter matrix) on n uniform nodes of a period."""
    d = np.arange(n)
    t = np.tan(np.pi * np.where(d == 0, 1, d) / n)
    row = np.where(d == 0, 0.0, 0.5 * (-1.0) ** d / t)
    if n % 2 == 0:
        row[n // 2] = 0.0
    k = np.where(d <= n // 2, d, n - d).astype(float)
    s = np.where(k > n / 3.0, 0.0, _sigma(k, n / 2.0))
    flt = (s[None, :] * np.cos(2 * np.pi * (np.outer(d, d) % n) / n)).sum(axis=1) / n
    idx = (d[:, None] - d[None, :]) % n
    return row[idx], flt[idx]


def _grid(c):
    E, nr, nt, npf = c["n_elem"], c["n_r"], c["n_theta"], c["n_phi"]
    dev = torch.device("cuda")

    def put(a):
        return torch.from_numpy(np.array(a, dtype=np.float64)).to(dev)

    pi = np.arctan(np.longdouble(1)) * 4
    b = c["r_min"] * (c["r_max"] / c["r_min"]) ** (np.arange(E + 1) / E)
    b[0], b[-1] = c["r_min"], c["r_max"]
    xr = -np.cos(pi * np.arange(nr, dtype=np.longdouble) / (nr - 1))
    r = 0.5 * (b[:-1] + b[1:])[:, None] + 0.5 * (b[1:] - b[:-1])[:, None] * xr[None, :].astype(float)
    g = SimpleNamespace(E=E, nr=nr, nt=nt, npf=npf, fourier=c["theta_basis"] == 1)
    if g.fourier:
        th = (np.arange(nt) + 0.5) * np.pi / nt
        D, F = _fourier(2 * nt)
        g.Dt, g.Ft = put(D[:nt]), put(F[:nt])
    else:
        xt = -np.cos(pi * (2 * np.arange(nt, dtype=np.longdouble) + 1) / (2 * nt))
        th = BAND[0] + 0.5 * (BAND[1] - BAND[0]) * (1.0 + xt.astype(float))
        g.Dt = put(_bary_diff(xt) * (2 / (BAND[1] - BAND[0])))
        g.Ft = put(_cheb_filter(nt, False))
    g.Dr, g.Fr = put(_bary_diff(xr)), put(_cheb_filter(nr, True))
    Dp, Fp = _fourier(npf)
    g.Dp, g.Fp = put(Dp), put(Fp)
    g.scale = put(2.0 / (b[1:] - b[:-1]))
    g.r, g.th = put(r), put(th)
    # end weight of Clenshaw-Curtis quadrature on nr Lobatto nodes
    n = nr - 1
    g.w_end = 1.0 / (n * n - 1.0) if n % 2 == 0 else 1.0 / (n * n)
    return g


def _d_r(g, u):
    return torch.einsum("ij,...ejtp->...eitp", g.Dr, u) * g.scale[:, None, None, None]


def _along_theta(g, m, u, parity):
    if g.fourier:  # the line continued across the pole: parity u(theta, phi + pi)
        u = torch.cat([u, parity * torch.flip(torch.roll(u, g.npf // 2, -1), [-2])], dim=-2)
    return torch.einsum("ij,...jp->...ip", m, u)


def _d_t(g, u, parity):
    return _along_theta(g, g.Dt, u, parity)


def _d_p(g, u):
    return torch.einsum("ij,...j->...i", g.Dp, u)


def _mean_ends(g, u):
    """Both copies of every duplicated interface node replaced by their mean."""
    u = u.clone()
    if g.E > 1:
        m = 0.5 * (u[..., :-1, -1, :, :] + u[..., 1:, 0, :, :])
        u[..., :-1, -1, :, :] = m
        u[..., 1:, 0, :, :] = m
    return u


# sign of each variable across the pole: gammatilde, phi, Atilde, K, Gammatilde, alpha, beta, B driver,
# then the densities D, S, tau, B, and the scalar psi
_PARITY = [1, -1, 1, 1, -1, 1, 1, 1, -1, 1, 1, -1, 1, 1, 1, -1, 1, 1, 1, -1, 1, 1, -1, 1, -1, -1, 1, -1, -1, -1, 1, -1, 1]
_SECOND = [0, 1, 2, 3, 4, 5, 6, 17, 18, 19, 20]


def _par(g, idx):
    return torch.tensor([float(_PARITY[i]) for i in idx], device=g.r.device, dtype=torch.float64)[:, None, None, None, None]


# ------------------------------------------------------------------------------ tensor algebra
def _con(spec, *xs):
    """einsum over leading tensor indices of extent 3; the trailing axes are the points."""
    ins, out = spec.split("->")
    ins = ins.split(",")
    summed = sorted(set("".join(ins)) - set(out))
    total = None
    for n in range(3 ** len(summed)):
        at = {s: n // 3 ** k % 3 for k, s in enumerate(summed)}
        term = None
        for letters, x in zip(ins, xs):
            x = x[tuple(at.get(q, slice(None)) for q in letters)]
            left = [q for q in letters if q not in at]
            rest = x.dim() - len(left)
            x = x.permute([left.index(q) for q in sorted(left, key=out.index)] + list(range(len(left), x.dim())))
            x = x.reshape([3 if q in left else 1 for q in out] + list(x.shape[x.dim() - rest:] if rest else []))
            term = x if term is None else term * x
        total = term if total is None else total + term
    return total


def _sym(six):
    return torch.stack([torch.stack([six[i] for i in row]) for row in ((0, 1, 2), (1, 3, 4), (2, 4, 5))])


def _six(t):
    return [t[0, 0], t[0, 1], t[0, 2], t[1, 1], t[1, 2], t[2, 2]]


def _det(m):
    return (m[0, 0] * (m[1, 1] * m[2, 2] - m[1, 2] * m[2, 1]) - m[0, 1] * (m[1, 0] * m[2, 2] - m[1, 2] * m[2, 0])
            + m[0, 2] * (m[1, 0] * m[2, 1] - m[1, 1] * m[2, 0]))


def _inv(m):
    d = _det(m)
    c = [m[1, 1] * m[2, 2] - m[1, 2] ** 2, m[0, 2] * m[1, 2] - m[0, 1] * m[2, 2], m[0, 1] * m[1, 2] - m[0, 2] * m[1, 1],
         m[0, 0] * m[2, 2] - m[0, 2] ** 2, m[0, 1] * m[0, 2] - m[0, 0] * m[1, 2], m[0, 0] * m[1, 1] - m[0, 1] ** 2]
    return _sym([x / d for x in c])


# ------------------------------------------------------------------------------- initial states
def _slice(spin, r, th):
    """The 24 BSSN and gauge variables of the Kerr-Schild slice (M = 1) at (r, theta)."""
    def fields(r, th):
        s2 = torch.sin(th) ** 2
        sig = r * r + (spin * torch.cos(th)) ** 2
        h = 2.0 * r / sig
        o = torch.zeros_like(sig)
        gam = _sym([1.0 + h, o, -spin * s2 * (1.0 + h), sig, o, s2 * (sig + spin * spin * s2 * (1.0 + h))])
        gt = gam * _det(gam) ** (-1.0 / 3.0)
        return gam, torch.stack([h / (1.0 + h), o, o]), (1.0 + h) ** -0.5, gt, _inv(gt)

    one, zero = torch.ones_like(r), torch.zeros_like(r)
    (gam, beta, alpha, gt, _), by_r = torch.func.jvp(fields, (r, th), (one, zero))
    _, by_t = torch.func.jvp(fields, (r, th), (zero, one))
    dgam, dbeta, dgti = (torch.stack([by_r[k], by_t[k], torch.zeros_like(by_r[k])]) for k in (0, 1, 4))
    lie = _con("k,kij->ij", beta, dgam) + _con("kj,ik->ij", gam, dbeta) + _con("ik,jk->ij", gam, dbeta)
    Kij = lie / (2.0 * alpha)
    phi = torch.log(_det(gam)) / 12.0
    K = _con("ij,ij->", _inv(gam), Kij)
    At = torch.exp(-4.0 * phi) * (Kij - gam * K / 3.0)
    Gam = -_con("jji->i", dgti)
    return _six(gt) + [phi] + _six(At) + [K] + list(Gam) + [alpha] + list(beta) + [zero, zero, zero]


def _state(c, g, seed):
    """Canonical state [nv, E, Nr, Nt, Np]: the slice with gas falling in, density and pressure with
    seeded noise of 1e-3, and a poloidal field from a vector potential."""
    shape = (g.E, g.nr, g.nt, g.npf)
    r, th = torch.broadcast_tensors(g.r[:, :, None, None], g.th[None, None, :, None])
    U = torch.zeros((32 + c["glm"],) + shape, dtype=torch.float64, device=g.r.device)
    for v, f in enumerate(_slice(c["spin"], r.contiguous(), th.contiguous())):
        U[v] = f
    gen = torch.Generator(device=g.r.device)
    gen.manual_seed(seed)
    at = (torch.arange(g.E)[:, None] * (g.nr - 1) + torch.arange(g.nr)[None, :]).to(g.r.device)

    def noise():  # the two copies of an interface node get the same draw
        x = torch.rand((g.E * (g.nr - 1) + 1, g.nt, g.npf), generator=gen, device=g.r.device, dtype=torch.float64)
        return 1.0 + 1e-3 * (2.0 * x[at] - 1.0)

    if c["profile"] == "torus":
        rho_c = torch.exp(-((r - 10.0) ** 2 + (10.0 * torch.cos(th)) ** 2) / 8.0) + 1e-4
        A = 8.4e-3 * torch.clamp(rho_c - 2e-3, min=0.0)
    else:
        rho_c = c.get("rho0", 1e-2) * r ** -1.5
        A = 0.05 * torch.clamp(rho_c - 2e-3, min=0.0) * torch.sin(th) ** 2
    rho = rho_c * noise()
    p = 1e-3 * rho_c ** GAMMA * noise()
    v = torch.zeros((3,) + shape, dtype=torch.float64, device=g.r.device)
    v[0] = -0.3 * torch.sqrt(2.0 / r) / torch.sqrt(1.0 + 2.0 / r)
    A = A.expand(shape)
    U[29], U[30] = _d_t(g, A, 1.0), -_d_r(g, A)
    gam = torch.exp(4.0 * U[6]) * _sym(U[0:6])
    sg = torch.sqrt(_det(gam))
    B = U[29:32] / sg
    f = _fluid(rho, v, p / ((GAMMA - 1.0) * rho), B, gam)
    U[24], U[25:28], U[28] = sg * f.D, sg * f.S, sg * f.tau
    return U


def _cfl(c, g, U):
    gam = torch.exp(4.0 * U[6]) * _sym(U[0:6])
    a, b = U[17], U[18:21]
    lam = torch.sqrt(_con("i,ij,j->", b, gam, b)) + torch.maximum(a, torch.sqrt(2.0 * a))

    def gaps(x):
        d = x.diff(dim=-1)
        return torch.minimum(torch.cat([d[..., :1], d], -1), torch.cat([d, d[..., -1:]], -1))

    r = g.r[:, :, None]
    h = torch.minimum(torch.minimum(gaps(g.r)[:, :, None], r * gaps(g.th)), r * torch.sin(g.th) * (2 * math.pi / g.npf))
    return float(c["cfl"] * h.min() / lam.max())


# ----------------------------------------------------------------------------------- the calls
def _structs(c):
    g, p, o = pkg.defaults()
    g.n_elem, g.n_r, g.n_theta, g.n_phi = c["n_elem"], c["n_r"], c["n_theta"], c["n_phi"]
    g.r_min, g.r_max, g.theta_basis = c["r_min"], c["r_max"], c["theta_basis"]
    g.theta_min, g.theta_max = (0.0, math.pi) if c["theta_basis"] else BAND
    p.a, p.gamma_eos = c["spin"], GAMMA
    o.precision, o.integrator, o.glm, o.contraction = c["precision"], c["integrator"], c["glm"], c["contraction"]
    o.cfl = c["cfl"]
    return g, p, o


def prepare(case, seed):
    states, dts = [], []
    for n, c in enumerate(_instances(case)):
        g = _grid(c)
        states.append(_state(c, g, 64 * seed + n))
        if case["do"] == "batch":
            dts.append(_cfl(c, g, states[-1]))
    if case["do"] == "batch":
        solver = pkg.Batch([_structs(c) for c in _instances(case)])
    else:
        solver = pkg.Context(*_structs(case))
    shape = (pkg.NPRIM,) + tuple(states[0].shape[1:]) if case["do"] == "c2p" else None
    outs = [torch.empty_like(U) if shape is None else U.new_empty(shape) for U in states]
    return SimpleNamespace(do=case["do"], steps=case["steps"], solver=solver, states=states, outs=outs, dts=dts)


def run(state):
    s = state.solver
    if state.do == "batch":
        for i, U in enumerate(state.states):
            s.set_state(i, U, True)
        s.step(state.dts, state.steps)
        for i, out in enumerate(state.outs):
            s.get_state(i, out, True)
        return state.outs
    out = state.outs[0]
    s.set_state(state.states[0], True)
    if state.do == "rhs":
        s.rhs(out, True)
        return out
    if state.do == "c2p":
        return {"prims": out, "failed": s.con2prim(out, True)}
    dt = s.step(0.0, state.steps)
    s.get_state(out, True)
    return {"state": out, "dt": dt}


# ------------------------------------------------------------------- the equations in 64 bits
def _fluid(rho, v, eps, B, gam):
    """Conserved variables and Eulerian stresses of the gas and field (undensitized)."""
    v_d, B_d = _con("ij,j->i", gam, v), _con("ij,j->i", gam, B)
    W = 1.0 / torch.sqrt(1.0 - _con("i,i->", v_d, v))
    B2, vB = _con("i,i->", B_d, B), _con("i,i->", v_d, B)
    p = (GAMMA - 1.0) * rho * eps
    f = SimpleNamespace(W=W, vB=vB, v_d=v_d)
    b2 = B2 / (W * W) + vB * vB
    f.Z = (rho * (1.0 + eps) + p + b2) * W * W
    f.ps = p + 0.5 * b2
    f.b_u, f.b_d = B / W + W * vB * v, B_d / W + W * vB * v_d
    f.D = rho * W
    f.S = f.Z * v_d - W * vB * f.b_d
    # tau without the cancellation against D: W - 1 = W^2 v^2 / (W + 1)
    w2v2 = W * W * _con("i,i->", v_d, v)
    f.tau = rho * W * (eps * W + w2v2 / (W + 1.0)) + p * w2v2 + b2 * (W * W - 0.5) - (W * vB) ** 2
    return f


def _primitives(U, gam, gi, sg):
    """rho, v^i, eps, W by bisection on mu = 1/(h W) (Kastaun, Kalinani & Ciolfi 2021); the
    atmosphere at rest where the density is at or below its floor."""
    D, S, tau, B = U[24] / sg, U[25:28] / sg, U[28] / sg, U[29:32] / sg
    B_d, SB = _con("ij,j->i", gam, B), _con("i,i->", S, B)
    q, r2 = tau / D, _con("i,ij,j->", S, gi, S) / D ** 2
    bb, rb2 = _con("i,i->", B_d, B) / D, SB ** 2 / D ** 3
    v2max = r2 / (1.0 + r2)

    def master(mu):
        x = 1.0 / (1.0 + mu * bb)
        rbar2 = r2 * x * x + mu * x * (1.0 + x) * rb2
        qbar = q - 0.5 * bb - 0.5 * (mu * x) ** 2 * (bb * r2 - rb2)
        v2 = torch.minimum(mu * mu * rbar2, v2max)
        W = (1.0 - v2) ** -0.5
        eps = W * (qbar - mu * rbar2) + v2 * W * W / (1.0 + W)
        e = torch.clamp(eps, min=EPS_ATM)
        a = (GAMMA - 1.0) * e / (1.0 + e)
        nu = torch.maximum((1.0 + e) * (1.0 + a) / W, (1.0 + a) * (1.0 + qbar - mu * rbar2))
        return mu - 1.0 / (nu + mu * rbar2), x, W, eps

    lo, hi = torch.zeros_like(D), torch.ones_like(D)
    for _ in range(60):
        mid = 0.5 * (lo + hi)
        neg = master(mid)[0] < 0.0
        lo, hi = torch.where(neg, mid, lo), torch.where(neg, hi, mid)
    mu = 0.5 * (lo + hi)
    _, x, W, eps = master(mu)
    v = _con("ij,j->i", gi, mu * x * (S / D + mu * SB / D ** 2 * B_d))
    gas = D > RHO_ATM
    return (torch.where(gas, D / W, RHO_ATM), torch.where(gas, v, 0.0),
            torch.where(gas, torch.clamp(eps, min=EPS_ATM), EPS_ATM), torch.where(gas, W, 1.0))


def _algebra(c, U, d1, d2, f, gam, gi, sg):
    """Everything at a point but the flux divergence: the right-hand side of the BSSN and gauge
    variables and the Valencia sources.  d1[direction, variable], d2[pair, variable]."""
    gt, At, phi, K = _sym(U[0:6]), _sym(U[7:13]), U[6], U[13]
    Gam, alpha, beta, Bg = U[14:17], U[17], U[18:21], U[21:24]
    gti, e4 = _inv(gt), torch.exp(4.0 * phi)

    def first(a, n=1):
        x = d1[:, a:a + n]
        return x[:, 0] if n == 1 else (torch.stack([_sym(y) for y in x]) if n == 6 else x)

    dgt, dAt, dphi, dK, dGam, dal, dbe = first(0, 6), first(7, 6), first(6), first(13), first(14, 3), first(17), first(18, 3)
    ddgt = torch.stack([torch.stack([d2[q, v] for v in range(6)]) for q in range(6)])      # [pair, component]
    ddphi, ddal = _sym(d2[:, 6]), _sym(d2[:, 7])
    ddbe = torch.stack([_sym(d2[:, 8 + i]) for i in range(3)])                             # [i, j, k]
    # Valencia sources
    dgam = e4 * (dgt + 4.0 * _con("k,ij->kij", dphi, gt))
    Kij = e4 * (At + gt * K / 3.0)
    S_uu = f.Z * _con("i,j->ij", f.v, f.v) + f.ps * gi - _con("i,j->ij", f.b_u, f.b_u)
    S_dd = f.Z * _con("i,j->ij", f.v_d, f.v_d) + f.ps * gam - _con("i,j->ij", f.b_d, f.b_d)
    rho_e, tr_S = f.tau + f.D, _con("ij,ij->", gam, S_uu)
    src_S = sg * (0.5 * alpha * _con("ij,kij->k", S_uu, dgam) + _con("i,ki->k", f.S, dbe) - rho_e * dal)
    src_tau = sg * (alpha * _con("ij,ij->", S_uu, Kij) - _con("i,ij,j->", f.S, gi, dal))
    # curvature
    Cl = 0.5 * (_con("ikj->kij", dgt) + _con("jki->kij", dgt) - dgt)
    Cu = _con("kl,lij->kij", gti, Cl)
    Gc = _con("jk,ijk->i", gti, Cu)
    lap = _sym([gti[0, 0] * ddgt[0, v] + gti[1, 1] * ddgt[3, v] + gti[2, 2] * ddgt[5, v]
                + 2.0 * (gti[0, 1] * ddgt[1, v] + gti[0, 2] * ddgt[2, v] + gti[1, 2] * ddgt[4, v]) for v in range(6)])
    up = _con("lm,jkm->jkl", gti, Cl)                                                      # Gamma_jk^l
    a1 = 0.5 * _con("ki,jk->ij", gt, dGam) + 0.5 * _con("k,ijk->ij", Gc, Cl) + _con("kli,jkl->ij", Cu, up)
    DDphi = ddphi - _con("kij,k->ij", Cu, dphi)
    gphi = _con("kl,l->k", gti, dphi)
    Ric = (-0.5 * lap + a1 + a1.transpose(0, 1) + _con("kim,kmj->ij", Cu, _con("lm,klj->kmj", gti, Cl))
           - 2.0 * DDphi - 2.0 * gt * _con("ij,ij->", gti, DDphi) + 4.0 * _con("i,j->ij", dphi, dphi)
           - 4.0 * gt * _con("i,i->", gphi, dphi))
    m = _con("i,j->ij", dphi, dal)
    DDal = ddal - _con("kij,k->ij", Cu, dal) - 2.0 * (m + m.transpose(0, 1) - gt * _con("i,i->", gphi, dal))
    tr_DDal = _con("ij,ij->", gti, DDal) / e4
    X = -DDal + alpha * (Ric - 8.0 * math.pi * S_dd)
    XTF = X - gt * _con("ij,ij->", gti, X) / 3.0
    Aud = _con("kl,lj->kj", gti, At)
    Auu = _con("ik,kj->ij", Aud, gti)
    divb = dbe[0, 0] + dbe[1, 1] + dbe[2, 2]
    lg, la = _con("ik,jk->ij", gt, dbe), _con("ik,jk->ij", At, dbe)
    o_gt = -2.0 * alpha * At + _con("k,kij->ij", beta, dgt) + lg + lg.transpose(0, 1) - 2.0 / 3.0 * gt * divb
    o_At = (XTF / e4 + alpha * (K * At - 2.0 * _con("ik,kj->ij", At, Aud)) + _con("k,kij->ij", beta, dAt)
            + la + la.transpose(0, 1) - 2.0 / 3.0 * At * divb)
    o_phi = -alpha * K / 6.0 + _con("k,k->", beta, dphi) + divb / 6.0
    o_K = (-tr_DDal + alpha * (_con("ij,ij->", At, Auu) + K * K / 3.0) + 4.0 * math.pi * alpha * (rho_e + tr_S)
           + _con("k,k->", beta, dK))
    ddb_tr = torch.stack([ddbe[0, j, 0] + ddbe[1, j, 1] + ddbe[2, j, 2] for j in range(3)])
    o_Gam = (_con("jk,ijk->i", gti, ddbe) + _con("ij,j->i", gti, ddb_tr) / 3.0 + _con("j,ji->i", beta, dGam)
             - _con("j,ji->i", Gam, dbe) + 2.0 / 3.0 * Gam * divb - 2.0 * _con("ij,j->i", Auu, dal)
             + 2.0 * alpha * (_con("ijk,jk->i", Cu, Auu) + 6.0 * _con("ij,j->i", Auu, dphi)
                              - 2.0 / 3.0 * _con("ij,j->i", gti, dK))
             - 16.0 * math.pi * alpha * _con("ij,j->i", gti, f.S))
    o_al = -2.0 * alpha * K + _con("i,i->", beta, dal)
    out = _six(o_gt) + [o_phi] + _six(o_At) + [o_K] + list(o_Gam) + [o_al] + list(0.75 * Bg) + list(o_Gam - 2.0 * Bg)
    zero = torch.zeros_like(K)
    out += [zero] + list(src_S) + [src_tau, zero, zero, zero]
    if c["glm"]:
        dpsi = d1[:, 21]
        for k, x in enumerate(_con("ij,j->i", gi, dpsi)):
            out[29 + k] = -alpha * sg * x
        out.append(-alpha * U[32])
    return torch.stack(out)


def _rhs(c, g, U):
    P, shape = U[0].numel(), U.shape[1:]
    flat = U.reshape(len(U), P)
    idx1 = list(range(21)) + ([32] if c["glm"] else [])
    par = _par(g, idx1)
    u = U[idx1]
    d1 = torch.stack([_mean_ends(g, _d_r(g, u)), _d_t(g, u, par), _d_p(g, u)])
    s, par2 = d1[:, _SECOND], _par(g, _SECOND)
    d2 = torch.stack([_mean_ends(g, _d_r(g, s[0])), _d_t(g, s[0], par2), _d_p(g, s[0]), _d_t(g, s[1], -par2),
                      _d_p(g, s[1]), _d_p(g, s[2])])
    d1, d2 = d1.reshape(3, len(idx1), P), d2.reshape(6, 11, P)
    out, F, lam = torch.empty_like(flat), U.new_empty((3, 8, P)), U.new_empty((P,))
    for a in range(0, P, 1 << 18):
        at = slice(a, min(P, a + (1 << 18)))
        x = flat[:, at]
        gam = torch.exp(4.0 * x[6]) * _sym(x[0:6])
        gi, sg = _inv(gam), torch.sqrt(_det(gam))
        rho, v, eps, _ = _primitives(x, gam, gi, sg)
        B, al = x[29:32] / sg, x[17]
        f = _fluid(rho, v, eps, B, gam)
        f.v = v
        vt = al * v - x[18:21]
        F[:, 0, at] = sg * f.D * vt
        for i in range(3):
            for j in range(3):
                F[i, 1 + j, at] = sg * (f.S[j] * vt[i] - al * f.b_d[j] * B[i] / f.W + (al * f.ps if i == j else 0.0))
            F[i, 4, at] = sg * (f.tau * vt[i] + al * f.ps * v[i] - al * f.vB * B[i])
            for k in range(3):
                F[i, 5 + k, at] = sg * (vt[i] * B[k] - vt[k] * B[i])
        lam[at] = torch.abs(x[18]) + al * torch.sqrt(gi[0, 0])
        out[:, at] = _algebra(c, x, d1[:, :, at], d2[:, :, at], f, gam, gi, sg)
    out, F, lam = out.reshape(U.shape), F.reshape((3, 8) + shape), lam.reshape(shape)
    val = _par(g, range(24, 32))
    out[24:32] -= _d_r(g, F[0]) + _d_t(g, F[1], -val) + _d_p(g, F[2])
    if c["glm"]:
        div = _d_r(g, U[29:30]) + _d_t(g, U[30:31], _par(g, [30])) + _d_p(g, U[31:32])
        sg = torch.exp(6.0 * U[6]) * torch.sqrt(_det(_sym(U[0:6])))
        out[32] -= U[17] * _mean_ends(g, div)[0] / sg
    if g.E > 1:  # Rusanov flux at the element interfaces
        l, r = (slice(None), slice(0, -1), -1), (slice(None), slice(1, None), 0)
        top = torch.maximum(lam[l[1:]], lam[r[1:]])
        V = U[24:32]
        star = 0.5 * (F[0][l] + F[0][r]) - 0.5 * top * (V[r] - V[l])
        fac = (g.scale / g.w_end)[:, None, None]
        out[24:32, :-1, -1] += (F[0][l] - star) * fac[:-1]
        out[24:32, 1:, 0] -= (F[0][r] - star) * fac[1:]
    out[:, -1, -1] = 0.0
    return out


def _filter(g, U):
    def along(m, spec, u):
        return torch.einsum(spec, m, u)

    U = along(g.Fr, "ij,vejtp->veitp", U)
    val = list(range(24, len(U)))
    U[24:] = _along_theta(g, g.Ft, U[24:], _par(g, val))
    U = along(g.Fp, "ij,vertj->verti", U)
    U[:24] = _mean_ends(g, U[:24])
    if len(U) > 32:
        U[32] = _mean_ends(g, U[32])
    return U


def _advance(c, g, U, dt, steps):
    for _ in range(steps):
        if c["integrator"]:
            k1 = _rhs(c, g, U)
            k2 = _rhs(c, g, U + 0.5 * dt * k1)
            k3 = _rhs(c, g, U + 0.5 * dt * k2)
            k4 = _rhs(c, g, U + dt * k3)
            V = U + dt / 6.0 * (k1 + 2.0 * k2 + 2.0 * k3 + k4)
        else:
            V = U + dt * _rhs(c, g, U)
            V = 0.75 * U + 0.25 * (V + dt * _rhs(c, g, V))
            V = U / 3.0 + 2.0 / 3.0 * (V + dt * _rhs(c, g, V))
        U = _filter(g, V)
    return U


def exact(case, seed):
    outs = []
    for n, c in enumerate(_instances(case)):
        g = _grid(c)
        U = _state(c, g, 64 * seed + n)
        if case["do"] == "rhs":
            return _rhs(c, g, U)
        if case["do"] == "c2p":
            gam = torch.exp(4.0 * U[6]) * _sym(U[0:6])
            rho, v, eps, W = _primitives(U, gam, _inv(gam), torch.sqrt(_det(gam)))
            return {"prims": torch.stack([rho, *v, eps, (GAMMA - 1.0) * rho * eps, W]), "failed": 0}
        dt = _cfl(c, g, U)
        U = _advance(c, g, U, dt, case["steps"])
        if case["do"] == "step":
            return {"state": U, "dt": dt}
        outs.append(U)
    return outs
