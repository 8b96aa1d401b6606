"""The work that a user of this library has it do, as cases that can be timed.

Every case goes through the public binding (paper_0710_0066_gb300.lqcd): whole
trajectories, the solves and forces they consist of, and the operator and
gauge-field calls that measurements and tests make.  Gauge fields are SU(3)
fields thermalised by a pure-gauge heatbath (below) at the coupling whose
plaquette is that of the beta = 5.6 two-flavour ensembles (about 0.57);
sources are Gaussian.  Trajectories keep the evolved field whatever dH (as
thermalisation does), so that it is always the output.  Solves run to a relative residual of 1e-12, the one
that forces and reversible trajectories are run to.
"""
import math

import torch

from paper_0710_0066_gb300 import lqcd

KINDS = ("traj", "traj4", "solve", "blocks", "series", "hop", "force", "gauge")
PREC = {"f64": lqcd.PREC_F64, "f32": lqcd.PREC_F32, "f16": lqcd.PREC_F16, "bf16": lqcd.PREC_BF16}
LINK_BYTES = {"f64": 144, "f32": 48, "f16": 24, "bf16": 24}  # one link in the storage of the inner arithmetic
BETA, BETA_HEATBATH, LAMBDA, TOL = 5.6, 5.8, 0.1931833275037836, 1e-12
DEVICE = "cuda"
KRYLOV = 100  # iterations a solve is counted with in work()


def _case(kind, L, l0, prec="f32", kappa=0.1575, **more):
    return dict(kind=kind, L0=L[0], L1=L[1], L2=L[2], L3=L[3], l0=l0, prec=prec, kappa=kappa, **more)


def listed():
    return [
        # a short trajectory of the two-part action on a test-sized lattice:
        # launches, barriers and host round trips are what it costs
        dict(_case("traj", (8, 4, 4, 4), 2, kappa=0.14, tau=0.4, n0=2, n1=2, n2=2), name="traj 8x4^3"),
        # the production call: the first quarter of the benchmark's trajectory
        # (the same steps, a quarter of the length)
        dict(_case("traj", (32, 16, 16, 16), 4, tau=0.25, n0=2, n1=4, n2=2), name="traj 32x16^3"),
        # the paper's four-part action on five time scales (sub-slabs, mass
        # preconditioning, x0-dependent steps) on a medium lattice
        dict(_case("traj4", (16, 8, 8, 8), 8, kappa=0.15, rho=0.2, tau=0.5, n4=2), name="traj four-part 16x8^3"),
        # whole-lattice solves (propagators, the boundary term's force): a
        # small ragged lattice, the ordinary size, the largest
        dict(_case("solve", (12, 6, 6, 6), 3, kappa=0.15, dagger=0), name="solve 12x6^3"),
        dict(_case("solve", (32, 16, 16, 16), 4, dagger=0), name="solve 32x16^3"),
        dict(_case("solve", (64, 32, 32, 32), 8, dagger=1), name="solve 64x32^3"),
        # the same-launch solves of all slabs (W1 of the two-part action)
        dict(_case("blocks", (32, 16, 16, 16), 4, colour=-1, dagger=0), name="blocks 32x16^3"),
        # the geometric series of the mass-preconditioned sub-slab systems,
        # the lattice of the paper's timing remark
        dict(_case("series", (32, 24, 24, 24), 16, rho=0.15, dagger=0), name="series 32x24^3"),
        # one even-odd hopping sweep, single and half storage
        dict(_case("hop", (64, 32, 32, 32), 8, prec="f32", parity=0, dagger=0), name="hop f32 64x32^3"),
        dict(_case("hop", (32, 24, 24, 24), 16, prec="f16", parity=1, dagger=0), name="hop f16 32x24^3"),
        # pseudo-fermion action and force of the slab term in double precision
        dict(_case("force", (16, 8, 8, 8), 4, prec="f64", kappa=0.15), name="force f64 16x8^3"),
        # gauge force, action and plaquette (every measurement, every check)
        dict(_case("gauge", (32, 16, 16, 16), 4, prec="f64"), name="gauge 32x16^3"),
    ]


def _extent(rng, lo, hi, step=2):
    """an extent between lo and hi, even over the logarithm"""
    return max(lo, min(hi, step * round(math.exp(rng.uniform(math.log(lo), math.log(hi))) / step)))


def draw(rng):
    kind = rng.choice(KINDS)
    if kind == "traj":
        l0 = rng.choice((2, 4))
        L = (2 * l0 * rng.choice((1, 2, 3)),) + tuple(_extent(rng, 4, 12) for _ in range(3))
        return _case(kind, L, l0, kappa=0.14, tau=rng.choice((0.2, 0.4)), n0=2, n1=2, n2=rng.choice((2, 3, 4)))
    if kind == "traj4":
        L = (16,) + tuple(_extent(rng, 4, 10) for _ in range(3))
        return _case(kind, L, 8, kappa=0.14, rho=rng.choice((0.15, 0.2)), tau=0.25, n4=1)
    big = kind == "hop" or rng.random() < 0.3
    l0 = rng.choice((1, 2, 3, 4, 6, 8)) if kind in ("solve", "blocks", "hop") else rng.choice((2, 4, 6, 8))
    hi = 32 if big else 16
    L = (2 * l0 * rng.randint(1, 2 * hi // (2 * l0)),) + tuple(_extent(rng, 4, hi) for _ in range(3))
    volume = L[0] * L[1] * L[2] * L[3]
    kappa = 0.1575 if min(L[1:]) >= 12 else 0.15 if min(L[1:]) >= 8 else 0.14
    dagger = rng.randint(0, 1)
    if kind == "hop":
        return _case(kind, L, l0, prec=rng.choice(("f64", "f32", "f16", "bf16")), parity=rng.randint(0, 1), dagger=dagger)
    if kind == "solve":
        return _case(kind, L, l0, prec="f64" if volume < 30000 and rng.random() < 0.3 else "f32", kappa=kappa, dagger=dagger)
    if kind == "blocks":
        return _case(kind, L, l0, kappa=kappa, colour=rng.choice((-1, 0, 1)), dagger=dagger)
    if kind == "series":
        return _case(kind, L, l0, kappa=kappa, rho=rng.choice((0.15, 0.2)), dagger=dagger)
    if kind == "force":
        return _case(kind, L, l0, prec="f64", kappa=0.14) if volume < 70000 else _case("gauge", L, l0, prec="f64")
    return _case(kind, L, l0, prec="f64")


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _extents(case):
    return tuple(case["L%d" % mu] for mu in range(4))


def _subslabs(case):
    return case["l0"] // 2 if case["kind"] in ("traj4", "series") else 0


def _site_tables(L, device):
    """sites in the library's (checkerboard) order: coordinates (4, V) and,
    per direction, the sites x + mu and x - mu"""
    x = torch.stack(torch.meshgrid(*[torch.arange(n, device=device) for n in L], indexing="ij")).reshape(4, -1)
    order = torch.argsort(x.sum(0) % 2, stable=True)
    place = torch.empty_like(order)
    place[order] = torch.arange(order.numel(), device=device)
    x = x[:, order]
    near = []
    for step in (1, -1):
        for mu in range(4):
            y = x.clone()
            y[mu] = (y[mu] + step) % L[mu]
            near.append(place[((y[0] * L[1] + y[1]) * L[2] + y[2]) * L[3] + y[3]])
    return x, near[:4], near[4:]


def _mul(a, b):
    return a[..., :, 0:1] * b[..., 0:1, :] + a[..., :, 1:2] * b[..., 1:2, :] + a[..., :, 2:3] * b[..., 2:3, :]


def _dag(a):
    return a.mH


def _su3(a):
    """the rows of a made orthonormal, determinant one"""
    r0 = a[..., 0, :] / torch.linalg.vector_norm(a[..., 0, :], dim=-1, keepdim=True)
    r1 = a[..., 1, :] - (r0.conj() * a[..., 1, :]).sum(-1, keepdim=True) * r0
    r1 = r1 / torch.linalg.vector_norm(r1, dim=-1, keepdim=True)
    return torch.stack((r0, r1, torch.linalg.cross(r0, r1).conj()), -2)


def _su2_heatbath(U, W, i, j, gen):
    """one SU(2) subgroup of the links: a drawn from exp(2 beta k a0 / 3) (Kennedy and
    Pendleton), k and v the length and direction of the 2x2 block of W = U staple"""
    v = torch.stack((W[:, i, i].real + W[:, j, j].real, W[:, i, j].imag + W[:, j, i].imag,
                     W[:, i, j].real - W[:, j, i].real, W[:, i, i].imag - W[:, j, j].imag)) * 0.5
    k = torch.linalg.vector_norm(v, dim=0).clamp_min(1e-10)
    v = v / k
    alpha = 2.0 * BETA_HEATBATH / 3.0 * k
    a0 = torch.ones_like(k)
    todo = torch.ones_like(k, dtype=torch.bool)
    for _ in range(4):  # what is left then (well under a percent) keeps its old direction
        r = 1.0 - torch.rand((4,) + k.shape, generator=gen, device=k.device)
        d = -(r[0].log() + torch.cos(2 * math.pi * r[1]).square() * r[2].log()) / alpha
        ok = todo & (r[3].square() <= 1.0 - 0.5 * d)
        a0 = torch.where(ok, 1.0 - d, a0)
        todo = todo & ~ok
    n = torch.randn((3,) + k.shape, generator=gen, device=k.device)
    n = n * ((1.0 - a0.square()).clamp_min(0.0).sqrt() / torch.linalg.vector_norm(n, dim=0).clamp_min(1e-10))
    # a v^dagger as a quaternion
    b0 = torch.where(todo, torch.ones_like(a0), a0 * v[0] + (n * v[1:]).sum(0))
    b = torch.where(todo, torch.zeros_like(n), n * v[0] - a0 * v[1:] + torch.linalg.cross(n, v[1:], dim=0))
    g00, g01 = torch.complex(b0, b[2])[:, None], torch.complex(b[1], b[0])[:, None]
    for m in (U, W):
        p, q = m[:, i].clone(), m[:, j].clone()
        m[:, i] = g00 * p + g01 * q
        m[:, j] = -g01.conj() * p + g00.conj() * q


def gauge_field(L, seed, sweeps=12):
    """a seeded SU(3) field (4, V, 3, 3): disordered start a little below the right plaquette, then heatbath
    sweeps; a lattice of more than 2^17 sites repeats a smaller one periodically"""
    cell = list(L)
    while math.prod(cell) > 1 << 17 and any(n % 4 == 0 and n >= 16 for n in cell):
        cell[cell.index(max(n for n in cell if n % 4 == 0 and n >= 16))] //= 2
    if tuple(cell) != tuple(L):
        part = gauge_field(tuple(cell), seed, sweeps)
        x, _, _ = _site_tables(L, DEVICE)
        y = [x[mu] % cell[mu] for mu in range(4)]
        at = ((y[0] * cell[1] + y[1]) * cell[2] + y[2]) * cell[3] + y[3]
        return part[:, sum(y) % 2 * (math.prod(cell) // 2) + at // 2].contiguous()
    gen = torch.Generator(device=DEVICE)
    gen.manual_seed(int(seed))
    V = math.prod(L)
    _, up, down = _site_tables(L, DEVICE)
    U = torch.randn((4, V, 3, 3), dtype=torch.complex64, device=DEVICE, generator=gen)
    U = _su3(0.45 * U + torch.eye(3, device=DEVICE))
    half = [torch.arange(0, V // 2, device=DEVICE), torch.arange(V // 2, V, device=DEVICE)]
    for _ in range(sweeps):
        for mu in range(4):
            for at in half:
                A = 0
                for nu in range(4):
                    if nu != mu:
                        back = down[nu][at]
                        A = A + _mul(U[nu][up[mu][at]], _dag(_mul(U[nu][at], U[mu][up[nu][at]])))
                        A = A + _mul(_dag(_mul(U[mu][back], U[nu][up[mu][back]])), U[nu][back])
                link = U[mu][at]
                W = _mul(link, A)
                for i, j in ((0, 1), (0, 2), (1, 2)):
                    _su2_heatbath(link, W, i, j, gen)
                U[mu][at] = link
        U = _su3(U)
    return _su3(U.to(torch.complex128)).contiguous()


def _source(shape, seed):
    gen = torch.Generator(device=DEVICE)
    gen.manual_seed(int(seed) + 1)
    return torch.randn(shape, dtype=torch.complex128, device=DEVICE, generator=gen)


def _inputs(case, seed):
    """the gauge field and (where the case has one) the source"""
    V = math.prod(_extents(case))
    shape = {"solve": (V, 4, 3), "blocks": (V, 4, 3), "force": (V, 4, 3), "series": (V // 2, 4, 3),
             "hop": (V // 2, 4, 3)}.get(case["kind"])
    # (nothing in one sweep over the links depends on how well they are thermalised)
    U = gauge_field(_extents(case), seed, 2 if case["kind"] in ("hop", "gauge") else 12)
    return U, _source(shape, seed) if shape else None


def prepare(case, seed):
    U, b = _inputs(case, seed)
    lat = lqcd.Lattice(_extents(case), case["l0"], -1, l0s=_subslabs(case))
    lat.set_gauge(U)
    state = dict(case=case, lat=lat, U=U, b=b, seed=int(seed))
    if case["kind"] == "traj":
        # gauge / W1 / boundary term on three Omelyan levels, the molecular
        # dynamics as one graph, chronological guesses, series for W1
        state["prm"] = lqcd.hmc_params(
            BETA, case["kappa"], case["tau"], 3, (lqcd.SW, lqcd.SW, lqcd.SW if case["n1"] % 2 == 0 else lqcd.LF),
            (case["n0"], case["n1"], case["n2"]), 0, 1, 2, lam=LAMBDA, roll=1, metropolis=0,
            precision=PREC[case["prec"]], tol=TOL, block_solver=lqcd.SOLVER_SERIES, use_graph=1, chrono=2)
    elif case["kind"] == "traj4":
        # the paper's schedule: S_G, S1, S2, S3 (R2), S4 (R), scheme B
        state["prm"] = lqcd.hmc_params(
            BETA, case["kappa"], case["tau"], 5, (lqcd.SW, lqcd.SW, lqcd.LF, lqcd.LF, lqcd.LF), (4, 2, 3, 1, case["n4"]),
            0, -1, 4, lam=1.0 / 6.0, roll=1, metropolis=0, precision=PREC[case["prec"]], tol=TOL, step_scheme=2,
            level_schur2=3, rho=case["rho"], level_s2=2, level_s1=1, use_graph=1, chrono=2)
    return state


def run(state):
    case, lat, b = state["case"], state["lat"], state["b"]
    kind, prec = case["kind"], PREC[case["prec"]]
    if kind in ("traj", "traj4"):
        U, res = lat.hmc_trajectory(state["U"], state["prm"], state["seed"], 0)
        return dict(U=U, H0=res.H0, H1=res.H1, plaq=res.plaq, accepted=res.accepted, shift=res.shift,
                    n_solves=res.n_solves, n_force=res.n_force)
    if kind == "solve":
        return lat.solve(b, case["kappa"], case["dagger"], prec, TOL)[0]
    if kind == "blocks":
        return lat.block_solve(b, case["kappa"], case["colour"], case["dagger"], prec, TOL)[0]
    if kind == "series":
        return lat.solve_w3eo(b, case["kappa"], case["rho"], case["dagger"], prec, TOL, method=lqcd.SOLVER_SERIES)[0]
    if kind == "hop":
        return lat.dslash_eo(b, case["parity"], 0.0, case["dagger"], lqcd.OP_HOP, prec)
    if kind == "force":
        S, F = lat.pf_force(b, case["kappa"], lqcd.TERM_W1, prec, TOL)
        return dict(S=S, F=F)
    S, plaq, F = lat.gauge_force(BETA)
    return dict(S=S, plaq=plaq, F=F)


def work(case):
    """each field once, in the storage it has to be read or written in; a solve
    as KRYLOV iterations of two even-odd operators (four half-lattice hopping
    sweeps; the series one operator), a trajectory as its force solves"""
    V, kind, link = math.prod(_extents(case)), case["kind"], LINK_BYTES[case["prec"]]
    sweep = 1320.0 * V / 2
    if kind == "hop":
        return dict(bytes=V * 192 + 4 * V * link, flops=sweep)
    if kind == "solve" or kind == "blocks":
        part = 0.5 if case.get("colour", -1) >= 0 else 1.0
        return dict(bytes=part * (2 * V * 192 + 4 * V * link), flops=part * 4 * sweep * KRYLOV)
    if kind == "series":
        return dict(bytes=V * 192 + 4 * V * link, flops=2 * sweep * KRYLOV)
    if kind == "force":
        return dict(bytes=V * 192 + 4 * V * 144 + 4 * V * 64, flops=2 * 4 * sweep * KRYLOV)
    if kind == "gauge":
        return dict(bytes=4 * V * 144 + 4 * V * 64, flops=4 * V * 13 * 198.0)
    if kind == "traj":
        solves = 2 * (2 * case["n2"] + 1) * (1 + 2 * case["n1"])
    else:
        solves = 2 * (case["n4"] + 1) * (1 + 1 + 3 + 3 * 4)
    return dict(bytes=2 * 4 * V * 144, flops=solves * 2 * sweep * KRYLOV)


# ---------------------------------------------------------------------------
# the same in 64 bits, from the definitions
# ---------------------------------------------------------------------------
class _Wilson:
    """H of M = 1 - kappa H in complex128, hops between blocks of `block` time slices left out (0: none)"""

    def __init__(self, L, U, block):
        x, self.up, self.down = _site_tables(L, U.device)
        self.U, self.V = U, x.shape[1]
        one = torch.ones(self.V, dtype=torch.float64, device=U.device)
        t = torch.where(x[0] == L[0] - 1, -one, one)  # antiperiodic in x0
        if block:
            t = torch.where((x[0] + 1) % block == 0, torch.zeros_like(t), t)
        self.weight = [t, one, one, one]

    # row s of gamma_mu has the entry GAMMA[mu][1][s] in column GAMMA[mu][0][s]
    GAMMA = (((2, 3, 0, 1), (-1, -1, -1, -1)), ((3, 2, 1, 0), (-1j, -1j, 1j, 1j)),
             ((3, 2, 1, 0), (-1, 1, 1, -1)), ((2, 3, 0, 1), (-1j, 1j, 1j, -1j)))

    def spin(self, mu, sign, p):
        """(1 + sign gamma_mu) p"""
        column, entry = self.GAMMA[mu]
        return torch.stack([p[:, s] + (sign * entry[s]) * p[:, column[s]] for s in range(4)], 1)

    def hop(self, p, dagger=0):
        sign = 1 if dagger else -1
        out = torch.zeros_like(p)
        for mu in range(4):
            w, at, back = self.weight[mu][:, None, None], self.up[mu], self.down[mu]
            out += w * _mul(self.spin(mu, sign, p[at]), self.U[mu].transpose(-1, -2))
            out += w[back] * _mul(self.spin(mu, -sign, p[back]), self.U[mu][back].conj())
        return out

    def reduced(self, p_e, kappa, diag, dagger):
        """diag p_e - kappa^2 H_eo H_oe p_e on the even sites"""
        h = self.V // 2
        q = torch.cat((p_e, torch.zeros_like(p_e)))
        q = self.hop(q, dagger)
        q[:h] = 0
        return diag * p_e - kappa * kappa * self.hop(q, dagger)[:h]


def _bicgstab(A, b, tol=2e-15, most=4000):
    """A x = b in complex128, restarted from the true residual"""
    x, size, dot = torch.zeros_like(b), torch.linalg.vector_norm(b), lambda u, v: torch.vdot(u.reshape(-1), v.reshape(-1))
    steps, last = 0, math.inf
    while steps < most:
        r = b - A(x)
        now = float(torch.linalg.vector_norm(r) / size)
        if now < tol or now > 0.3 * last:
            return x
        last, goal = now, max(1e-5 * now, 0.3 * tol)
        rh, p, rho = r.clone(), r.clone(), dot(r, r)
        while steps < most:
            v = A(p)
            alpha = rho / dot(rh, v)
            s = r - alpha * v
            t = A(s)
            omega = dot(t, s) / dot(t, t)
            x = x + alpha * p + omega * s
            r = s - omega * t
            steps += 1
            if float(torch.linalg.vector_norm(r) / size) < goal:
                break
            new = dot(rh, r)
            p = r + (new / rho) * (alpha / omega) * (p - omega * v)
            rho = new
    return x


def _lie(Y):
    """2 Im tr(T^a Y), T^a half the Gell-Mann matrices"""
    return torch.stack((Y[..., 1, 0].imag + Y[..., 0, 1].imag, Y[..., 0, 1].real - Y[..., 1, 0].real,
                        Y[..., 0, 0].imag - Y[..., 1, 1].imag, Y[..., 2, 0].imag + Y[..., 0, 2].imag,
                        Y[..., 0, 2].real - Y[..., 2, 0].real, Y[..., 2, 1].imag + Y[..., 1, 2].imag,
                        Y[..., 1, 2].real - Y[..., 2, 1].real,
                        (Y[..., 0, 0].imag + Y[..., 1, 1].imag - 2 * Y[..., 2, 2].imag) / math.sqrt(3.0)), -1)


def exact(case, seed):
    kind, L, kappa = case["kind"], _extents(case), case["kappa"]
    if kind in ("traj", "traj4"):
        return None  # thousands of solves in 64 bits
    if kind == "gauge":
        U, _ = _inputs(case, seed)
        _, up, down = _site_tables(L, DEVICE)
        total, F = 0.0, []
        for mu in range(4):
            A = 0
            for nu in range(4):
                if nu != mu:
                    loop = _mul(U[nu][up[mu]], _dag(_mul(U[nu], U[mu][up[nu]])))
                    if nu < mu:
                        total += float((U[mu] * loop.transpose(-1, -2)).sum().real)
                    back = down[nu]
                    A = A + loop + _mul(_dag(_mul(U[mu][back], U[nu][up[mu][back]])), U[nu][back])
            F.append(BETA / 6.0 * _lie(_mul(U[mu], A)))
        return dict(S=-BETA / 3.0 * total, plaq=total / (18.0 * math.prod(L)), F=torch.stack(F))
    U, b = _inputs(case, seed)
    if kind == "hop":
        h, par = b.shape[0], case["parity"]
        p = torch.zeros((2 * h, 4, 3), dtype=torch.complex128, device=b.device)
        p[(1 - par) * h:(2 - par) * h] = b
        return _Wilson(L, U, 0).hop(p, case["dagger"])[par * h:(par + 1) * h]
    if kind == "series":
        D = _Wilson(L, U, _subslabs(case))
        return _bicgstab(lambda p: D.reduced(p, kappa, 1.0 + case["rho"], case["dagger"]), b)
    D = _Wilson(L, U, 0 if kind == "solve" else case["l0"])
    if kind == "blocks" and case["colour"] >= 0:
        x, _, _ = _site_tables(L, b.device)
        b = b * ((x[0] // case["l0"]) % 2 == case["colour"]).to(b.dtype)[:, None, None]
    if kind in ("solve", "blocks"):
        return _bicgstab(lambda p: p - kappa * D.hop(p, case["dagger"]), b)
    # force: eta = W1^-1 phi, xi = W1^-dag eta, dS = 2 kappa Re <xi, dH eta>
    eta = _bicgstab(lambda p: p - kappa * D.hop(p), b)
    xi = _bicgstab(lambda p: p - kappa * D.hop(p, 1), eta)
    F = []
    for mu in range(4):
        at, w = D.up[mu], D.weight[mu][:, None]
        X = torch.matmul(D.spin(mu, -1, eta[at]).transpose(-1, -2), xi.conj())
        Z = torch.matmul(eta.transpose(-1, -2), D.spin(mu, 1, xi[at]).conj())
        F.append(-kappa * w * _lie(_mul(U[mu], X) - _mul(Z, _dag(U[mu]))))
    return dict(S=float(torch.linalg.vector_norm(eta).square()), F=torch.stack(F))
