"""The measured cases: what a user of the Helmholtz solver has it do.

A case names an entry point (``call``), a grid, a strip decomposition, a medium, a
precision and a number of right-hand sides.  Calls:

* ``solve``      ``HelmDD.solve`` on a factored handle (the framework's main path:
                 FP64 FGMRES around the double sweep);
* ``reduced``    ``HelmDD.solve_reduced`` on a factored handle (Algorithm 5 on the
                 interface lines, the route with the small Krylov basis);
* ``newmodel``   a medium the program has not seen: create, factor, solve, close
                 (one step of a frequency sweep or of a model update);
* ``misfit``     ``helm.misfit`` and its backward pass: factor, forward solves, then
                 forward and adjoint solves, as one step of an inversion;
* ``precond``    ``HelmDD.apply_precond``, the double sweep inside a caller's own
                 Krylov method;
* ``matvec``     ``HelmDD.matvec``, the FP64 operator.

Solves run to a relative residual of 1e-8, as fields do that feed data misfits and
gradients (the paper's stopping rule is 1e-6).  Media and sources come from the seed.
"""
import math

import numpy as np
import torch

from paper_1208_3956_gb300 import helm, media

DEV = "cuda"


def _case(name, call, n, J, w_outer, w_sub, precision, nrhs, medium="smooth", tol=1e-8):
    n = tuple(n) + (1,) * (3 - len(n))
    c = {"call": call, "nx": n[0], "ny": n[1], "nz": n[2], "J": J, "w_outer": w_outer, "w_sub": w_sub,
         "precision": precision, "nrhs": nrhs, "medium": medium, "tol": tol}
    if name:
        c = {"name": name, **c}
    return c


def listed():
    return [
        # the smallest solve of the repository's workloads: launches, latency and host work
        _case("small2d", "solve", (127, 127), 8, 10, 8, "mixed", 1),
        # the headline workload's grid: one shot, one field
        _case("point2d", "solve", (1023, 1023), 64, 16, 12, "mixed", 1),
        # complex128 factors and sweeps, for users who want no complex64 anywhere
        _case("point2d_fp64", "solve", (511, 511), 32, 16, 12, "fp64", 1),
        # a shot gather: 32 sources on the top row in one panel
        _case("shots2d", "solve", (1023, 1023), 64, 16, 12, "mixed", 32),
        # a layered medium in the interface-reduced space, ragged grid
        _case("layered2d_reduced", "reduced", (1021, 765), 64, 20, 16, "mixed", 4, "layered", 1e-9),
        # one inversion step on a ragged grid: misfit and gradient, 8 shots
        _case("misfit2d", "misfit", (383, 255), 24, 16, 12, "mixed", 8),
        # a new 2-D medium and one shot: the factorisation is most of it
        _case("newmodel2d", "newmodel", (511, 511), 32, 16, 12, "mixed", 1),
        # the 3-D workload's grid: dense slab blocks streamed from memory
        _case("point3d", "solve", (63, 63, 63), 8, 8, 6, "mixed", 1),
        # 16 sources on a 3-D grid in one call
        _case("shots3d", "solve", (47, 47, 47), 6, 8, 6, "mixed", 16),
        # a new 3-D medium and one shot, ragged sides: block inversions on the tensor cores
        _case("newmodel3d", "newmodel", (33, 37, 29), 4, 6, 5, "mixed", 1),
        # the double sweep alone in complex128, two fields, inside a caller's own Krylov method
        _case("precond2d_fp64", "precond", (447, 383), 28, 16, 12, "fp64", 2),
        # the FP64 operator on fields larger than the cache
        _case("matvec2d", "matvec", (2047, 1535), 128, 16, 12, "mixed", 4),
    ]


def _log(rng, lo, hi):
    return lo * (hi / lo) ** rng.random()


def draw(rng):
    """One more case of the listed ranges; none costs more than the largest listed one."""
    call, precision, dim = rng.choice([("solve", "mixed", 2), ("solve", "mixed", 2), ("solve", "fp64", 2),
                                       ("reduced", "mixed", 2), ("newmodel", "mixed", 2), ("misfit", "mixed", 2),
                                       ("solve", "mixed", 3), ("newmodel", "mixed", 3), ("precond", "fp64", 2),
                                       ("matvec", "mixed", 2)])
    medium = "smooth"
    tol = 1e-8
    if dim == 3:
        nx, ny, nz = (int(round(_log(rng, 19, 56 if call == "solve" else 40))) for _ in range(3))
        J = max(2, nx // 8)
        nrhs = int(round(_log(rng, 1, 16))) if call == "solve" else 1
        return _case(None, call, (nx, ny, nz), J, rng.randint(5, 8), rng.randint(4, 6), precision, nrhs, medium, tol)
    top = {"solve": 1023 if precision == "mixed" else 511, "newmodel": 700, "misfit": 400, "reduced": 900,
           "precond": 511, "matvec": 2047}[call]
    nx, ny = (int(round(_log(rng, 127, top))) for _ in range(2))
    J = max(2, nx // rng.randint(14, 17))
    w_outer, w_sub = rng.randint(10, 18), rng.randint(8, 14)
    if precision == "fp64":   # complex128 strips hold about 50 columns
        w_outer, w_sub = min(w_outer, 16), min(w_sub, 12)
    nrhs = 1
    if call in ("solve", "reduced", "misfit", "precond", "matvec"):
        most = {"solve": 32 if precision == "mixed" else 4, "reduced": 6, "misfit": 12, "precond": 8, "matvec": 4}[call]
        nrhs = int(round(_log(rng, 1, most)))
    if call == "reduced":
        medium, tol = rng.choice(["smooth", "layered"]), 1e-9
    return _case(None, call, (nx, ny), J, w_outer, w_sub, precision, nrhs, medium, tol)


# ---------------------------------------------------------------- inputs
def _grid(case):
    dim = 3 if case["nz"] > 1 else 2
    n = (case["nx"], case["ny"], case["nz"])[:dim]
    return n, 1.0 / (n[0] + 1)


def _medium(case, seed):
    n, _ = _grid(case)
    if case["medium"] == "layered":
        return media.layered_medium(n, seed=seed, nlayers=8, pert_sigma=30.0, pert_seed=seed + 1)
    # correlation length about a twentieth (2-D) or an eighth (3-D) of the side, as the
    # repository's smooth workloads have it; c in [1, 3] and [1, 2]
    sigma = max(2.0, max(n) / (20.0 if len(n) == 2 else 8.0))
    return media.smooth_medium(n, sigma, 1.0, 3.0 if len(n) == 2 else 2.0, seed)


def _positions(case, seed):
    """One source: anywhere inside.  Several: on the top row (2-D) or top plane (3-D)."""
    n, _ = _grid(case)
    rng = np.random.default_rng(seed + 7)
    if case["nrhs"] == 1:
        return [tuple(int(rng.integers(k // 4, k - k // 4)) for k in n)]
    pts = []
    for _ in range(case["nrhs"]):
        p = [int(rng.integers(0, k)) for k in n]
        p[1] = 0
        pts.append(tuple(p))
    return pts


def _omega(case, c):
    _, h = _grid(case)
    return media.omega_for(c, h, 8.0)


def _handle(case, c, omega):
    _, h = _grid(case)
    panel = case["nrhs"] if case["nrhs"] > 4 else 0
    return helm.HelmDD(c, h, omega, case["w_outer"], case["w_sub"], case["J"], case["precision"], panel=panel)


def _padded_shape(case):
    n, _ = _grid(case)
    return tuple(k + 2 * case["w_outer"] for k in reversed(n))


def _sources(case, seed):
    n, h = _grid(case)
    f = torch.zeros((case["nrhs"], math.prod(_padded_shape(case))), dtype=torch.complex128, device=DEV)
    for b, p in enumerate(_positions(case, seed)):
        f[b, media.padded_index(p, n, case["w_outer"])] = 1.0 / h ** len(n)
    return f.reshape((case["nrhs"],) + _padded_shape(case))


def _random_field(case, seed):
    g = torch.Generator(device=DEV).manual_seed(seed)
    s = (case["nrhs"],) + _padded_shape(case) + (2,)
    return torch.view_as_complex(torch.randn(s, dtype=torch.float64, device=DEV, generator=g))


def _receivers(case):
    n, _ = _grid(case)
    return np.array([media.padded_index((x, 0), n, case["w_outer"]) for x in range(1, n[0], 5)], dtype=np.int64)


def _misfit_inputs(case, seed):
    """Squared slowness of the current model, a background model, sources and receivers."""
    n, h = _grid(case)
    c0 = _medium(case, seed)
    c = media.blob_medium(n, h, c0, seed=seed + 3)
    src = np.array([media.padded_index(p, n, case["w_outer"]) for p in _positions(case, seed)], dtype=np.int64)
    return 1.0 / (c * c), c0, src, _receivers(case), float(max(c.max(), c0.max()))


def prepare(case, seed):
    call = case["call"]
    if call == "misfit":
        m, c0, src, rec, c_ref = _misfit_inputs(case, seed)
        _, h = _grid(case)
        omega = _omega(case, c0)
        # observed data: the background model's fields at the receivers
        g0 = helm.HelmDD(c0, h, omega, case["w_outer"], case["w_sub"], case["J"], case["precision"], c_ref=c_ref).factor()
        u, _ = g0.solve(_sources(case, seed), tol=1e-10)
        d = u.reshape(case["nrhs"], -1)[:, torch.as_tensor(rec, device=DEV)].cpu().numpy()
        g0.close()
        spec = dict(h=h, omega=omega, w_outer=case["w_outer"], w_sub=case["w_sub"], J=case["J"], src=src, rec=rec,
                    d=d, precision=case["precision"], c_ref=c_ref, tol=case["tol"],
                    panel=case["nrhs"] if case["nrhs"] > 4 else 0)
        return {"case": case, "m": torch.tensor(m, dtype=torch.float64, device=DEV), "spec": spec}
    c = _medium(case, seed)
    omega = _omega(case, c)
    if call == "newmodel":
        return {"case": case, "c": c, "omega": omega, "f": _sources(case, seed)}
    state = {"case": case, "g": _handle(case, c, omega)}
    if call == "matvec":
        state["f"] = _random_field(case, seed)
        return state
    state["g"].factor()
    state["f"] = _random_field(case, seed) if call == "precond" else _sources(case, seed)
    return state


def run(state):
    case = state["case"]
    call = case["call"]
    if call == "solve":
        return state["g"].solve(state["f"], tol=case["tol"])[0]
    if call == "reduced":
        return state["g"].solve_reduced(state["f"], tol=case["tol"])[0]
    if call == "precond":
        return state["g"].apply_precond(state["f"])
    if call == "matvec":
        return state["g"].matvec(state["f"])
    if call == "newmodel":
        g = _handle(case, state["c"], state["omega"]).factor()
        u, _ = g.solve(state["f"], tol=case["tol"])
        g.close()
        return u
    m = state["m"].detach().requires_grad_(True)
    J = helm.misfit(m, state["spec"])
    J.backward()
    return {"misfit": J.detach(), "grad": m.grad}


def work(case):
    """One pass: the factor blocks read once per strip solve, fields read and written once per
    iteration, and the arithmetic of the block solves, for a nominal number of iterations."""
    n, _ = _grid(case)
    N = [k + 2 * case["w_outer"] for k in n]
    vol, B, J = math.prod(N), case["nrhs"], case["J"]
    field = 16.0 * vol * B
    if case["call"] == "matvec":
        return {"bytes": 2 * field + 8.0 * vol, "flops": 26.0 * vol * B}
    esz = 16 if case["precision"] == "fp64" else 8
    Nz = N[2] if len(N) == 3 else 1
    W = N[0] / J + 1 + 2.0 * case["w_sub"] * (J - 1) / J      # mean strip width
    blk = W * Nz
    entries = N[1] * blk * blk                                # of one strip's diagonal blocks
    solves = 2 * J - 1
    sweep = {"bytes": solves * entries * esz + 4 * field, "flops": solves * 16.0 * entries * B + 30.0 * vol * B}
    factor = {"bytes": J * entries * esz, "flops": 8.0 * J * entries * blk}
    iters = {"precond": 1, "solve": 8, "newmodel": 8, "reduced": 24, "misfit": 24}[case["call"]]
    once = 1 if case["call"] in ("newmodel", "misfit") else 0
    return {k: iters * sweep[k] + once * factor[k] for k in ("bytes", "flops")}


# ---------------------------------------------------------------- 64-bit answers
# The operator from its definition: on each axis -alpha(x) d/dx (alpha d/dx) by centred
# differences with alpha at grid and half points, minus k^2; alpha = 1 / (1 + i sigma / omega),
# sigma = sigma0 (d / L)^2, sigma0 = 3 c_ref ln(1e6) / (2 L) in a layer of width L; zero one
# point beyond the grid; the speed is extended by its edge values.
def _alpha(x2, lo2, hi2, w, h, omega, c_ref):
    """alpha at positions x2 (half steps) with layers of w points beyond lo2 and hi2 (None: no layer)."""
    d2 = np.zeros(len(x2))
    if w > 0:
        if lo2 is not None:
            d2 = np.maximum(d2, lo2 - x2)
        if hi2 is not None:
            d2 = np.maximum(d2, x2 - hi2)
    L = max(w, 1) * h
    sigma = 3.0 * c_ref * math.log(1e6) / (2.0 * L) * (np.minimum(0.5 * d2 * h, L) / L) ** 2
    return 1.0 / (1.0 + 1j * sigma / omega)


def _axis(N, w, h, omega, c_ref):
    """alpha at the grid points and at the half points -1/2 .. N-1/2 of a padded axis."""
    lo, hi = 2 * w - 1, 2 * (N - w) - 1
    return (_alpha(2 * np.arange(N), lo, hi, w, h, omega, c_ref),
            _alpha(2 * np.arange(N + 1) - 1, lo, hi, w, h, omega, c_ref))


def _tri(a, ah, h):
    """The axis operator divided by alpha at the point: symmetric tridiagonal (diagonal, off-diagonal)."""
    return (ah[:-1] + ah[1:]) / h ** 2, -ah[1:-1] / h ** 2


def _k2_padded(case, c, omega):
    return (omega / np.pad(c, case["w_outer"], mode="edge")) ** 2


class _Direct:
    """A u = f by block elimination along y, blocks of N_x N_z unknowns, complex128 on the GPU."""

    def __init__(self, case, c, omega, c_ref):
        n, h = _grid(case)
        w = case["w_outer"]
        N = [k + 2 * w for k in n]
        ax = [_axis(Na, w, h, omega, c_ref) for Na in N]
        k2 = _k2_padded(case, c, omega)
        k2 = k2 if len(n) == 3 else k2[None]                     # [Nz, Ny, Nx]
        if len(n) == 2:
            ax.append((np.ones(1), None))
            N.append(1)
        self.N = N
        Nx, Ny, Nz = N
        sx, sy, sz = (1.0 / a[0] for a in ax)
        dx, ox = _tri(*ax[0], h)
        dy, _ = _tri(*ax[1], h)
        T = lambda v: torch.as_tensor(np.ascontiguousarray(v), device=DEV)  # noqa: E731
        Tx = torch.diag(T(dx)) + torch.diag(T(ox), 1) + torch.diag(T(ox), -1)
        P = torch.kron(torch.diag(T(sz.astype(complex))), Tx)
        if Nz > 1:
            dz, oz = _tri(*ax[2], h)
            P = P + torch.kron(torch.diag(T(dz)) + torch.diag(T(oz), 1) + torch.diag(T(oz), -1), torch.diag(T(sx)))
        sxz = T(np.kron(sz, sx))
        cy = T(ax[1][1])
        self.C = [-sxz * cy[k] / h ** 2 for k in range(Ny + 1)]   # coupling of rows k-1 and k
        self.sxz, self.sy = sxz, T(sy)
        k2 = T(k2)
        self.X = []
        for k in range(Ny):
            D = P * self.sy[k] + torch.diag(sxz * T(dy)[k] - sxz * self.sy[k] * k2[:, k, :].reshape(-1))
            if k:
                D = D - self.C[k][:, None] * self.X[-1] * self.C[k][None, :]
            self.X.append(torch.linalg.inv(D))

    def solve(self, f):
        """f [B, Nz, Ny, Nx] -> u, both torch complex128."""
        Nx, Ny, Nz = self.N
        B = f.shape[0]
        f = f.reshape(B, Nz, Ny, Nx)
        r = [(f[:, :, k, :].reshape(B, -1) * self.sxz * self.sy[k]).T for k in range(Ny)]
        for k in range(Ny):
            r[k] = self.X[k] @ (r[k] - self.C[k][:, None] * r[k - 1] if k else r[k])
        for k in range(Ny - 2, -1, -1):
            r[k] = r[k] - self.X[k] @ (self.C[k + 1][:, None] * r[k + 1])
        return torch.stack([v.T.reshape(B, Nz, Nx) for v in r], dim=2)


def _exact_matvec(case, c, omega, u):
    n, h = _grid(case)
    N = [k + 2 * case["w_outer"] for k in n]
    out = -torch.as_tensor(_k2_padded(case, c, omega), device=DEV) * u
    for a, Na in enumerate(N):
        al, ah = (torch.as_tensor(v, device=DEV) for v in _axis(Na, case["w_outer"], h, omega, float(c.max())))
        v = u.movedim(-1 - a, -1)
        z = torch.zeros_like(v[..., :1])
        flux = ah * torch.diff(torch.cat([z, v, z], -1), dim=-1)
        out = out - (al * torch.diff(flux, dim=-1) / h ** 2).movedim(-1, -1 - a)
    return out


def _exact_precond(case, c, omega, f):
    """The double sweep: strips of the columns beta_j+1 .. beta_{j+1}+1 with added layers, forward on
    f, backward on the residual, each strip passing -+2 delta d_x of its solution to the next."""
    (nx, _), h = _grid(case)
    w, ws, J, c_ref = case["w_outer"], case["w_sub"], case["J"], float(c.max())
    k2 = _k2_padded(case, c, omega)
    Ny, Nx = k2.shape
    ay, ayh = _axis(Ny, w, h, omega, c_ref)
    sy, (dy, _) = 1.0 / ay, _tri(ay, ayh, h)
    beta = [w - 1 + int(math.floor(j * nx / J + 0.5)) for j in range(J + 1)]
    beta[0], beta[J] = -1, Nx - 1
    strips = []
    for j in range(J):
        lo, hi = beta[j] + 1, beta[j + 1] + 1 if j < J - 1 else Nx - 1
        lp, rp = (ws if j > 0 else 0), (ws if j < J - 1 else 0)
        W = lp + hi - lo + 1 + rp

        def al(x2):
            g = x2 + 2 * (lo - lp)
            a = _alpha(g, 2 * w - 1, 2 * (Nx - w) - 1, w, h, omega, c_ref)
            if lp:
                a = np.where(g < 2 * lo - 1, _alpha(g, 2 * lo - 1, None, ws, h, omega, c_ref), a)
            if rp:
                a = np.where(g > 2 * hi + 1, _alpha(g, None, 2 * hi + 1, ws, h, omega, c_ref), a)
            return a
        ax, axh = al(2 * np.arange(W)), al(2 * np.arange(W + 1) - 1)
        sx, (dx, ox) = 1.0 / ax, _tri(ax, axh, h)
        col = np.clip(np.arange(W) + lo - lp, lo, hi)
        strips.append(dict(lo=lo, hi=hi, lp=lp, W=W, sx=sx, dx=dx, ox=ox, k2=k2[:, col]))
    # block elimination along y of all strips of one width together
    for W in sorted({s["W"] for s in strips}):
        grp = [s for s in strips if s["W"] == W]
        i = np.arange(W)
        S = lambda key: np.stack([s[key] for s in grp])  # noqa: E731
        sx, dx, ox, kk = S("sx"), S("dx"), S("ox"), S("k2")
        X, prev = [], None
        for k in range(Ny):
            D = np.zeros((len(grp), W, W), complex)
            D[:, i, i] = sy[k] * dx + sx * dy[k] - sx * sy[k] * kk[:, k]
            D[:, i[:-1], i[1:]] = sy[k] * ox
            D[:, i[1:], i[:-1]] = sy[k] * ox
            if k:
                cc = -sx * ayh[k] / h ** 2
                D -= cc[:, :, None] * prev * cc[:, None, :]
            prev = np.linalg.inv(D)
            X.append(prev)
        for q, s in enumerate(grp):
            s["X"] = [x[q] for x in X]

    def solve(s, r):   # r [Ny, W, B], paper form
        cy = [-s["sx"][:, None] * ayh[k] / h ** 2 for k in range(Ny + 1)]
        y = [None] * Ny
        for k in range(Ny):
            b = r[k] * s["sx"][:, None] * sy[k]
            y[k] = s["X"][k] @ (b - cy[k] * y[k - 1] if k else b)
        for k in range(Ny - 2, -1, -1):
            y[k] = y[k] - s["X"][k] @ (cy[k + 1] * y[k + 1])
        return np.stack(y)

    F = np.moveaxis(f.cpu().numpy(), 0, -1)                     # [Ny, Nx, B]
    B = F.shape[-1]

    def rhs(s, field, a, b):
        r = np.zeros((Ny, s["W"], B), complex)
        a, b = max(a, 0), min(b, Nx - 1)
        r[:, a - s["lo"] + s["lp"]:b + 1 - s["lo"] + s["lp"]] = field[:, a:b + 1]
        return r
    V = np.zeros_like(F)
    jump = None
    for j, s in enumerate(strips):
        r = rhs(s, F, beta[j] + 1, beta[j + 1])
        if j:                                                   # columns beta_j, beta_j + 1
            q = beta[j] - s["lo"] + s["lp"]
            r[:, q:q + 2] -= jump[:, None] / h ** 2
        x = solve(s, r)
        o = s["lp"]
        V[:, beta[j] + 1:beta[j + 1] + 1] = x[:, o:o + beta[j + 1] - beta[j]]
        e = o + s["hi"] - s["lo"]
        jump = x[:, e] - x[:, e - 1]
    if J == 1:
        return torch.as_tensor(np.moveaxis(V, -1, 0).copy())
    Vt = torch.as_tensor(np.moveaxis(V, -1, 0).copy(), device=DEV)
    G = np.moveaxis((f - _exact_matvec(case, c, omega, Vt)).cpu().numpy(), 0, -1)
    out = V.copy()
    jump = None
    for j in range(J - 2, -1, -1):
        s = strips[j]
        a, b = (beta[j] + 2 if j else 0), beta[j + 1] + 1
        r = rhs(s, G, a, b)
        if jump is not None:                                    # columns beta_{j+1} + 1, + 2
            q = beta[j + 1] + 1 - s["lo"] + s["lp"]
            r[:, q:q + 2] += jump[:, None] / h ** 2
        x = solve(s, r)
        o = s["lp"] - s["lo"]
        out[:, a:b + 1] += x[:, o + a:o + b + 1]
        jump = x[:, s["lp"] + 1] - x[:, s["lp"]]
    return torch.as_tensor(np.moveaxis(out, -1, 0).copy())


def exact(case, seed):
    n, h = _grid(case)
    N = [k + 2 * case["w_outer"] for k in n]
    if case["call"] == "precond":
        c = _medium(case, seed)
        return _exact_precond(case, c, _omega(case, c), _random_field(case, seed))
    if case["call"] == "matvec":
        c = _medium(case, seed)
        return _exact_matvec(case, c, _omega(case, c), _random_field(case, seed))
    blk = N[0] * (N[2] if len(N) == 3 else 1)
    if 8.0 * N[1] * blk ** 3 > 4e12 or 16.0 * N[1] * blk ** 2 > 6e10:   # over about 20 seconds, or too large
        return None
    if case["call"] != "misfit":
        c = _medium(case, seed)
        return _Direct(case, c, _omega(case, c), float(c.max())).solve(_sources(case, seed)).reshape(
            (case["nrhs"],) + _padded_shape(case))
    m, c0, src, rec, c_ref = _misfit_inputs(case, seed)
    omega = _omega(case, c0)
    f = _sources(case, seed)
    rec = torch.as_tensor(rec, device=DEV)
    d = _Direct(case, c0, omega, c_ref).solve(f).reshape(case["nrhs"], -1)[:, rec]
    A = _Direct(case, 1.0 / np.sqrt(m), omega, c_ref)
    u = A.solve(f).reshape(case["nrhs"], -1)
    res = u[:, rec] - d
    S = (A.sy[:, None] * A.sxz[None, :]).reshape(-1)              # diagonal scaling that symmetrises A
    q = torch.zeros_like(u)
    q[:, rec] = res.conj()
    mu = A.solve((q / S).reshape(f.shape)).reshape(case["nrhs"], -1)
    g = (omega ** 2 * (S * mu * u).real.sum(0)).reshape(_padded_shape(case))
    w = case["w_outer"]
    for axis in (0, 1):                                          # adjoint of the edge extension
        g = g.movedim(axis, 0)
        k = g.shape[0]
        mid = g[w:k - w].clone()
        mid[0] += g[:w].sum(0)
        mid[-1] += g[k - w:].sum(0)
        g = mid.movedim(0, axis)
    return {"misfit": 0.5 * (res.abs() ** 2).sum(), "grad": g}
