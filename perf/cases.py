"""The workloads this library is timed on.

Every case goes through the public entry points: the operators of
`gpe.Context`, `gpe.Batch`, the autograd wrappers.  A case is a dict of plain
values; `kind` selects one of the calls below.  Grids are powers of two per axis
(8 .. 512, the library's range); batches have any number of fields.

    h         H_phi f on one field (gpe_apply_H)
    hbatch    H_phi f on many 2D fields with one potential (gpe_apply_H_batch)
    precond   P_C r with the adaptive shift (gpe_precond)
    energy    E and its gradient with respect to phi, V, eta and omega
              (autograd.energy, forward and backward)
    adjoint   dL/dV of a loss of the ground-state density (gpe_density_adjoint)
    solve     a ground state to the default tolerance (gpe_pcg_solve)
    sweep     many ground states in one launch (gpe.Batch)
    start     Thomas-Fermi initial data on a grid and its interpolation onto the
              twice as fine one (gpe_thomas_fermi, gpe_interpolate)

Ground states are computed in traps and at rotation speeds below the entry of
vortices, where the state reached from the Gaussian is the same for every order
of the sums; mixed-precision solves hand their state on in complex64, the type
that the context's operators take.
"""
import math

import numpy as np
import torch

from paper_1611_02045_gb300 import autograd, gpe, inputs

DEV = "cuda"
F64, C64, C128 = torch.float64, torch.complex64, torch.complex128


def listed():
    return [
        # one operator call on a small 2D field: what a user's own iteration on a laptop-size grid pays per call
        dict(name="h_64x64_c64", kind="h", nx=64, ny=64, nz=0, prec="c64", same=False),
        # H phi in double precision on a 3D grid (spectral accuracy, reference energies)
        dict(name="h_128cube_c128", kind="h", nx=128, ny=128, nz=128, prec="c128", same=False),
        # H phi on a field beyond the L2 cache (268 MB), the FFT passes' own workload
        dict(name="h_256x256x512_c64", kind="h", nx=256, ny=256, nz=512, prec="c64", same=True),
        # residuals of a whole batch of states, the roofline workload of the benchmark
        dict(name="hbatch_512x256sq_c64", kind="hbatch", nx=256, count=512, prec="c64", same=True),
        # linear responses of an odd number of states: operand and density differ
        dict(name="hbatch_333x128sq_c64", kind="hbatch", nx=128, count=333, prec="c64", same=False),
        # the preconditioner with its adaptive shift on an anisotropic 3D grid
        dict(name="precond_256x128x64_c64", kind="precond", nx=256, ny=128, nz=64, prec="c64"),
        # a training step on the energy at a fixed field: gradients of phi, V, eta, omega
        dict(name="energy_grad_256sq_c128", kind="energy", nx=256, ny=256, nz=0, prec="c128"),
        # the backward pass of a loss of the ground-state density
        dict(name="adjoint_256sq_c128", kind="adjoint", nx=256, prec="c128", eta=500.0, omega=0.3),
        # one ground state in 2D, mixed precision (the default mode of the README)
        dict(name="solve_256sq_mixed", kind="solve", nx=256, nz=0, prec="mixed", eta=500.0, omega=0.3, L=16.0),
        # one ground state in 3D, mixed precision
        dict(name="solve_128cube_mixed", kind="solve", nx=128, nz=128, prec="mixed", eta=1000.0, omega=0.2, L=8.0),
        # a parameter sweep: 24 ground states on 128^2, 256^2 and 512^2 grids in one launch
        dict(name="sweep_24_mixed", kind="sweep", count=24, small=128, large=512),
        # the first steps of a multigrid run: initial data on 256^2, interpolated onto 512^2
        dict(name="start_256sq_to_512sq", kind="start", nx=256, ny=256, nz=0, eta=500.0),
    ]


def _grid(rng, lo, hi, dims, least=3, most=9):
    """log2 sizes of `dims` axes with lo <= their sum <= hi, not too flat."""
    while True:
        e = [rng.randint(least, most) for _ in range(dims)]
        if lo <= sum(e) <= hi and max(e) - min(e) <= 4:
            return [1 << k for k in e]


def draw(rng):
    kind = rng.choice(["h", "h", "hbatch", "hbatch", "precond", "energy", "adjoint", "solve", "solve", "sweep", "start"])
    prec = rng.choice(["c64", "c64", "c128"])
    if kind in ("h", "precond", "energy"):
        dims = rng.choice([2, 3])
        hi = 25 if prec == "c64" else 22
        total = rng.uniform(12, hi if dims == 3 else 18)
        n = _grid(rng, math.floor(total), math.ceil(total), dims) + [0]
        case = dict(kind=kind, nx=n[0], ny=n[1], nz=n[2], prec=prec)
        if kind == "h":
            case["same"] = rng.random() < 0.5
        return case
    if kind == "hbatch":
        nx = rng.choice([32, 64, 128, 256, 256])
        top = (1 << (25 if prec == "c64" else 22)) // (nx * nx)
        return dict(kind=kind, nx=nx, count=int(round(math.exp(rng.uniform(0.0, math.log(top))))), prec=prec,
                    same=rng.random() < 0.5)
    if kind == "adjoint":
        return dict(kind=kind, nx=rng.choice([64, 128, 256]), prec="c128", eta=round(rng.uniform(50, 600), 1),
                    omega=round(rng.uniform(0.0, 0.35), 3))
    if kind == "solve":
        eta, omega = round(rng.uniform(50, 600), 1), round(rng.uniform(0.0, 0.35), 3)
        prec = rng.choice(["mixed", "mixed", "c128"])
        if rng.random() < 0.3:
            return dict(kind=kind, nx=rng.choice([32, 64]), nz=64, prec=prec, eta=eta, omega=omega, L=8.0)
        return dict(kind=kind, nx=rng.choice([64, 128, 256, 512]), nz=0, prec=prec, eta=eta, omega=omega,
                    L=round(rng.uniform(10.0, 16.0), 2))
    if kind == "sweep":
        return dict(kind=kind, count=rng.randint(2, 24), small=rng.choice([32, 64, 128]), large=rng.choice([128, 256, 512]))
    dims = rng.choice([2, 3])
    n = _grid(rng, 10, 20 if dims == 3 else 16, dims, 4, 8) + [0]
    return dict(kind=kind, nx=n[0], ny=n[1], nz=n[2], eta=round(math.exp(rng.uniform(4, 8)), 1))


# --- problems ------------------------------------------------------------------

def _n(case):
    n = (case["nx"], case.get("ny", case["nx"]))
    return n + (case["nz"],) if case.get("nz") else n


def _box(n, L=8.0):
    return tuple(float(L) for _ in n)


def _trap(n, L, seed, amp=0.1, kappa=0.0):
    """Harmonic trap (twice as stiff along z), a quartic part and a few seeded bumps."""
    gammas = [1.0, 1.0, 2.0][:len(n)]
    return inputs.harmonic_quartic(n, L, kappa, gammas) + amp * inputs.smooth_bumps(n, L, seed)


def _guess(n, L, seed):
    g = inputs.anisotropic_gaussian(n, L, [1.0, 1.0, 2.0]) if len(n) == 3 else inputs.phi_a(n, L)
    return inputs.perturbed(g, seed, n, L)


def _field(shape, dtype, seed):
    """Dense random fields (uniform real and imaginary parts) on the device."""
    g = torch.Generator(device=DEV).manual_seed(seed)
    real = F64 if dtype == C128 else torch.float32
    x = torch.rand(tuple(shape) + (2,), dtype=real, device=DEV, generator=g).mul_(2.0).sub_(1.0)
    return torch.view_as_complex(x)


def _instances(case, seed):
    """The sweep: grids small, 2 small, .. large in turn, parameters from the seed."""
    sizes, n = [], case["small"]
    while n <= max(case["small"], case["large"]):
        sizes.append(n)
        n *= 2
    u = inputs.uniform_pm1(seed, 3 * case["count"]).reshape(-1, 3)
    out = []
    for i in range(case["count"]):
        m = sizes[i % len(sizes)]
        n, L = (m, m), _box((m, m), 12.0)
        kappa = 0.05 if u[i, 2] > 0 else 0.0
        out.append(dict(n=n, L=L, eta=(100.0, 250.0, 500.0)[min(int(1.5 * (u[i, 1] + 1.0)), 2)],
                        omega=0.3 * 0.5 * (u[i, 0] + 1.0), V=_trap(n, L, seed + i, 0.05, kappa),
                        phi0=_guess(n, L, seed + 100 + i), prec=gpe.GPE_MIXED))
    return out


ETA, OMEGA = 100.0, 0.6  # of the single operator calls


def _dtype(case):
    return C128 if case["prec"] == "c128" else C64


def _prec(case):
    return gpe.GPE_FP64 if case["prec"] == "c128" else gpe.GPE_MIXED


def _operator_inputs(case, seed):
    """(V, phi, operand) of the operator cases; the operand of `same` is phi itself."""
    n = _n(case)
    shape = n[::-1]
    if case["kind"] == "hbatch":
        shape = (case["count"],) + shape
    phi = _field(shape, _dtype(case), seed)
    f = phi if case.get("same") else _field(shape, _dtype(case), seed + 1)
    V = torch.from_numpy(inputs.harmonic(n, _box(n))).to(DEV)
    return V, phi, f


def _adjoint_inputs(case, seed):
    n = _n(case)
    L = _box(n, 16.0 if case["nx"] >= 256 else 12.0)
    V = _trap(n, L, seed)
    X, Y = inputs.mesh(n, L)
    u = inputs.uniform_pm1(seed + 7, 2)
    g_rho = np.exp(-((X - 2 * u[0]) ** 2 + (Y - 2 * u[1]) ** 2) / 8.0)  # a detector window
    return n, L, torch.from_numpy(V).to(DEV), torch.from_numpy(_guess(n, L, seed + 1)).to(DEV), \
        torch.from_numpy(g_rho).to(DEV)


ADJ_TOL = 1e-12


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("h", "hbatch", "precond", "energy"):
        n = _n(case)
        V, phi, f = _operator_inputs(case, seed)
        ctx = gpe.Context(n, _box(n), ETA, OMEGA, V, prec=_prec(case))
        state = dict(case=case, ctx=ctx, phi=phi, f=f, out=torch.empty_like(f))
        if kind == "energy":
            state["V"] = V.requires_grad_()
            state["phi"] = phi.requires_grad_()
            state["eta"] = torch.tensor(ETA, dtype=F64, requires_grad=True)
            state["omega"] = torch.tensor(OMEGA, dtype=F64, requires_grad=True)
        return state
    if kind == "adjoint":
        n, L, V, phi, g_rho = _adjoint_inputs(case, seed)
        ctx = gpe.Context(n, L, case["eta"], case["omega"], V, prec=_prec(case))
        opts = gpe.solve_opts_default()
        opts.tol_res_inf = 1e-11
        ctx.pcg_solve(phi, opts)
        return dict(case=case, ctx=ctx, phi=phi, g_rho=g_rho, grad=torch.empty_like(g_rho))
    if kind == "solve":
        n = _n(case)
        L = _box(n, case["L"])
        ctx = gpe.Context(n, L, case["eta"], case["omega"], _trap(n, L, seed), prec=_prec(case))
        return dict(case=case, ctx=ctx, phi0=torch.from_numpy(_guess(n, L, seed + 1)).to(DEV))
    if kind == "sweep":
        ws = _instances(case, seed)
        return dict(case=case, batch=gpe.Batch(ws), phi0=[torch.from_numpy(w["phi0"]).to(DEV) for w in ws])
    n = _n(case)
    fine = tuple(2 * m for m in n)
    L, eta = _box(n, 16.0), case["eta"]
    coarse_ctx = gpe.Context(n, L, eta, 0.0, _trap(n, L, seed), prec=gpe.GPE_MIXED)
    fine_ctx = gpe.Context(fine, L, eta, 0.0, _trap(fine, L, seed), prec=gpe.GPE_MIXED)
    return dict(case=case, ctx=coarse_ctx, fine=fine_ctx, coarse_phi=torch.empty(n[::-1], dtype=C128, device=DEV),
                fine_phi=torch.empty(fine[::-1], dtype=C128, device=DEV))


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "h":
        s["ctx"].apply_H(s["phi"], s["f"], s["out"])
        return s["out"]
    if kind == "hbatch":
        s["ctx"].apply_H_batch(case["count"], s["phi"], s["f"], s["out"])
        return s["out"]
    if kind == "precond":
        s["ctx"].precond(s["phi"], s["f"], 0.0, s["out"])
        return s["out"]
    if kind == "energy":
        E = autograd.energy(s["phi"], s["V"], s["eta"], s["omega"], s["ctx"])
        grads = torch.autograd.grad(E, (s["phi"], s["V"], s["eta"], s["omega"]))
        return (E.detach(),) + grads
    if kind == "adjoint":
        s["ctx"].density_adjoint(s["phi"], s["g_rho"], s["grad"], tol=ADJ_TOL, check=False)
        return s["grad"]
    if kind == "solve":
        phi = s["phi0"].clone()
        rep = s["ctx"].pcg_solve(phi)
        return phi.to(C64), rep["E"], rep["lam"]
    if kind == "sweep":
        phis = [p.clone() for p in s["phi0"]]
        _, reps = s["batch"].solve(phis)
        return [p.to(C64) for p in phis], [r["E"] for r in reps]
    mu = s["ctx"].thomas_fermi(s["coarse_phi"])
    s["ctx"].interpolate_to(s["fine"], s["coarse_phi"], s["fine_phi"])
    return s["coarse_phi"], s["fine_phi"], mu


# --- work ------------------------------------------------------------------------

def _pair_flops(n):
    """Forward and inverse transforms along every axis, 5 M log2 M per line and direction."""
    N = math.prod(n)
    return 10.0 * N * sum(math.log2(m) for m in n)


#: iterations of one solve: about what Algorithm 2 takes from the Gaussian in these traps
SOLVE_ITERS = 60
ADJOINT_ITERS = 60


def _iteration_flops(n):
    """H phi, P_C r (a transform pair each) and the forward transforms of A p, with the pointwise work."""
    return 2.5 * _pair_flops(n) + 100.0 * math.prod(n)


def work(case):
    kind = case["kind"]
    n = _n(case) if kind != "sweep" else None
    if kind in ("h", "hbatch", "precond", "energy"):
        N = math.prod(n)
        e = 16 if case["prec"] == "c128" else 8
        v = e // 2
        if kind == "hbatch":
            B = case["count"]
            return dict(bytes=B * N * e * (2 if case["same"] else 3) + N * v, flops=B * (_pair_flops(n) + 20.0 * N))
        if kind == "h":
            return dict(bytes=N * (e * (2 if case["same"] else 3) + v), flops=_pair_flops(n) + 20.0 * N)
        if kind == "precond":  # the shift lambda~(phi) and P_C r
            return dict(bytes=N * (3 * e + v), flops=2 * _pair_flops(n) + 40.0 * N)
        return dict(bytes=N * (2 * e + 8 + 8), flops=_pair_flops(n) + 30.0 * N)
    if kind == "adjoint":
        N = math.prod(n)
        return dict(bytes=N * (16 + 8 + 8 + 8), flops=ADJOINT_ITERS * (2 * _pair_flops(n) + 100.0 * N))
    if kind == "solve":
        N = math.prod(n)
        return dict(bytes=N * 40, flops=SOLVE_ITERS * _iteration_flops(n))
    if kind == "sweep":
        sizes, m = [], case["small"]
        while m <= max(case["small"], case["large"]):
            sizes.append(m)
            m *= 2
        grids = [(sizes[i % len(sizes)],) * 2 for i in range(case["count"])]
        return dict(bytes=sum(40 * math.prod(g) for g in grids), flops=SOLVE_ITERS * sum(_iteration_flops(g) for g in grids))
    N = math.prod(n)  # the coarse V and both states; the mass integral and one interpolation
    return dict(bytes=N * (8 + 16) + 16 * N * 2 ** len(n), flops=60.0 * N + 5.0 * 2 ** len(n) * N * sum(math.log2(m) for m in n))


# --- exact values: plain torch in 64 bits ------------------------------------------

class _Exact:
    """The discrete operators (Fourier pseudo-spectral, x fastest) in complex128 by torch.fft."""

    def __init__(self, n, L, eta, omega, V):
        self.d, self.eta, self.omega = len(n), eta, omega
        self.V = torch.as_tensor(V, dtype=F64, device=DEV)
        self.w = math.prod(2.0 * l / m for l, m in zip(L, n))
        self.x, self.k = [], []
        for i, (m, l) in enumerate(zip(n, L)):
            j = torch.arange(m, dtype=F64, device=DEV)
            shape = [1] * self.d
            shape[self.d - 1 - i] = m
            self.x.append((-l + j * (2.0 * l / m)).reshape(shape))
            self.k.append((torch.where(j < m // 2, j, j - m) * (math.pi / l)).reshape(shape))

    def along(self, f, axis, mult):
        return torch.fft.ifft(torch.fft.fft(f, dim=-1 - axis) * mult, dim=-1 - axis)

    def kin_rot(self, f):
        x, k = self.x, self.k
        out = self.along(f, 0, 0.5 * k[0] ** 2 + self.omega * x[1] * k[0])
        out += self.along(f, 1, 0.5 * k[1] ** 2 - self.omega * x[0] * k[1])
        return out + self.along(f, 2, 0.5 * k[2] ** 2) if self.d == 3 else out

    def H(self, phi, f):
        return self.kin_rot(f) + (self.V + self.eta * self.abs2(phi)) * f

    @staticmethod
    def abs2(f):
        return f.real ** 2 + f.imag ** 2

    def dot(self, f, g):
        return self.w * (f.real * g.real + f.imag * g.imag).sum()

    def rotation(self, phi):
        """<phi, L_z phi>"""
        x, k = self.x, self.k
        return -self.dot(phi, self.along(phi, 0, x[1] * k[0]) - self.along(phi, 1, x[0] * k[1]))

    def shift(self, phi, lam):
        """lambda~ = int 1/2 |grad phi|^2 + V |phi|^2 + eta |phi|^4"""
        return lam + self.omega * self.rotation(phi)

    def P(self, phi, r, alpha):
        s = (alpha + self.V + self.eta * self.abs2(phi)).rsqrt()
        dims = tuple(range(-self.d, 0))
        return s * torch.fft.ifftn(torch.fft.fftn(s * r, dim=dims) / (alpha + 0.5 * sum(k * k for k in self.k)), dim=dims)

    def energy(self, phi, lam):
        return lam - 0.5 * self.eta * self.w * (self.abs2(phi) ** 2).sum()

    def ground_state(self, phi, tol, most=600):
        """Algorithm 2 with P_C, Polak-Ribiere, the model step and its halving; (phi, E, lambda)."""
        eta, w = self.eta, self.w
        phi = phi / self.dot(phi, phi).sqrt()
        p = r0 = rp0 = None
        for _ in range(most):
            Hp = self.H(phi, phi)
            lam = self.dot(phi, Hp)
            r = Hp - lam * phi
            if float(r.abs().max()) < tol:
                break
            Pr = self.P(phi, r, self.shift(phi, lam))
            rp = self.dot(r, Pr)
            d = -Pr
            if p is not None:
                d = d + torch.clamp(self.dot(r - r0, Pr) / rp0, min=0.0) * p
            p = d - self.dot(d, phi) * phi
            if float(self.dot(Hp, p)) >= 0:
                p = -Pr + self.dot(Pr, phi) * phi
            q = p / self.dot(p, p).sqrt()
            u, v, t = self.abs2(phi), phi.real * q.real + phi.imag * q.imag, self.abs2(q)
            R, aqq = self.dot(Hp, q), self.dot(q, self.kin_rot(q) + self.V * q)
            m = torch.stack([(u * u).sum(), (u * v).sum(), (v * v).sum(), (u * t).sum(), (v * t).sum(), (t * t).sum()]) * w
            R, aqq, lm, (U0, U1, V2, UW, VW, W2) = float(R), float(aqq), float(lam), m.tolist()
            curv = aqq + eta * UW + 2.0 * eta * V2 - lm
            th = -R / curv if curv > 0 else 0.1

            def dE(a):
                c, s = math.cos(a), math.sin(a)
                return (2 * c * s * R + s * s * (aqq - lm) + 0.5 * eta * (s ** 4 * (U0 + W2) + c * c * s * s * (4 * V2 + 2 * UW)
                                                                          + 4 * c * s ** 3 * (VW - U1)))
            for _ in range(30):
                if dE(th) < 0:
                    break
                th *= 0.5
            phi = math.cos(th) * phi + math.sin(th) * q
            phi = phi / self.dot(phi, phi).sqrt()
            r0, rp0 = r, rp
        return phi, self.energy(phi, lam), lam

    def density_adjoint(self, phi, g_rho, tol=1e-14, most=2000):
        """dL/dV: conjugate gradients for K z = P rhs on the space orthogonal to phi (complex), rhs = 2/w g phi."""
        eta = self.eta
        lam = self.dot(phi, self.H(phi, phi))
        alpha = self.shift(phi, lam)

        def proj(h):
            return h - self.w * (phi.conj() * h).sum() * phi

        def K(f):
            return proj(self.H(phi, f) + eta * self.abs2(phi) * f + eta * phi * phi * f.conj() - lam * f)

        r = proj(2.0 / self.w * g_rho * phi)
        z, stop = torch.zeros_like(r), tol * float(self.dot(r, r).sqrt())
        y = proj(self.P(phi, r, alpha))
        p, ry = y, self.dot(r, y)
        for _ in range(most):
            q = K(p)
            a = ry / self.dot(p, q)
            z, r = z + a * p, r - a * q
            if float(self.dot(r, r).sqrt()) <= stop:
                break
            y = proj(self.P(phi, r, alpha))
            new = self.dot(r, y)
            p, ry = y + (new / ry) * p, new
        return -self.w * (z.real * phi.real + z.imag * phi.imag)


def _refine(f, axis):
    """Trigonometric interpolation onto twice the points along one axis, the Nyquist mode shared by both ends."""
    f = f.movedim(-1 - axis, -1)
    m = f.shape[-1]
    F = torch.fft.fft(f)
    G = torch.zeros(f.shape[:-1] + (2 * m,), dtype=f.dtype, device=f.device)
    G[..., :m // 2] = F[..., :m // 2]
    G[..., -m // 2 + 1:] = F[..., -m // 2 + 1:]
    G[..., m // 2] = G[..., -m // 2] = 0.5 * F[..., m // 2]
    return (2.0 * torch.fft.ifft(G)).movedim(-1, -1 - axis)


def exact(case, seed):
    kind = case["kind"]
    if kind in ("h", "hbatch", "precond", "energy"):
        n = _n(case)
        V, phi, f = _operator_inputs(case, seed)
        op = _Exact(n, _box(n), ETA, OMEGA, V)
        if kind == "hbatch":
            out = torch.empty(phi.shape, dtype=C128, device=DEV)
            for i in range(0, case["count"], 64):
                out[i:i + 64] = op.H(phi[i:i + 64].to(C128), f[i:i + 64].to(C128))
            return out
        phi, f = phi.to(C128), f.to(C128)
        if kind == "h":
            return op.H(phi, f)
        Hp = op.H(phi, phi)
        lam = op.dot(phi, Hp)
        if kind == "precond":
            return op.P(phi, f, op.shift(phi, lam))
        u = op.abs2(phi)
        return (op.energy(phi, lam), 2.0 * op.w * Hp, op.w * u, 0.5 * op.w * (u * u).sum(), -op.rotation(phi))
    if kind == "adjoint":
        n, L, V, phi, g_rho = _adjoint_inputs(case, seed)
        op = _Exact(n, L, case["eta"], case["omega"], V)
        phi, _, _ = op.ground_state(phi, 2e-12)
        return op.density_adjoint(phi, g_rho)
    if kind == "solve":
        n = _n(case)
        L = _box(n, case["L"])
        op = _Exact(n, L, case["eta"], case["omega"], _trap(n, L, seed))
        phi, E, lam = op.ground_state(torch.from_numpy(_guess(n, L, seed + 1)).to(DEV), 1e-10)
        return phi, E, lam
    if kind == "sweep":
        got = []
        for w in _instances(case, seed):
            op = _Exact(w["n"], w["L"], w["eta"], w["omega"], w["V"])
            got.append(op.ground_state(torch.from_numpy(w["phi0"]).to(DEV), 1e-10))
        return [g[0] for g in got], [g[1] for g in got]
    n = _n(case)
    L = _box(n, 16.0)
    V = torch.from_numpy(_trap(n, L, seed)).to(DEV)
    eta, w = case["eta"], math.prod(2.0 * l / m for l, m in zip(L, n))
    lo, hi = float(V.min()), float(V.max()) + eta / (w * V.numel())
    for _ in range(120):
        mid = 0.5 * (lo + hi)
        if w / eta * float(torch.clamp(mid - V, min=0.0).sum()) < 1.0:
            lo = mid
        else:
            hi = mid
    mu = 0.5 * (lo + hi)
    phi = torch.sqrt(torch.clamp(mu - V, min=0.0) / eta).to(C128)
    fine = phi
    for axis in range(len(n)):
        fine = _refine(fine, axis)
    return phi, fine, mu
