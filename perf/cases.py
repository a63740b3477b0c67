"""What the library is timed on: its public entry points over the sizes its users run.

A case is one call of the library on one synthetic cell (Gaussian wells in a
periodic cubic box, see ``workloads.gaussian_wells``) with its occupied states
set.  The cells are the repository's own workloads (tiny, molecule,
differentiation, block_freq and its reduced slice) and uneven cells of the
recipe of its many-cell batch.  The occupied states are what a user's program
has in hand from its ground-state code: they are computed here in plain torch
FP64 (dense for up to ``DENSE`` plane waves, block eigensolver above) once per
cell and process.  The fields change with the seed, the cell does not.

Times depend on the iteration counts of the solver; ``work`` takes nominal ones.  Calls that
amplify the errors of their solves step by step (Lanczos, gradient, many cells) set the
tolerance of the mixed path to 1e-12, single applications keep the default.
"""
import functools
import math

import numpy as np
import torch

import paper_1408_3036_gb300 as gw

DENSE = 4000                     # plane waves up to which H is diagonalised whole
PREC = {"fp64": gw.GW_FP64, "mixed": gw.GW_MIXED}
SIZES = (16, 18, 20, 24, 25, 30, 32, 36, 40, 45, 48)     # factors 2, 3, 5


def _case(**kw):
    c = dict(call="eps", prec="mixed", L=10.0, N=16, ecut=5.0, wells=4, depth=-2.0, sigma=1.0, nocc=4, cell=0,
             closed=True, nb=1, w_re=0.0, w_im=0.0, k=1, tol=0.0)
    c.update(kw)
    return c


def listed():
    mol = dict(L=20.0, N=48, ecut=10.0, wells=8, depth=-3.0, sigma=0.8, nocc=16, cell=1, closed=False)
    return [
        # one static eps~ application on the smallest cell: launches and latency
        _case(name="tiny_static_fp64", prec="fp64"),
        # a real frequency above the gap (the residue term of the self-energy) on an odd grid: indefinite SQMR, FP64
        _case(name="cell30_real_fp64", prec="fp64", L=9.3, N=30, ecut=5.5, wells=5, nocc=7, cell=11, w_re=0.21),
        # a complex frequency, one field, an odd grid with odd numbers of states and columns: a batch cell's step
        _case(name="cell45_complex_mixed", L=13.1, N=45, ecut=7.1, wells=9, nocc=13, cell=12, w_re=0.3, w_im=0.1),
        # the headline operation: static screening of the molecule, one field, mixed precision
        _case(name="molecule_static_mixed", **mol),
        # the same in FP64 throughout
        _case(name="molecule_static_fp64", prec="fp64", **mol),
        # the headline call: Lanczos with full re-orthogonalisation, then the inverse in the basis (solves to 1e-12: the
        # recursion amplifies their errors step by step)
        _case(name="molecule_lanczos_mixed", call="lanczos", k=16, tol=1e-12, **mol),
        # the model dielectric operator of the same cell (no linear solves)
        _case(name="molecule_model", call="model", prec="fp64", **mol),
        # density response to a block of perturbations at once, static
        _case(name="cell32_chi0_block_mixed", call="chi0", L=14.0, N=32, ecut=8.0, wells=6, nocc=8, cell=4, nb=8),
        # the adjoint: s = <phi|eps~^-1|phi> and ds/dV_loc, forward Lanczos and backward solves
        _case(name="cell32_gradient_mixed", call="grad", L=14.0, N=32, ecut=8.0, wells=6, nocc=8, cell=4, k=20,
              tol=1e-12),
        # frequency-dependent screening of a block: 1024 solver columns against 64 occupied states
        _case(name="slice32_block_mixed", L=16.0, N=32, ecut=5.0, wells=24, depth=-3.0, sigma=0.8, nocc=64, cell=7,
              nb=8, w_re=0.957, w_im=0.1),
        # the same at full size (38401 plane waves), two fields: 256 columns, far beyond L2
        _case(name="full64_block_mixed", L=24.0, N=64, ecut=15.0, wells=24, depth=-3.0, sigma=0.8, nocc=64, cell=2,
              nb=2, w_re=0.957, w_im=0.1),
        # many uneven cells at once, host arrays, a static and a complex frequency each
        _case(name="batch6_mixed", call="batch", L=0.0, N=0, ecut=0.0, wells=0, nocc=0, cell=13, nb=6, k=5, w_re=0.3,
              w_im=0.1, tol=1e-12),
    ]


def draw(rng):
    call = rng.choice(["eps", "eps", "eps", "chi0", "lanczos", "model", "grad"])
    N = rng.choice(SIZES)
    L = rng.uniform(6.0, 16.0)
    full = 0.5 * (2.0 * math.pi * ((N - 1) // 2) / L) ** 2          # cutoff of the largest sphere the grid holds
    room = 0.5 * (2.0 * math.pi / L * (3.0 * 3800 / (4.0 * math.pi)) ** (1.0 / 3.0)) ** 2
    ecut = min(full * rng.uniform(0.35, 0.97), room, 12.0)
    npw = 4.0 / 3.0 * math.pi * (math.sqrt(2.0 * ecut) * L / (2.0 * math.pi)) ** 3
    nocc = max(2, min(int(round(math.exp(rng.uniform(math.log(2), math.log(33))))), int(npw / 10)))
    w_re = w_im = 0.0
    if call in ("eps", "chi0") and rng.random() < 0.5:
        w_re, w_im = rng.choice([(rng.uniform(0.0, 2.0), rng.uniform(0.05, 0.3)), (0.0, rng.uniform(0.1, 1.0))])
    prec = "fp64" if call == "model" else rng.choice(["mixed", "mixed", "fp64"])
    nb = max(1, min(int(round(math.exp(rng.uniform(0.0, math.log(9))))), 512 // nocc)) if call in ("eps", "chi0") else 1
    k = rng.randint(2, 12) if call in ("lanczos", "grad") else 1
    return _case(call=call, prec=prec, L=round(L, 3), N=N, ecut=round(ecut, 3), wells=rng.randint(2, 12), nocc=nocc,
                 cell=rng.randrange(100, 10000), nb=nb, w_re=round(w_re, 4), w_im=round(w_im, 4), k=k,
                 tol=1e-12 if prec == "mixed" and call in ("lanczos", "grad") else 0.0)


def _batch_cells(case):
    """Uneven cells of the many-cell recipe (sizes from the case's cell number)."""
    rng = np.random.default_rng(case["cell"])
    out = []
    for i in range(case["nb"]):
        L = float(rng.uniform(8.0, 14.0))
        N = int(rng.choice([24, 30, 32, 36, 40, 45]))
        full = 0.5 * (2.0 * math.pi * ((N - 1) // 2) / L) ** 2
        ecut = min(full * 0.95, float(rng.uniform(4.0, 8.0)))
        out.append(_case(L=L, N=N, ecut=ecut, wells=int(rng.integers(4, 13)), nocc=int(rng.integers(4, 20)),
                         cell=1000 * case["cell"] + i))
    return out


# ---------------------------------------------------------------------------
# the cell in plain torch, FP64
# ---------------------------------------------------------------------------
class System:
    def __init__(self, L, N, ecut, wells, depth, sigma, nocc, cell, closed, attempt=0):
        self.L, self.N, self.ecut, self.vol = L, N, ecut, L ** 3
        dev = self.dev = torch.device("cuda")
        rng = np.random.Generator(np.random.PCG64(14083036 + cell + 1000 * attempt))
        centres = rng.uniform(0.0, L, size=(wells, 3))
        x = torch.arange(N, dtype=torch.float64, device=dev) * (L / N)
        V = torch.zeros((N, N, N), dtype=torch.float64, device=dev)
        for c in centres:           # the periodic images separate along the axes
            e = [sum(torch.exp(-(x - c[d] - L * m) ** 2 / (2.0 * sigma * sigma)) for m in (-1, 0, 1))
                 for d in range(3)]
            V += e[0][:, None, None] * e[1][None, :, None] * e[2][None, None, :]
        self.V = depth * V
        n = torch.fft.fftfreq(N, 1.0 / N, dtype=torch.float64, device=dev).round()
        n2 = (n[:, None, None] ** 2 + n[None, :, None] ** 2 + n[None, None, :] ** 2).reshape(-1)
        self.g2 = (2.0 * math.pi / L) ** 2
        self.idx = torch.nonzero(0.5 * self.g2 * n2 <= ecut).reshape(-1)
        self.npw = len(self.idx)
        self.kin = 0.5 * self.g2 * n2[self.idx]
        G2 = (self.g2 * n2).reshape(N, N, N)
        v = 4.0 * math.pi * (1.0 - torch.cos(torch.sqrt(G2) * 0.5 * L)) / G2.clamp(min=1e-300)
        v[0, 0, 0] = 2.0 * math.pi * (0.5 * L) ** 2
        self.sqv = torch.sqrt(v)
        self.dense = self.npw <= DENSE
        want = min(self.npw - 1, nocc + max(2, nocc // 4) + 1)
        if self.dense:
            self.e_all, self.c_all = self._diagonalise()
            e, c = self.e_all, self.c_all
        else:
            e, c = self._lowest(nocc + 1)
        lo, hi = (max(1, nocc - nocc // 4), want) if closed and self.dense else (nocc, nocc + 1)
        gaps = [float(e[m] - e[m - 1]) for m in range(lo, hi)]
        self.nocc = lo + max(range(len(gaps)), key=lambda i: gaps[i])      # the widest gap near the asked number
        self.gap = max(gaps)
        self.eps, self.C = e[:self.nocc].clone(), c[:self.nocc].clone()
        self.u = self.to_grid(self.C).real.reshape(self.nocc, -1)

    def to_grid(self, c):
        g = torch.zeros((c.shape[0], self.N ** 3), dtype=torch.complex128, device=self.dev)
        g[:, self.idx] = c
        return torch.fft.ifftn(g.view(-1, self.N, self.N, self.N), dim=(1, 2, 3), norm="forward")

    def to_sphere(self, f):
        f = f.reshape(-1, self.N, self.N, self.N).to(torch.complex128)
        return torch.fft.fftn(f, dim=(1, 2, 3), norm="forward").reshape(f.shape[0], -1)[:, self.idx]

    def H(self, c):
        return self.kin * c + self.to_sphere(self.V * self.to_grid(c))

    def sqrtv(self, f):
        f = f.reshape(-1, self.N, self.N, self.N)
        g = torch.fft.ifftn(self.sqv * torch.fft.fftn(f, dim=(1, 2, 3)), dim=(1, 2, 3)).reshape(f.shape[0], -1)
        return g if f.is_complex() else g.real

    def _diagonalise(self):
        """All eigenpairs, in the real basis cos(G r), sin(G r)."""
        N, n = self.N, self.npw
        m = torch.stack((self.idx // (N * N), self.idx // N % N, self.idx % N), 1)
        neg = (-m) % N
        order = torch.searchsorted(self.idx, (neg[:, 0] * N + neg[:, 1]) * N + neg[:, 2])
        ar = torch.arange(n, device=self.dev)
        p, z = ar[ar < order], ar[ar == order]
        q = order[p]
        vh = torch.fft.fftn(self.V.to(torch.complex128), norm="forward").reshape(-1)
        d = [(m[:, None, k] - m[None, :, k]) % N for k in range(3)]
        h = vh[(d[0] * N + d[1]) * N + d[2]]
        del d
        r2 = math.sqrt(0.5)
        cols = torch.cat((h[:, z], r2 * (h[:, p] + h[:, q]), -1j * r2 * (h[:, p] - h[:, q])), 1)
        h = torch.cat((cols[z], r2 * (cols[p] + cols[q]), 1j * r2 * (cols[p] - cols[q])), 0).real.contiguous()
        h[torch.arange(n), torch.arange(n)] += torch.cat((self.kin[z], self.kin[p], self.kin[p]))
        e, W = torch.linalg.eigh(0.5 * (h + h.T))
        W = W.T
        a, b, c = W[:, :len(z)], W[:, len(z):len(z) + len(p)], W[:, len(z) + len(p):]
        C = torch.zeros((n, n), dtype=torch.complex128, device=self.dev)
        C[:, z] = a.to(torch.complex128)
        C[:, p] = torch.complex(r2 * b, -r2 * c)
        C[:, q] = torch.complex(r2 * b, r2 * c)
        return e, C

    def _lowest(self, n, tol=2e-12):
        """The n lowest eigenpairs by a block Davidson iteration with previous directions (LOBPCG)."""
        m = n + max(8, n // 2)
        g = torch.Generator().manual_seed(5)
        X = torch.randn((m, self.npw), generator=g, dtype=torch.float64).to(self.dev).to(torch.complex128)
        T = 1.0 / (1.0 + self.kin)
        orth = lambda Y: torch.linalg.qr(Y.T)[0].T.contiguous()          # noqa: E731
        X, P, best = orth(X * T), None, None
        for _ in range(400):
            HX = self.H(X)
            e, U = np.linalg.eigh((X.conj() @ HX.T).cpu().numpy())
            U = torch.from_numpy(U).to(self.dev)
            X, HX = U.T @ X, U.T @ HX
            e = torch.from_numpy(e).to(self.dev)
            R = HX - e[:, None] * X
            res = float(R[:n].abs().pow(2).sum(1).max().sqrt())
            if best is None or res < best[0]:
                best = (res, e[:n].clone(), X[:n].clone())
            if res < tol or (best[0] < 1e-10 and res > 4.0 * best[0]):
                break
            Z = R * T if P is None else torch.cat((R * T, P))
            Z = Z / Z.abs().pow(2).sum(1, keepdim=True).sqrt().clamp(min=1e-300)
            for _ in range(2):
                Z = orth(Z - (Z @ X.conj().T) @ X)
            S = torch.cat((X, Z))
            w, U = np.linalg.eigh((S.conj() @ self.H(S).T).cpu().numpy())
            U = torch.from_numpy(np.ascontiguousarray(U[:, :m])).to(self.dev)
            P = U[m:].T @ Z
            X = orth(U.T @ S)
        # each state real in real space (V is real): c(G) -> c(G) e^{-i t/2}, t the phase of sum_G c(G) c(-G)
        C = best[2]
        q = self.to_grid(C).reshape(n, -1).pow(2).sum(1)
        return best[1], C * torch.sqrt(q / q.abs()).conj()[:, None]

    # -- response in 64 bits: sums over states (dense), or conjugate gradients for static fields
    @functools.cached_property
    def uc(self):
        c = self.c_all[self.nocc:]
        out = torch.empty((c.shape[0], self.N ** 3), dtype=torch.float64, device=self.dev)
        for i in range(0, c.shape[0], 256):
            out[i:i + 256] = self.to_grid(c[i:i + 256]).real.reshape(-1, self.N ** 3)
        return out

    def chi0(self, y, w):
        """chi0(w) y, y real [nb][N^3]."""
        out = []
        den = (self.e_all[self.nocc:, None] - self.eps[None, :]) if self.dense else None
        for f in y:
            if self.dense:
                b = self.uc @ (self.u * f).T / self.N ** 3                  # [c][v]
                s = 1.0 / (den - w) + 1.0 / (den + w)
                x = b * s
                if x.is_complex():
                    x = torch.complex(self.uc.T @ x.real, self.uc.T @ x.imag)
                else:
                    x = self.uc.T @ x
                out.append(-2.0 / self.vol * (self.u.T * x).sum(1))
            else:
                x = 2.0 * self.solve(self.to_sphere(self.u * f))
                out.append(-2.0 / self.vol * (self.u * self.to_grid(x).real.reshape(self.nocc, -1)).sum(0))
        return torch.stack(out)

    def solve(self, b):
        """(H - e_v) x_v = P_c b_v by preconditioned CG, restarted once on the true residual."""
        pc = lambda y: y - (y @ self.C.conj().T) @ self.C                   # noqa: E731
        dot = lambda a, c: (a.conj() * c).sum(1, keepdim=True).real         # noqa: E731
        A = lambda y: pc(self.H(y) - self.eps[:, None] * y)                 # noqa: E731
        t = self.kin / dot(self.C, self.kin * self.C).clamp(min=1e-3)
        num = 27 + t * (18 + t * (12 + t * 8))
        K = num / (num + 16 * t ** 4)
        b = pc(pc(b))
        b0 = dot(b, b)
        x = torch.zeros_like(b)
        for _ in range(3):
            r = b - A(x)
            p = z = pc(K * r)
            rz = dot(r, z)
            for it in range(300):
                q = A(p)
                pq = dot(p, q)
                live = (dot(r, r) > 1e-29 * b0) & (pq > 0.0)        # a converged column rests
                if it % 8 == 7 and not bool(live.any()):
                    break
                a = torch.where(live, rz / torch.where(live, pq, 1.0), 0.0)
                x = x + a * p
                r = r - a * q
                z = pc(K * r)
                new = dot(r, z)
                p = z + torch.where(live, new / torch.where(live, rz, 1.0), 0.0) * p
                rz = new
        return pc(x)

    def model(self, y):
        out = []
        pc = lambda c: c - (c @ self.C.conj().T) @ self.C                   # noqa: E731
        for f in y:
            x = pc(2.0 / (self.kin[None, :] - self.eps[:, None]) * pc(self.to_sphere(self.u * f)))
            out.append(-2.0 / self.vol * (self.u * self.to_grid(x).real.reshape(self.nocc, -1)).sum(0))
        return torch.stack(out)

    def epst(self, x, w=0.0, chi0=None):
        chi0 = chi0 or (lambda y: self.chi0(y, w))
        return x - self.sqrtv(chi0(self.sqrtv(x)))

    def epst_c(self, x, w):
        """eps~(w) on complex fields (linear: real and imaginary parts apart)."""
        return self.epst(x.real.contiguous(), w) + 1j * self.epst(x.imag.contiguous(), w)

    def lanczos(self, x0, k):
        wgt = self.vol / self.N ** 3
        Q = [x0 / math.sqrt(wgt * float(x0 @ x0))]
        al, be = [], []
        for j in range(k):
            r = self.epst(Q[j][None])[0]
            al.append(wgt * float(Q[j] @ r))
            B = torch.stack(Q)
            for _ in range(3):
                r = r - B.T @ (wgt * (B @ r))
            if j + 1 < k:
                be.append(math.sqrt(wgt * float(r @ r)))
                Q.append(r / be[-1])
        return torch.tensor(al, dtype=torch.float64), torch.tensor(be, dtype=torch.float64), torch.stack(Q)

    def lanczos_c(self, x0, k, w):
        """Complex-symmetric recursion (bilinear form, principal square roots), block size one."""
        wgt = self.vol / self.N ** 3
        x0 = x0.to(torch.complex128)
        Q = [x0 / torch.sqrt(wgt * (x0 * x0).sum())]
        al, be = [], []
        for j in range(k):
            r = self.epst_c(Q[j][None], w)[0]
            al.append(wgt * (Q[j] * r).sum())
            B = torch.stack(Q)
            for _ in range(3):
                r = r - B.T @ (wgt * (B @ r))
            if j + 1 < k:
                be.append(torch.sqrt(wgt * (r * r).sum()))
                Q.append(r / be[-1])
        return torch.stack(al), torch.stack(be) if be else torch.zeros(0, dtype=torch.complex128)

    def gradient(self, phi, k):
        """s and ds/dV_loc from k Lanczos steps (third-order perturbation theory in the eigenbasis)."""
        ng, wgt = self.N ** 3, self.vol / self.N ** 3
        a, b, Q = self.lanczos(phi, k)
        T = torch.diag(a) + (torch.diag(b, 1) + torch.diag(b, -1) if k > 1 else 0.0)
        t0 = torch.linalg.inv(T)[:, 0].to(self.dev)
        norm2 = wgt * (phi @ phi)
        s = norm2 * t0[0]
        w = self.sqrtv((torch.sqrt(norm2) * (Q.T @ t0))[None])[0]
        den = self.e_all[self.nocc:, None] - self.eps[None, :]
        d = -(self.uc @ (self.u * w).T / ng) / den                          # [c][v]
        dU = (self.uc.T @ d).T
        S = d.T @ d
        W = (self.u * w) @ self.u.T / ng
        g1 = ((dU * dU).sum(0) - ((S @ self.u) * self.u).sum(0)) / self.vol
        lam = (self.uc @ (dU * w).T / ng - d @ W) / den
        g2 = -((self.uc.T @ lam).T * self.u).sum(0) / self.vol
        return s, wgt * (4.0 * g1 + 8.0 * g2)


@functools.lru_cache(maxsize=8)
def _system(L, N, ecut, wells, depth, sigma, nocc, cell, closed):
    for attempt in range(20):
        s = System(L, N, ecut, wells, depth, sigma, nocc, cell, closed, attempt)
        if s.gap > 1e-3:         # a closed shell, as the static response needs
            return s
    raise RuntimeError("no closed shell near %d states" % nocc)


def _sys(case):
    return _system(*(case[k] for k in ("L", "N", "ecut", "wells", "depth", "sigma", "nocc", "cell", "closed")))


def _omega(case, s):
    """The frequency; a real one is moved (by less than a tenth) to the middle of a gap between transitions."""
    if case["w_im"] != 0.0 or case["w_re"] == 0.0:
        return complex(case["w_re"], case["w_im"])
    t = (s.e_all[s.nocc:, None] - s.eps[None, :]).reshape(-1).sort().values
    w = case["w_re"] * torch.linspace(0.9, 1.1, 201, dtype=torch.float64, device=t.device)
    far = (t[None, :] - w[:, None]).abs().min(1).values
    return complex(float(w[int(far.argmax())]), 0.0)


def _fields(case, s, seed):
    g = torch.Generator(device=s.dev).manual_seed(seed)
    if case["call"] == "grad":          # Gaussian test fields of width 1.5 bohr somewhere in the cell
        x = torch.arange(s.N, dtype=torch.float64, device=s.dev) * (s.L / s.N)
        c = torch.rand(3, generator=g, dtype=torch.float64, device=s.dev) * s.L
        e = [sum(torch.exp(-(x - c[d] - s.L * m) ** 2 / 4.5) for m in (-1, 0, 1)) for d in range(3)]
        return (e[0][:, None, None] * e[1][None, :, None] * e[2][None, None, :]).reshape(1, -1)
    return torch.randn((case["nb"], s.N ** 3), generator=g, dtype=torch.float64, device=s.dev)


def _host(s):
    """The occupied states as a ground-state code hands them over, kept on the host."""
    if not hasattr(s, "handed"):
        s.handed = (s.V.reshape(-1).cpu().numpy(), s.C.cpu().numpy(), s.eps.cpu().numpy())
    return s.handed


def _batch_inputs(case, seed):
    cells = [_sys(c) for c in _batch_cells(case)]
    rng = np.random.default_rng([seed, 9])
    return cells, [rng.standard_normal(s.N ** 3) for s in cells]


def prepare(case, seed):
    if case["call"] == "batch":
        cells, starts = _batch_inputs(case, seed)
        b = gw.Batch([(s.L, s.N, s.ecut, _host(s)[0]) for s in cells])
        for i, s in enumerate(cells):
            b.cell(i).set_occupied(*_host(s)[1:])
            if case["tol"]:
                b.cell(i).set_solver(tol=case["tol"])
        return dict(call="batch", batch=b, starts=starts, k=case["k"], prec=PREC[case["prec"]],
                    omegas=np.array([0.0, complex(case["w_re"], case["w_im"])]))
    s = _sys(case)
    cell = gw.Cell(s.L, s.N, s.ecut, _host(s)[0])
    cell.set_occupied(*_host(s)[1:])
    if case["tol"]:
        cell.set_solver(tol=case["tol"])
    x = _fields(case, s, seed)
    w = _omega(case, s)
    st = dict(call=case["call"], cell=cell, x=x, w=w, k=case["k"], prec=PREC[case["prec"]])
    new = lambda *shape, **kw: torch.empty(shape, device=s.dev, **{"dtype": torch.float64, **kw})   # noqa: E731
    if case["call"] in ("eps", "chi0", "model"):
        st["out"] = new(1, len(x), s.N ** 3, dtype=torch.complex128 if w.imag else torch.float64)
        if case["call"] == "model":
            cell.set_operator(gw.GW_OP_MODEL)
    elif case["call"] == "lanczos":
        k = case["k"]
        st.update(alpha=new(k), beta=new(max(k - 1, 1)), basis=new(k, s.N ** 3), inv=new(k, k))
    else:
        st.update(s=new(1), grad=new(s.N ** 3))
    return st


def run(st):
    call = st["call"]
    if call == "batch":
        A, B = st["batch"].lanczos(st["starts"], st["k"], st["omegas"], st["prec"])
        return A, B
    ctx = st["cell"].ctx
    if call in ("eps", "model"):
        return gw.gw_apply_eps(ctx, st["x"], [st["w"]], st["out"], st["prec"])
    if call == "chi0":
        return gw.gw_apply_chi0(ctx, st["x"], [st["w"]], st["out"], st["prec"])
    if call == "lanczos":
        gw.gw_lanczos(ctx, st["x"], st["k"], 0.0, st["alpha"], st["beta"], st["basis"], st["prec"])
        gw.gw_epsinv_elements(ctx, st["alpha"], st["beta"], st["k"], st["inv"])
        return st["alpha"], st["beta"][:st["k"] - 1], st["basis"], st["inv"]
    gw.gw_grad_vloc(ctx, st["x"], st["k"], st["s"], st["grad"], st["prec"])
    return st["s"], st["grad"]


def exact(case, seed):
    if case["call"] == "batch":
        cells, starts = _batch_inputs(case, seed)
        n, k = len(cells), case["k"]
        A, B = np.zeros((n, 2, k), np.complex128), np.zeros((n, 2, k - 1), np.complex128)
        for i, s in enumerate(cells):
            x = torch.from_numpy(starts[i]).to(s.dev)
            a, b, _ = s.lanczos(x, k)
            A[i, 0], B[i, 0] = a.cpu().numpy(), b.cpu().numpy()
            a, b = s.lanczos_c(x, k, complex(case["w_re"], case["w_im"]))
            A[i, 1], B[i, 1] = a.cpu().numpy(), b.cpu().numpy()
            s.__dict__.pop("uc", None)
        return A, B
    s = _sys(case)
    x, w = _fields(case, s, seed), _omega(case, s)
    w = w if w.imag else w.real
    if case["call"] in ("eps", "chi0", "model") and not s.dense and w != 0.0:
        return None              # dynamic response of a cell too large to diagonalise
    if case["call"] == "eps":
        out = s.epst(x, w)[None]
    elif case["call"] == "chi0":
        out = s.chi0(x, w)[None]
    elif case["call"] == "model":
        out = s.epst(x, chi0=s.model)[None]
    elif case["call"] == "lanczos":
        a, b, Q = s.lanczos(x[0], case["k"])
        T = torch.diag(a) + (torch.diag(b, 1) + torch.diag(b, -1) if case["k"] > 1 else 0.0)
        out = a, b, Q, torch.linalg.inv(T)
    else:
        out = s.gradient(x[0], case["k"])
    s.__dict__.pop("uc", None)
    return out


def _cost(case):
    """(bytes, flops) of the inputs and outputs and of the operator applications of one pass."""
    N3 = case["N"] ** 3
    npw = 4.0 / 3.0 * math.pi * (math.sqrt(2.0 * case["ecut"]) * case["L"] / (2.0 * math.pi)) ** 3
    nb, nocc, k = case["nb"], case["nocc"], case["k"]
    call = case["call"]
    steps = k + 2 if call == "grad" else k
    dyn = case["w_re"] != 0.0 or case["w_im"] != 0.0
    # operator applications per column: none (model), or nominal solver iterations to 1e-10
    iters = 0 if call == "model" else (50 if dyn else 30)
    cols = nocc * nb * (2 if dyn else 1)
    fft = 2.0 * 5.0 * N3 * math.log2(N3) * 0.6              # a pair of transforms, pruned to the sphere
    proj = 2.0 * 4.0 * nocc * npw * 2.0 / 2.0                # coefficients and update, real coefficients
    flops = steps * cols * ((iters + 2) * (fft + proj))
    if not dyn:
        flops *= 0.75                                        # two real columns share each complex transform
    out = {"eps": 8.0 * nb * N3, "chi0": 8.0 * nb * N3, "model": 8.0 * N3, "lanczos": 8.0 * k * N3,
           "grad": 8.0 * N3}[call] * (2 if case["w_im"] else 1)
    return 8.0 * nb * N3 + out + 16.0 * nocc * npw + 16.0 * N3, flops


def work(case):
    if case["call"] == "batch":
        b = f = 0.0
        for c in _batch_cells(case):
            for dyn in (0.0, case["w_im"]):
                x = _cost(dict(c, call="lanczos", k=case["k"], w_re=0.0, w_im=dyn))
                b, f = b + x[0], f + x[1]
        return {"bytes": b, "flops": f}
    b, f = _cost(case)
    return {"bytes": b, "flops": f}
