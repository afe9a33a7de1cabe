"""Workloads of the screening library: what a program that links it spends its time on.

Systems are seeded Gaussian-well crystals: cubic cell of side L (bohr), n^3 grid, plane waves with
|G|^2 <= ecut (bohr^-2), wells of 12 hartree and width 1 bohr, one attractive s and three repulsive
p Kleinman-Bylander projectors per atom, two occupied orbitals per atom. The occupied orbitals
are an input of the library (a ground-state code supplies them), so they are made here: a
Chebyshev-filtered subspace iteration in single precision with a double-precision Rayleigh-Ritz
step. Perturbations are orthonormal Gaussian vectors, as a PDEP start block is.

Sizes are those of the library's model systems: L = 28 n / 96 bohr and one atom per 171 bohr^3 for
the 24^3 ... 96^3 family, the 30^3, 64^3 and 96^3 systems with their own cells.

chi0bar applications and Sternheimer solves ask for 1e-10 residuals, the setting for converged
eigenpotentials: their results then agree to far better than the eigensolver's tolerance.
"""

import math

import numpy as np
import torch

from paper_2607_14025_gb300 import wdf

WELL, SIGMA, BETA_SIGMA, D_S, D_P = 12.0, 1.0, 0.8, -2.0, 5.0
TOL = 1e-10


# ------------------------------------------------------------------------------------------------
# cases


def listed():
    return [
        # one perturbation on the smallest system: a host program that probes the response one
        # vector at a time; latency of launches and host round trips
        {"name": "chi0_24_one", "kind": "chi0", "n": 24, "L": 7.0, "ecut": 25.0, "atoms": 2, "pert": 1, "form": "mixed", "learned": False},
        # a small molecule-sized cell on a 2-3-5 grid, an odd block, density response wanted too
        {"name": "chi0_30_odd", "kind": "chi0", "n": 30, "L": 11.0, "ecut": 16.0, "atoms": 3, "pert": 5, "form": "mixed_df", "learned": False},
        # the plain FP64 form that a user runs to check the mixed ones
        {"name": "chi0_36_fp64", "kind": "chi0", "n": 36, "L": 10.5, "ecut": 25.0, "atoms": 7, "pert": 4, "form": "fp64", "learned": False},
        # a mid-sized cell with the learned preconditioner: one Davidson expansion block
        {"name": "chi0_48_learned", "kind": "chi0", "n": 48, "L": 14.0, "ecut": 25.0, "atoms": 16, "pert": 24, "form": "mixed_df", "learned": True},
        # the 64^3 system (64 orbitals, 128 projectors): a block of a PDEP iteration
        {"name": "chi0_64_block", "kind": "chi0", "n": 64, "L": 20.0, "ecut": 25.0, "atoms": 32, "pert": 32, "form": "mixed_df", "learned": False},
        # the 96^3 system (256 orbitals, 512 projectors): a block of a PDEP iteration
        {"name": "chi0_96_block", "kind": "chi0", "n": 96, "L": 28.0, "ecut": 25.0, "atoms": 128, "pert": 6, "form": "mixed_df", "learned": False},
        # several uneven systems in one call, host buffers (a screening service)
        {"name": "chi0_multi", "kind": "multi", "grids": "32,45,54,72", "pert": 9, "form": "mixed_df"},
        # Sternheimer solves alone on an odd grid, right-hand sides of another perturbation theory
        {"name": "solve_75_odd", "kind": "solve", "n": 75, "L": 21.875, "ecut": 25.0, "atoms": 61, "vec": 201, "form": "mixed_df"},
        # the residual operator on a block of trial vectors: error estimates of given solutions
        {"name": "residual_96", "kind": "residual", "n": 96, "L": 28.0, "ecut": 25.0, "atoms": 128, "vec": 512, "form": "mixed_df"},
        # the same on three vectors of the 64^3 system: an iterative refinement outside the library
        {"name": "residual_64_few", "kind": "residual", "n": 64, "L": 20.0, "ecut": 25.0, "atoms": 32, "vec": 3, "form": "mixed_df"},
        # H on a block: a caller's eigensolver for empty states
        {"name": "hamiltonian_64", "kind": "hamiltonian", "n": 64, "L": 20.0, "ecut": 25.0, "atoms": 32, "vec": 48},
        # screened interaction from 64 eigenpotentials on an odd block of vectors
        {"name": "wp_64", "kind": "wp", "n": 64, "L": 20.0, "ecut": 25.0, "atoms": 32, "neig": 64, "vec": 47},
    ]


GRIDS = (24, 25, 27, 30, 32, 36, 40, 45, 48, 50, 54, 60, 64, 72, 75, 80, 96)


def draw(rng):
    """One more case: grids of the family from 24^3 to 96^3, blocks from one vector to as many as
    cost no more than the largest listed case."""

    def log_int(lo, hi):
        return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(max(lo, hi))))))))

    kind = rng.choice(["chi0", "chi0", "chi0", "chi0", "multi", "solve", "residual", "residual", "hamiltonian", "wp"])
    if kind == "multi":
        grids = rng.sample([g for g in GRIDS if 30 <= g <= 72], rng.randint(2, 4))
        return {"kind": "multi", "grids": ",".join(str(g) for g in grids), "pert": rng.randint(2, 9), "form": rng.choice(["mixed", "mixed_df", "mixed_df"])}
    form = "fp64" if rng.random() < 0.1 else ("mixed" if rng.random() < 0.2 else "mixed_df")
    heavy = form == "fp64" or (kind in ("chi0", "solve") and form == "mixed")
    n = rng.choice([g for g in GRIDS if g <= (48 if heavy else 96)])
    L = 28.0 * n / 96.0
    atoms = max(2, int(round(L ** 3 / 171.0 * rng.uniform(0.3, 1.0))))
    case = {"kind": kind, "n": n, "L": L, "ecut": 25.0, "atoms": atoms}
    # solves (or vectors) up to the largest listed work at this grid and number of orbitals
    scale = (96.0 / n) ** 3
    if kind == "chi0":
        most = int(min(1536 * scale / (2 * atoms), 8192 / (2 * atoms), 64)) // (8 if heavy else 1)
        case.update(pert=log_int(1, max(1, most)), form=form, learned=form == "mixed_df" and rng.random() < 0.3)
    elif kind == "solve":
        most = int(min(1024 * scale, 4096)) // (8 if heavy else 1)
        case.update(vec=log_int(1, most), form=form)
    elif kind == "residual":
        case.update(vec=log_int(1, int(min(512 * scale, 4096)) // (8 if form != "mixed_df" else 1)), form=form)
    elif kind == "hamiltonian":
        case.update(vec=log_int(1, int(min(64 * scale, 512))))
    else:
        case.update(neig=log_int(4, 128), vec=log_int(1, 256))
    return case


# ------------------------------------------------------------------------------------------------
# model systems


def _half_sphere(L, ecut):
    """Miller indices of the Gamma half sphere, G = 0 first."""
    t = int(math.floor(ecut * (L / (2.0 * math.pi)) ** 2 + 1e-9))
    m = math.isqrt(t)
    r = np.arange(-m, m + 1)
    a, b, c = (v.ravel() for v in np.meshgrid(r, r, r, indexing="ij"))
    nn = a * a + b * b + c * c
    keep = (nn <= t) & ((c > 0) | ((c == 0) & (b > 0)) | ((c == 0) & (b == 0) & (a >= 0)))
    a, b, c, nn = a[keep], b[keep], c[keep], nn[keep]
    o = np.lexsort((c, b, a, nn))
    return np.stack([a[o], b[o], c[o]], axis=1).astype(np.int32)


def _place(L, natom, rng):
    """Random positions, any two at least dist apart (minimum image); dist shrinks if they do not fit."""
    dist, pos, tries = 5.0, np.zeros((0, 3)), 0
    while len(pos) < natom:
        x = rng.random(3) * L
        d = x - pos
        d -= L * np.round(d / L)
        if len(pos) == 0 or (d * d).sum(1).min() >= dist * dist:
            pos = np.concatenate([pos, x[None]])
            tries = 0
        tries += 1
        if tries > 400:
            dist, pos, tries = dist * 0.97, np.zeros((0, 3)), 0
    return pos


class _System:
    """Arrays of a model system on the GPU, in the layout that wdf.Context takes."""

    def __init__(self, n, L, ecut, natom, rng, dev):
        self.grid, self.cell, self.L, self.omega = (n, n, n), np.eye(3) * L, L, L ** 3
        self.miller = _half_sphere(L, ecut)
        self.m = len(self.miller)
        atoms = torch.from_numpy(_place(L, natom, rng)).to(dev)
        mil = torch.from_numpy(self.miller.astype(np.int64)).to(dev)
        g = mil.double() * (2.0 * math.pi / L)
        self.g2 = (g * g).sum(1)
        self.nocc = 2 * natom
        # wells: separable Gaussians over the atoms and their lattice images
        x = torch.arange(n, device=dev, dtype=torch.float64) * (L / n)
        im = torch.arange(-4, 5, device=dev, dtype=torch.float64) * L
        e = torch.exp(-((x[None, None, :, None] - atoms.T[:, :, None, None] + im) ** 2) / (2.0 * SIGMA ** 2)).sum(-1)
        self.vloc_r = (-WELL * torch.einsum("az,ay,ax->zyx", e[2], e[1], e[0])).contiguous()
        radial = torch.exp(-0.5 * self.g2 * BETA_SIGMA ** 2)[None] * torch.exp(-1j * (atoms @ g.T))
        rows = torch.stack([radial] + [-1j * g[:, a][None] * radial for a in range(3)], dim=1).reshape(4 * natom, self.m)
        nrm = (rows[:, 0].abs() ** 2 + 2.0 * (rows[:, 1:].abs() ** 2).sum(1)).sqrt()
        self.beta = (rows / nrm[:, None]).contiguous()
        self.dij = np.tile(np.array([D_S, D_P, D_P, D_P]), natom)
        # flat indices of the half sphere in an (n3 // 2 + 1, n2, n1) array, and the mirrors of n3 = 0
        self.h3 = n // 2 + 1
        self.idx = (mil[:, 2] * n + mil[:, 1] % n) * n + mil[:, 0] % n
        self.flat = torch.nonzero((mil[:, 2] == 0) & (self.g2 > 0)).ravel()
        f = mil[self.flat]
        self.idm = ((-f[:, 1]) % n) * n + (-f[:, 0]) % n
        self.dev = dev

    # real coordinates [c0, sqrt2 Re c, sqrt2 Im c]: Gamma inner products become plain ones
    def pack(self, c):
        s = math.sqrt(2.0)
        return torch.cat([c[:, :1].real, s * c[:, 1:].real, s * c[:, 1:].imag], dim=1)

    def unpack(self, q):
        r = math.sqrt(0.5)
        c = torch.complex(r * q[:, 1:self.m], r * q[:, self.m:])
        return torch.cat([torch.complex(q[:, :1], torch.zeros_like(q[:, :1])), c], dim=1)

    def to_grid(self, c):
        """Real fields sum_G c(G) exp(iGr) of half-sphere rows."""
        n = self.grid[0]
        F = torch.zeros((c.shape[0], self.h3 * n * n), dtype=c.dtype, device=self.dev)
        F[:, self.idx] = c
        F[:, self.idm] = c[:, self.flat].conj()
        return torch.fft.irfftn(F.view(-1, self.h3, n, n), s=(n, n, n), dim=(-1, -2, -3), norm="forward")

    def to_sphere(self, f):
        F = torch.fft.rfftn(f, dim=(-1, -2, -3), norm="forward")
        return F.reshape(f.shape[0], -1)[:, self.idx]

    def work(self, dtype):
        """The operator's tables in one precision: kinetic energies, potential, projectors."""
        rt = torch.float32 if dtype == torch.complex64 else torch.float64
        t = 0.5 * self.g2
        return {"kin": torch.cat([t, t[1:]]).to(rt), "v": self.vloc_r.to(rt), "b": self.pack(self.beta).to(rt),
                "d": torch.from_numpy(self.dij).to(self.dev).to(rt), "c": dtype}

    def ham(self, q, w, block=256):
        """H on packed rows, a block of rows at a time."""
        out = w["kin"] * q
        for i in range(0, q.shape[0], block):
            c = self.unpack(q[i:i + block])
            out[i:i + block] += self.pack(self.to_sphere(self.to_grid(c) * w["v"]))
        return out + ((q @ w["b"].T) * w["d"]) @ w["b"]

    def ground_state(self, gen):
        """Occupied orbitals and eigenvalues: Chebyshev-filtered subspace iteration."""
        nb = self.nocc + max(6, self.nocc // 8)
        w32, w64 = self.work(torch.complex64), self.work(torch.complex128)
        q = torch.randn((nb, 2 * self.m - 1), generator=gen, device=self.dev, dtype=torch.float32)
        q = q / (1.0 + w32["kin"]) ** 2
        top = float(0.5 * self.g2.max()) + 8.0
        for it in range(7):
            q = _orthonormal(q.double())
            h = q @ self.ham(q.float(), w32).double().T
            e, u = np.linalg.eigh((0.5 * (h + h.T)).cpu().numpy())
            q = (torch.from_numpy(np.ascontiguousarray(u.T)).to(self.dev) @ q).float()
            lo = float(e[-1])  # damp [lo, top], amplify below
            c, half = 0.5 * (top + lo), 0.5 * (top - lo)
            y0, y1 = q, (self.ham(q, w32) - c * q) / half
            for _ in range(14):
                y0, y1 = y1, 2.0 * (self.ham(y1, w32) - c * y1) / half - y0
                s = y1.abs().amax(dim=1, keepdim=True)
                y0, y1 = y0 / s, y1 / s
            q = y1
        q = _orthonormal(q.double())
        h = q @ self.ham(q, w64).T
        e, u = np.linalg.eigh((0.5 * (h + h.T)).cpu().numpy())
        q = torch.from_numpy(np.ascontiguousarray(u.T)).to(self.dev) @ q
        self.eps = e[:self.nocc].copy()
        self.q = _orthonormal(q[:self.nocc])
        self.psi = self.unpack(self.q).contiguous()


def _orthonormal(q):
    """Rows with the same span (Cholesky, twice)."""
    for _ in range(2):
        q = torch.linalg.solve_triangular(torch.linalg.cholesky(q @ q.T), q, upper=False)
    return q


def _system(n, L, ecut, natom, seed, orbitals=True):
    dev = torch.device("cuda")
    rng = np.random.default_rng([seed, n, natom])
    gen = torch.Generator(device=dev)
    gen.manual_seed(seed * 1009 + 7)
    s = _System(n, L, ecut, natom, rng, dev)
    if orbitals:
        s.ground_state(gen)
    else:  # the operator alone: an orthonormal occupied space, levels of the family's spread
        s.q = _orthonormal(torch.randn((s.nocc, 2 * s.m - 1), generator=gen, device=dev, dtype=torch.float64) / (1.0 + s.work(torch.complex128)["kin"]) ** 2)
        s.psi, s.eps = s.unpack(s.q).contiguous(), np.linspace(-7.0, -2.5, s.nocc)
    return s, gen


def _vectors(s, count, gen, g0):
    """Orthonormal Gaussian half-sphere vectors (without G = 0 unless g0)."""
    q = torch.randn((count, 2 * s.m - 1), generator=gen, device=s.dev, dtype=torch.float64)
    if not g0:
        q[:, 0] = 0.0
    return s.unpack(_orthonormal(q)).contiguous()


def _atoms_of(n):
    return max(4, int(round((28.0 * n / 96.0) ** 3 / 171.0)))


def _inputs(case, seed):
    """Systems and vectors of a case (exact() and prepare() start from the same)."""
    kind = case["kind"]
    if kind == "multi":
        out = []
        for k, n in enumerate(int(v) for v in case["grids"].split(",")):
            s, gen = _system(n, 28.0 * n / 96.0, 25.0, _atoms_of(n), seed + 100003 * (k + 1))
            out.append((s, _vectors(s, case["pert"], gen, False)))
        return out
    s, gen = _system(case["n"], case["L"], case["ecut"], case["atoms"], seed, orbitals=kind in ("chi0", "solve"))
    if kind == "chi0":
        return [(s, _vectors(s, case["pert"], gen, False))]
    if kind == "wp":
        return [(s, _vectors(s, case["neig"], gen, False), _vectors(s, case["vec"], gen, False))]
    x = _vectors(s, case["vec"], gen, True)
    if kind == "solve":  # smooth sources without an occupied component
        q = s.pack(x) / (1.0 + 0.25 * s.work(torch.complex128)["kin"])
        x = s.unpack(q - (q @ s.q.T) @ s.q).contiguous()
    return [(s, x)]


def _vidx(s, count):
    return (np.arange(count) * 7 % s.nocc).astype(np.int32)


def _lambda(neig):
    return -4.0 * np.exp(-np.arange(neig) / 12.0)


# ------------------------------------------------------------------------------------------------
# what a user's program does


def prepare(case, seed):
    kind = case["kind"]
    ins = _inputs(case, seed)
    state = {"case": dict(case), "ctx": []}
    for t in ins:
        s = t[0]
        state["ctx"].append(wdf.Context(s, psi=s.psi, eps=s.eps, precision=case.get("form", "mixed"), cg_tol=TOL))
    s, x = ins[0][0], ins[0][-1]
    if kind == "multi":
        state["x"] = [t[1].cpu().numpy() for t in ins]
    else:
        state["x"] = x
    state["vidx"] = _vidx(s, x.shape[0])
    if kind == "wp":
        state["phibar"], state["lam"] = ins[0][1], _lambda(case["neig"])
    if case.get("learned"):  # trained on solves of another, small system, as a service would keep it
        d, _ = _system(24, 7.0, 25.0, 2, 12345)
        donor = wdf.Context(d, psi=d.psi, eps=d.eps, precision="mixed_df", cg_tol=1e-8)
        model, _ = wdf.train_preconditioner([donor], npert=4, steps=100, seed=5)
        state["ctx"][0].set_model(model)
        model.close()
        donor.close()
    return state


def run(state):
    case, ctx = state["case"], state["ctx"]
    kind = case["kind"]
    if kind == "multi":
        return wdf.apply_chi0_multi(ctx, state["x"])[0]
    if kind == "chi0":
        out, drho, _ = ctx[0].apply_chi0(state["x"], want_drho=case["pert"] % 2 == 1)
        return [out] if drho is None else [out, drho]
    if kind == "solve":
        return ctx[0].sternheimer(state["vidx"], state["x"])[0]
    if kind == "residual":
        return ctx[0].apply_sternheimer_operator(state["vidx"], state["x"])
    if kind == "hamiltonian":
        return ctx[0].apply_hamiltonian(state["x"])
    return ctx[0].apply_wp(state["lam"], state["phibar"], state["x"])


# ------------------------------------------------------------------------------------------------
# what a pass cannot do without


def _sizes(n, L, ecut):
    m = len(_half_sphere(L, ecut))
    xm = math.isqrt(int(math.floor(ecut * (L / (2.0 * math.pi)) ** 2 + 1e-9)))
    return m, 2 * xm + 1


def _op_flops(n, L, ecut, rows):
    """One operator application per vector: transforms of the occupied columns (two vectors per
    complex transform), the local product, projections on `rows` vectors."""
    m, nx = _sizes(n, L, ecut)
    line = 5.0 * n * math.log2(n)
    disk = math.pi / 4.0 * nx * nx
    fft = 2.0 * line * (disk + n * nx + n * n) / 2.0
    return fft + n ** 3 + 8.0 * rows * m


def work(case):
    """Bytes: inputs read and outputs written once (the system's projectors, orbitals and potential
    among the inputs). Operations: the least number of operator applications that conjugate
    gradients need (25 for these systems at 1e-10), one residual, right-hand sides and density."""
    kind = case["kind"]
    if kind == "multi":
        parts = [dict(kind="chi0", n=n, L=28.0 * n / 96.0, ecut=25.0, atoms=_atoms_of(n), pert=case["pert"])
                 for n in (int(v) for v in case["grids"].split(","))]
        w = [work(p) for p in parts]
        return {"bytes": sum(v["bytes"] for v in w), "flops": sum(v["flops"] for v in w)}
    n, L, ecut, atoms = case["n"], case["L"], case["ecut"], case["atoms"]
    m, _ = _sizes(n, L, ecut)
    system = 16.0 * m * 6 * atoms + 8.0 * n ** 3
    rows = 6 * atoms
    if kind == "chi0":
        ns = 2 * atoms * case["pert"]
        return {"bytes": system + 32.0 * m * case["pert"], "flops": ns * 28.0 * _op_flops(n, L, ecut, rows)}
    if kind == "solve":
        return {"bytes": system + 32.0 * m * case["vec"], "flops": case["vec"] * 26.0 * _op_flops(n, L, ecut, rows)}
    if kind == "residual":
        return {"bytes": system + 32.0 * m * case["vec"], "flops": case["vec"] * _op_flops(n, L, ecut, rows)}
    if kind == "hamiltonian":
        return {"bytes": 16.0 * m * 4 * atoms + 8.0 * n ** 3 + 32.0 * m * case["vec"], "flops": case["vec"] * _op_flops(n, L, ecut, 4 * atoms)}
    return {"bytes": 16.0 * m * case["neig"] + 32.0 * m * case["vec"], "flops": 8.0 * m * case["neig"] * case["vec"]}


# ------------------------------------------------------------------------------------------------
# the same results in 64 bits by plain torch


class _Operator:
    """A_v = H - eps_v + alpha P on packed rows, in one precision."""

    def __init__(self, s, dtype):
        self.s, self.w = s, s.work(dtype)
        rt = self.w["kin"].dtype
        self.p = s.q.to(rt)
        self.eps = torch.from_numpy(s.eps).to(s.dev).to(rt)
        self.alpha = float(s.eps.max() - s.eps.min() + 1.0)
        # Teter-Payne-Allan preconditioner of each orbital
        x = s.work(torch.complex128)["kin"][None] / ((s.q * s.q) @ s.work(torch.complex128)["kin"]).clamp_min(1e-3)[:, None]
        t = 27.0 + x * (18.0 + x * (12.0 + 8.0 * x))
        self.k = (t / (t + 16.0 * x ** 4)).to(rt)

    def __call__(self, q, v):
        return self.s.ham(q, self.w) - self.eps[v][:, None] * q + self.alpha * ((q @ self.p.T) @ self.p)

    def solve(self, b, v, tol):
        """Preconditioned conjugate gradients to tol on every row."""
        x, r = torch.zeros_like(b), b.clone()
        z = self.k[v] * r
        p, rz = z, (r * z).sum(1)
        stop = tol * b.norm(dim=1)
        for _ in range(400):
            ap = self(p, v)
            a = rz / (p * ap).sum(1).clamp_min(1e-300 if b.dtype == torch.float64 else 1e-36)
            x, r = x + a[:, None] * p, r - a[:, None] * ap
            if bool((r.norm(dim=1) <= stop).all()):
                break
            z = self.k[v] * r
            new = (r * z).sum(1)
            p, rz = z + (new / rz.clamp_min(1e-300 if b.dtype == torch.float64 else 1e-36))[:, None] * p, new
        return x


def _solve_exact(s, b, v):
    """A_v x = b with double-precision residuals and single-precision corrections."""
    hi, lo = _Operator(s, torch.complex128), _Operator(s, torch.complex64)
    x, nb = torch.zeros_like(b), b.norm(dim=1).clamp_min(1e-300)
    r = b
    for _ in range(8):
        scale = r.norm(dim=1, keepdim=True).clamp_min(1e-300)
        x = x + scale * lo.solve((r / scale).float(), v, 1e-4).double()
        r = b - hi(x, v)
        if float((r.norm(dim=1) / nb).max()) < 1e-13:
            break
    return x


def _chi0_exact(s, phi):
    nocc, npert = s.nocc, phi.shape[0]
    half = torch.where(s.g2 > 0, math.sqrt(4.0 * math.pi) / s.g2.clamp_min(1e-30).sqrt(), torch.zeros_like(s.g2))
    psi_r = s.to_grid(s.psi)
    out = []
    per = max(1, 2048 // nocc)  # perturbations solved together
    for p0 in range(0, npert, per):
        x = phi[p0:p0 + per] * half
        k = x.shape[0]
        b = torch.cat([s.pack(s.to_sphere(d[None] * psi_r)) for d in s.to_grid(x)])
        b = (b @ s.q.T) @ s.q - b
        v = torch.arange(nocc, device=s.dev).repeat(k)
        d = _solve_exact(s, b, v)
        rho = torch.stack([(psi_r * s.to_grid(s.unpack(d[i * nocc:(i + 1) * nocc]))).sum(0) for i in range(k)])
        out.append((4.0 / s.omega) * s.to_sphere(rho))
    rho = torch.cat(out)
    return rho * half, rho


def exact(case, seed):
    kind = case["kind"]
    ins = _inputs(case, seed)
    if kind == "multi":
        return [_chi0_exact(s, x)[0].cpu().numpy() for s, x in ins]
    s, x = ins[0][0], ins[0][-1]
    if kind == "chi0":
        out, rho = _chi0_exact(s, x)
        return [out] if case["pert"] % 2 == 0 else [out, rho]
    if kind == "hamiltonian":
        return s.unpack(s.ham(s.pack(x), s.work(torch.complex128)))
    if kind == "wp":
        half = torch.where(s.g2 > 0, math.sqrt(4.0 * math.pi) / s.g2.clamp_min(1e-30).sqrt(), torch.zeros_like(s.g2))
        f, y = s.pack(ins[0][1]), s.pack(x * half)
        lam = torch.from_numpy(_lambda(case["neig"])).to(s.dev)
        return s.unpack(((y @ f.T) * (lam / (1.0 - lam))) @ f) * half
    v = torch.from_numpy(_vidx(s, x.shape[0]).astype(np.int64)).to(s.dev)
    if kind == "residual":
        return s.unpack(_Operator(s, torch.complex128)(s.pack(x), v))
    return s.unpack(_solve_exact(s, s.pack(x), v))
