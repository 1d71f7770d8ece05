"""Performance cases of the ParO plane-wave library: the work a program has it do, through its public
entry points (paro.Context, paro.Batch, paro.hpsi).

The cells are the diamond-lattice supercells of the library's own workloads (8, 64 and 512 atoms and the
216 atoms between them, a = 9.8 .. 10.8 Bohr per conventional cell, cutoffs 8 .. 15 Ha, displaced by
+-0.05 Bohr), with the same pseudopotential forms. Orbitals are random with the decay over |k+G|^2 that
Kohn-Sham orbitals have, so the kinetic energies and the convergence of the inner solves are realistic.

  apply    H psi of a block of orbitals: the call every other step is made of
  solve    the source problems of a block of orbitals (preconditioned CG, the default 0.25 / 8 steps)
  orth     Cholesky orthonormalisation of a block of rows (n_bands, or 2 n_bands for Algorithm 2)
  adjoint  forward and backward of paro.hpsi: H psi and its gradients by orbitals, potential and positions
  batch    H psi of every k-point of a mesh, or of many uneven cells, in one batched call
  scf      one SCF iteration of a whole cell (Algorithm 1), the library's headline call

Each path runs in FP64 and in the mixed-precision (FP32) form. `exact` computes the same outputs in plain
torch, complex128, with none of the library's code.
"""
from __future__ import annotations

import math

import numpy as np
import torch

PP = dict(Z=4.0, rc=0.8, A=2.0, a=1.0)  # local pseudopotential -Z erf(r/rc)/r + A exp(-(r/a)^2)
KB_RC = 1.2                             # radius of the s and p projectors, four per atom
KT = 0.002                              # smearing of the SCF cells (Ha)
INNER_TOL, INNER_IT = 0.25, 8           # the library's default stopping rule of the inner solves
BETA_MIX = 0.7                          # its default mixing parameter
A0 = 10.26                              # Bohr, conventional cell of the configurations


def _case(name, path, n_rep, ecut, nb, dtype, kb=True, a=A0, **more):
    return dict(name=name, path=path, n_rep=n_rep, a=a, ecut=ecut, nb=nb, dtype=dtype, kb=kb, **more)


def listed():
    return [
        # one vector of the smallest cell, as a Lanczos or line-search step applies H: launch latency counts
        _case("apply_f64_8at_1band", "apply", 1, 10.0, 1, "f64", kb=False),
        # a small cell's block with an odd band count, a ragged cell and the high end of the cutoffs
        _case("apply_f32_8at_odd", "apply", 1, 14.0, 23, "f32", a=10.61),
        # the ordinary block: all orbitals of the 64-atom cell, as the Rayleigh-Ritz step applies H to them
        _case("apply_f32_64at", "apply", 2, 15.0, 144, "f32"),
        _case("apply_f64_64at", "apply", 2, 15.0, 144, "f64"),
        # the same cell at another cutoff (another FFT grid), an odd band count
        _case("apply_f32_64at_grid64", "apply", 2, 11.0, 133, "f32"),
        # all orbitals of the 512-atom cell
        _case("apply_f32_512at", "apply", 4, 12.0, 1088, "f32"),
        # step 3 of the iteration for a caller that drives it itself
        _case("solve_f64_8at", "solve", 1, 10.0, 20, "f64"),
        # the doubled basis of Algorithm 2 on the 64-atom cell
        _case("orth_f64_64at", "orth", 2, 15.0, 288, "f64"),
        # gradients by orbitals, potential and positions (FP32 training)
        _case("adjoint_f32_64at", "adjoint", 2, 15.0, 144, "f32"),
        # the 27 k-points of a 3x3x3 mesh of the 8-atom cell
        _case("batch_f32_mesh27", "batch", 1, 10.0, 20, "f32", kb=False, q=3, cells=0),
        # whole SCF iterations of the 64-atom cell, both precisions: the headline workload and its FP64 form
        _case("scf_f32_64at", "scf", 2, 15.0, 144, "f32", n_occ=128),
        _case("scf_f64_64at", "scf", 2, 15.0, 144, "f64", n_occ=128),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    path = rng.choice(["apply", "apply", "apply", "solve", "orth", "adjoint", "batch", "scf"])
    dtype = rng.choice(["f32", "f64"])
    a = round(rng.uniform(9.8, 10.8), 3)
    ecut = round(rng.uniform(8.0, 15.0), 2)
    if path == "apply":
        n_rep = rng.choice([1, 2, 2, 3])
        if n_rep == 3:  # FP64 planes of the larger grids exceed the library's limit
            ecut = round(rng.uniform(8.0, 12.0), 2)
        return _case("", path, n_rep, ecut, _log_int(rng, 1, 18 * n_rep ** 3), dtype, rng.random() < 0.8, a)
    if path == "solve":
        n_rep = rng.choice([1, 2])
        return _case("", path, n_rep, ecut, _log_int(rng, 4, 18 * n_rep ** 3), dtype, rng.random() < 0.8, a)
    if path == "orth":
        n_rep = rng.choice([1, 2])
        return _case("", path, n_rep, ecut, _log_int(rng, 2, 36 * n_rep ** 3), dtype, False, a)
    if path == "adjoint":
        n_rep = rng.choice([1, 2])
        return _case("", path, n_rep, ecut, _log_int(rng, 4, 18 * n_rep ** 3), dtype, True, a)
    if path == "batch":
        ecut = round(rng.uniform(8.0, 14.0), 2)
        if rng.random() < 0.5:
            return _case("", path, 1, ecut, rng.randint(12, 24), dtype, False, a, q=rng.choice([2, 3]), cells=0)
        return _case("", path, 1, ecut, rng.randint(12, 24), dtype, False, a, q=1, cells=rng.randint(3, 24))
    n_occ = rng.randint(12, 16)
    ecut = round(rng.uniform(8.0, 14.0), 2)
    return _case("", path, 1, ecut, n_occ + rng.randint(4, 8), dtype, True, a, n_occ=n_occ)


# ---- geometry and inputs --------------------------------------------------------------------------
_FCC = np.array([[0.0, 0.0, 0.0], [0.0, 0.5, 0.5], [0.5, 0.0, 0.5], [0.5, 0.5, 0.0]])


def _cell(n_rep, a, seed):
    """Lattice, displaced positions, one projector strength per (atom, l)."""
    rng = np.random.default_rng(seed)
    lat = np.eye(3) * (a * n_rep)
    corner = np.array([[i, j, k] for i in range(n_rep) for j in range(n_rep) for k in range(n_rep)], dtype=float)
    frac = (corner[:, None, :] + np.concatenate([_FCC, _FCC + 0.25])[None]).reshape(-1, 3) / n_rep
    pos = frac @ lat + rng.uniform(-0.05, 0.05, size=(len(frac), 3))
    return lat, np.ascontiguousarray(pos), rng.uniform(-1.0, 1.0, size=(len(frac), 2))


def _problems(case, seed):
    """(lattice, positions, strengths, cutoff, k-points) of every cell of the case."""
    if case["path"] != "batch" or not case["cells"]:
        k = np.zeros((1, 3))
        if case["path"] == "batch":
            q = case["q"]
            r = (2.0 * np.arange(1, q + 1) - q - 1) / (2.0 * q)
            k = np.array([[x, y, z] for x in r for y in r for z in r])
        return [_cell(case["n_rep"], case["a"], seed) + (case["ecut"], k)]
    rng = np.random.default_rng(1000 + int(case["ecut"] * 100))  # uneven cells: sizes belong to the case
    out = []
    for i in range(case["cells"]):
        a, e = case["a"] * rng.uniform(0.97, 1.03), case["ecut"] * rng.uniform(0.85, 1.15)
        out.append(_cell(case["n_rep"], a, seed * 64 + i) + (e, np.zeros((1, 3))))
    return out


def _sphere(lat, ecut, kfrac=(0.0, 0.0, 0.0)):
    """Miller indices with |k+G|^2/2 <= ecut in lexicographic order, k+G, kinetic energies."""
    b = 2 * math.pi * np.linalg.inv(lat).T
    lim = [int(math.sqrt(2 * ecut) * np.linalg.norm(lat[i]) / (2 * math.pi) + abs(kfrac[i])) + 1 for i in range(3)]
    n = np.stack(np.meshgrid(*[np.arange(-m, m + 1) for m in lim], indexing="ij"), axis=-1).reshape(-1, 3)
    g = (n + np.asarray(kfrac)) @ b
    kin = 0.5 * np.sum(g * g, axis=1)
    keep = kin <= ecut
    return n[keep], g[keep], kin[keep]


def _rows(n, kin, seed, dtype):
    """n random rows with the decay of Kohn-Sham orbitals over the kinetic energy, each of norm one."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    amp = torch.as_tensor(1.0 / (1.0 + np.asarray(kin) ** 2), device="cuda")
    out = torch.empty((n, len(kin)), dtype=torch.complex128 if dtype == "f64" else torch.complex64, device="cuda")
    for i in range(0, n, 64):
        m = min(64, n - i)
        r = torch.randn((m, len(kin), 2), generator=g, device="cuda", dtype=torch.float64)
        z = torch.view_as_complex(r) * amp
        out[i:i + m] = z / torch.linalg.vector_norm(z, dim=1, keepdim=True)
    return out


def _levels(rows, kin):
    """Eigenvalue estimates of the rows: their kinetic energy and a mean potential."""
    return ((rows.abs().double() ** 2 @ torch.as_tensor(kin, device="cuda")) - 0.4).cpu().numpy()


def _v_rest(grid, seed, dtype):
    """A smooth Hartree- and exchange-like part of the potential."""
    x = [2 * math.pi * torch.arange(n, device="cuda", dtype=torch.float64) / n for n in grid]
    p = np.random.default_rng(seed + 7).uniform(0, 2 * math.pi, 3)
    v = 0.3 * (torch.cos(x[0] + p[0])[:, None, None] + torch.sin(x[1] + p[1])[None, :, None]
               + torch.cos(2 * x[2] + p[2])[None, None, :]) - 0.2
    return v.to(torch.float64 if dtype == "f64" else torch.float32).contiguous()


def _real(case):
    return torch.float64 if case["dtype"] == "f64" else torch.float32


def prepare(case, seed):
    from paper_1702_04045_gb300 import paro
    ctxs, rows = [], []
    n_occ = case.get("n_occ", case["nb"])
    for lat, pos, d, ecut, kpts in _problems(case, seed):
        bases = [_sphere(lat, ecut, k) for k in kpts]
        ctx = paro.Context(lat, pos, ecut, case["nb"], n_occ, "fp64" if case["dtype"] == "f64" else "mixed",
                           kpts=kpts)
        ctx.set_local_pp(**PP)
        if case["kb"]:
            ctx.set_kb(KB_RC, d)
        ctxs.append(ctx)
        rows += [_rows(case["nb"], kin, seed * 100 + len(rows) + i, case["dtype"])
                 for i, (_, _, kin) in enumerate(bases)]
    s = dict(case=case, ctx=ctxs[0], psi=rows[0])
    if case["path"] == "solve":
        s["eps"] = _levels(rows[0], bases[0][2])
    elif case["path"] == "adjoint":
        s["psi"] = rows[0].requires_grad_(True)
        s["v"] = _v_rest(ctxs[0].grid, seed, case["dtype"]).requires_grad_(True)
        s["pos"] = torch.as_tensor(pos, device="cuda").to(_real(case)).requires_grad_(True)
        s["w"] = _rows(case["nb"], bases[0][2], seed * 100 + 50, case["dtype"])
    elif case["path"] == "batch":
        s["batch"], s["psi"] = paro.Batch(ctxs), rows
    elif case["path"] == "scf":
        ctxs[0].set_smearing(KT)
        ctxs[0].set_orbitals(rows[0])
        del s["psi"]
    return s


def run(s):
    case, ctx = s["case"], s["ctx"]
    if case["path"] == "apply":
        return ctx.apply_h(s["psi"])
    if case["path"] == "solve":
        x, its = ctx.solve_source(s["eps"], s["psi"], INNER_TOL, INNER_IT)
        return dict(x=x, its=its)
    if case["path"] == "orth":
        return ctx.orthonormalize(s["psi"])
    if case["path"] == "adjoint":
        from paper_1702_04045_gb300 import paro
        y = paro.hpsi(ctx, s["psi"], s["v"], s["pos"])
        g_psi, g_v, g_pos = torch.autograd.grad(y, (s["psi"], s["v"], s["pos"]), s["w"])
        return dict(y=y.detach(), g_psi=g_psi, g_v=g_v, g_pos=g_pos)
    if case["path"] == "batch":
        return s["batch"].apply_h(s["psi"])
    # scf: each pass continues the iteration. The mixed-precision iteration holds its orbitals in FP32, and a
    # program that keeps its results keeps them in that type; its orbitals of close levels are fixed only up to
    # a rotation among themselves at that precision, so their state is read as the density they form.
    terms, resid = ctx.scf_step()
    t = _real(case)
    out = dict(energy=torch.tensor([terms[k] for k in sorted(terms)], dtype=torch.float64).to(t),
               resid=torch.tensor(resid, dtype=torch.float64).to(t), eps=torch.from_numpy(ctx.eigenvalues()).to(t),
               rho=ctx.density().to(t))
    if case["dtype"] == "f64":
        out["psi"] = ctx.get_orbitals(device=True)
    return out


# ---- what a pass cannot do without ----------------------------------------------------------------
def _smooth(m):
    x = m + 1
    while True:
        y = x
        for p in (2, 3):
            while y % p == 0:
                y //= p
        if y == 1:
            return x
        x += 1


def work(case):
    """Bytes: the orbitals in and out, the potential and the projectors once. Operations: the stick-pruned
    FFTs (5 n log2 n a line, both directions), the potential, the projector and subspace products."""
    n_cells = case.get("cells", 0) or 1
    n_k = case.get("q", 1) ** 3
    length = case["a"] * case["n_rep"]
    r = math.sqrt(2 * case["ecut"]) * length / (2 * math.pi)  # radius of the sphere in Miller indices
    n = _smooth(int(2 * r) + 2 * int(r))
    npw, ncol, nrow = 4 / 3 * math.pi * r ** 3, math.pi * r * r, 2 * int(r) + 1
    nb, e = case["nb"], 16 if case["dtype"] == "f64" else 8
    nproj = 32 * case["n_rep"] ** 3 if case["kb"] else 0
    line = 5 * n * math.log2(n)
    fft = 2 * line * (ncol + n * nrow + n * n) + 2 * n ** 3
    table = n ** 3 * e / 2 + nproj * npw * e
    h_flops = nb * (fft + 16 * nproj * npw + 4 * npw)
    h_bytes = 2 * nb * npw * e + table
    gram = 4 * nb * nb * npw
    rot = 8 * nb * nb * npw
    if case["path"] == "apply":
        w = h_bytes, h_flops
    elif case["path"] == "batch":
        w = n_cells * n_k * h_bytes, n_cells * n_k * h_flops
    elif case["path"] == "solve":
        w = h_bytes, 4 * h_flops
    elif case["path"] == "orth":
        w = 2 * nb * npw * e, gram + rot / 2 + 8 / 3 * nb ** 3
    elif case["path"] == "adjoint":
        w = 2 * h_bytes + n ** 3 * e, 3 * h_flops + 4 * 8 * nproj * nb * npw
    else:
        w = h_bytes + 4 * nb * npw * e, 4 * h_flops + 2 * gram + 3 * rot + nb * fft
    return {"bytes": float(w[0]), "flops": float(w[1])}


# ---- the same outputs in 64 bits, plain torch -----------------------------------------------------
def _grid(lat, ecut, kpts):
    m = np.abs(_sphere(lat, 4 * ecut)[0]).max(axis=0)
    span = np.max([n.max(axis=0) - n.min(axis=0) for n in (_sphere(lat, ecut, k)[0] for k in kpts)], axis=0)
    return tuple(_smooth(int(x)) for x in m + span)


def _t(x):
    return torch.as_tensor(x, device="cuda")


class _Exact:
    """H of one k-point in complex128; pos may require a gradient."""

    def __init__(self, lat, pos, d, ecut, kfrac, grid, kb):
        self.lat, self.grid, self.n = lat, grid, int(np.prod(grid))
        self.pos = _t(pos).double() if not torch.is_tensor(pos) else pos
        self.omega = abs(np.linalg.det(lat))
        mil, g, kin = _sphere(lat, ecut, kfrac)
        idx = np.mod(mil, grid)
        self.idx = _t((idx[:, 0] * grid[1] + idx[:, 1]) * grid[2] + idx[:, 2])
        self.g, self.kin = _t(g), _t(kin)
        # local potential on the density sphere |G|^2/2 <= 4 ecut (the divergent G = 0 term dropped)
        ax = [np.where(2 * np.arange(m) < m, np.arange(m), np.arange(m) - m) for m in grid]
        nm = np.stack(np.meshgrid(*ax, indexing="ij"), axis=-1).reshape(-1, 3)
        gg = nm @ (2 * math.pi * np.linalg.inv(lat).T)
        self.g2 = _t(np.sum(gg * gg, axis=1))
        keep = np.nonzero((0.5 * np.sum(gg * gg, axis=1) <= 4 * ecut) & np.all(2 * np.abs(nm) < grid, axis=1))[0]
        g2, gk = self.g2[_t(keep)], _t(gg[keep])
        z, rc, amp, a = PP["Z"], PP["rc"], PP["A"], PP["a"]
        safe = torch.where(g2 > 0, g2, torch.ones_like(g2))
        form = torch.where(g2 > 0, -4 * math.pi * z * torch.exp(-g2 * rc * rc / 4) / safe,
                           torch.full_like(g2, math.pi * z * rc * rc))
        form = (form + amp * math.pi ** 1.5 * a ** 3 * torch.exp(-g2 * a * a / 4)) / self.omega
        sf = torch.exp(-1j * (gk @ self.pos.T)).sum(dim=1)
        vg = torch.zeros(self.n, dtype=torch.complex128, device="cuda").index_put((_t(keep),), sf * form)
        self.vloc = torch.fft.ifftn(vg.reshape(grid)).real * self.n
        self.v, self.beta, self.dvec, self.d = self.vloc, None, None, d
        if kb:
            q2 = (self.g ** 2).sum(dim=1)
            gauss = torch.exp(-q2 * KB_RC ** 2 / 4)
            n0 = ((math.pi / 2) ** 1.5 * KB_RC ** 3) ** -0.5
            n1 = ((math.pi / 2) ** 1.5 * KB_RC ** 5 / 4) ** -0.5
            forms = torch.cat([(n0 * math.pi ** 1.5 * KB_RC ** 3 * gauss)[None].to(torch.complex128),
                               -1j * n1 * (math.pi ** 1.5 * KB_RC ** 5 / 2) * self.g.T * gauss])
            phase = torch.exp(-1j * (self.pos @ self.g.T)) / math.sqrt(self.omega)
            self.beta = (phase[:, None, :] * forms[None]).reshape(-1, len(kin))
            self.dvec = _t(np.stack([d[:, 0], d[:, 1], d[:, 1], d[:, 1]], axis=1).reshape(-1))

    def real(self, c):
        f = torch.zeros((c.shape[0], self.n), dtype=torch.complex128, device="cuda")
        f = f.index_put((torch.arange(c.shape[0], device="cuda")[:, None], self.idx[None, :]), c)
        return torch.fft.ifftn(f.reshape((-1,) + self.grid), dim=(1, 2, 3)) * self.n

    def h(self, c):
        out = []
        for x in c.split(max(1, 2 ** 27 // self.n)):
            f = torch.fft.fftn(self.real(x) * self.v, dim=(1, 2, 3)).reshape(x.shape[0], -1) / self.n
            out.append(self.kin * x + f[:, self.idx])
        y = torch.cat(out)
        if self.beta is not None:
            y = y + (self.dvec[:, None] * (self.beta.conj() @ c.T)).T @ self.beta
        return y

    def sigma(self):
        lb = float(self.v.min())
        if self.beta is not None:
            bn = (self.beta.abs() ** 2).sum(dim=1).reshape(-1, 4).cpu().numpy()
            lb += sum(d[0] * b[0] * (d[0] < 0) + 3 * d[1] * max(b[1:]) * (d[1] < 0) for d, b in zip(self.d, bn))
        return lb - 0.5

    def solve(self, eps, psi):
        """Preconditioned CG of (H - sigma) x = (eps - sigma) psi from x = psi; (x, steps per row)."""
        s = self.sigma()
        pre = 1.0 / (self.kin + float(self.v.mean()) - s)
        x = psi.clone()
        r = (eps - s)[:, None] * psi - (self.h(x) - s * x)
        z = pre * r
        p, rz = z.clone(), (r.conj() * z).sum(dim=1).real
        r0 = torch.linalg.vector_norm(r, dim=1)
        on = r0 > 0
        its = torch.zeros(len(r0), dtype=torch.int32, device="cuda")
        for _ in range(INNER_IT):
            if not bool(on.any()):
                break
            ap = self.h(p) - s * p
            pap = (p.conj() * ap).sum(dim=1).real
            al = torch.where(on, rz / torch.where(on, pap, torch.ones_like(pap)), torch.zeros_like(rz))
            x, r, its = x + al[:, None] * p, r - al[:, None] * ap, its + on.int()
            go = on & (torch.linalg.vector_norm(r, dim=1) > INNER_TOL * r0)
            z = pre * r
            rzn = (r.conj() * z).sum(dim=1).real
            p = torch.where(go[:, None], z + torch.where(go, rzn / rz, torch.zeros_like(rz))[:, None] * p, p)
            rz, on = torch.where(go, rzn, rz), go
        return x, its

    def ritz(self, y):
        hy = self.h(y)
        m = y.conj() @ hy.T
        eps, c = torch.linalg.eigh(0.5 * (m + m.conj().T))
        return eps, c.T @ y, c.T @ hy

    def density(self, c, f):
        rho = torch.zeros(self.grid, dtype=torch.float64, device="cuda")
        step = max(1, 2 ** 27 // self.n)
        for x, o in zip(c.split(step), f.split(step)):
            rho += (o[:, None, None, None] * self.real(x).abs() ** 2).sum(dim=0)
        return rho / self.omega

    def hartree_xc(self, rho):
        """V_H + V_xc, E_H, E_xc (Perdew-Zunger LDA)."""
        rg = torch.fft.fftn(rho.to(torch.complex128)).reshape(-1) / self.n
        k = torch.where(self.g2 > 0, 4 * math.pi / torch.where(self.g2 > 0, self.g2, torch.ones_like(self.g2)),
                        torch.zeros_like(self.g2))
        vh = torch.fft.ifftn((k * rg).reshape(self.grid)).real * self.n
        eh = 0.5 * self.omega * float((k * rg.abs() ** 2).sum())
        r = rho.clamp(min=1e-30)
        ex = -0.75 * (3 * r / math.pi) ** (1 / 3)
        rs = (3 / (4 * math.pi * r)) ** (1 / 3)
        sq, ln = rs.sqrt(), rs.log()
        den = 1 + 1.0529 * sq + 0.3334 * rs
        ec = torch.where(rs >= 1, -0.1423 / den, 0.0311 * ln - 0.048 + 0.0020 * rs * ln - 0.0116 * rs)
        vc = torch.where(rs >= 1, -0.1423 / den * (1 + 7 / 6 * 1.0529 * sq + 4 / 3 * 0.3334 * rs) / den,
                         0.0311 * ln - 0.048 - 0.0311 / 3 + 2 / 3 * 0.0020 * rs * ln + (-2 * 0.0116 - 0.0020) / 3 * rs)
        ok = rho >= 1e-30
        vxc = torch.where(ok, 4 / 3 * ex + vc, torch.zeros_like(r))
        exc = torch.where(ok, rho * (ex + ec), torch.zeros_like(r))
        return vh + vxc, eh, self.omega / self.n * float(exc.sum())

    def ewald(self):
        z, pos, lat = PP["Z"], self.pos, _t(self.lat)
        eta = math.sqrt(math.pi) / self.omega ** (1 / 3)
        edge = min(np.linalg.norm(self.lat, axis=1))  # cubic cells
        m = int(6.2 / eta / edge) + 2
        ax = torch.arange(-m, m + 1, device="cuda", dtype=torch.float64)
        shift = torch.cartesian_prod(ax, ax, ax) @ lat
        e = 0.0
        for t in shift:
            dist = torch.linalg.vector_norm(pos[:, None] - pos[None] + t, dim=2)
            ok = dist > 1e-12
            dist = torch.where(ok, dist, torch.ones_like(dist))
            e += 0.5 * z * z * float(torch.where(ok, torch.erfc(eta * dist) / dist, torch.zeros_like(dist)).sum())
        m = int(2 * eta * 6.2 * edge / (2 * math.pi)) + 2
        ax = torch.arange(-m, m + 1, device="cuda", dtype=torch.float64)
        g = torch.cartesian_prod(ax, ax, ax) @ (2 * math.pi * torch.linalg.inv(lat).T)
        g2 = (g * g).sum(dim=1)
        g, g2 = g[g2 > 0], g2[g2 > 0]
        sf = z * torch.exp(1j * (g @ pos.T)).sum(dim=1)
        e += 2 * math.pi / self.omega * float((sf.abs() ** 2 * torch.exp(-g2 / (4 * eta * eta)) / g2).sum())
        nz = z * len(pos)
        return e - eta / math.sqrt(math.pi) * z * nz - math.pi * nz * nz / (2 * self.omega * eta * eta)


def _orthonormal(x):
    s = x.conj() @ x.T
    low = torch.linalg.cholesky(0.5 * (s + s.conj().T))
    return torch.linalg.solve_triangular(low.conj(), x, upper=False)


def _fermi(eps, n_el):
    lo, hi = float(eps.min()) - 1, float(eps.max()) + 1
    for _ in range(200):
        mu = 0.5 * (lo + hi)
        lo, hi = (mu, hi) if float((2 * torch.special.expit((mu - eps) / KT)).sum()) < n_el else (lo, mu)
    g = torch.special.expit((mu - eps) / KT)
    ent = -(torch.special.xlogy(g, g) + torch.special.xlogy(1 - g, 1 - g)).sum()
    return 2 * g, -2 * KT * float(ent)


def _exact_scf(e, psi, n_occ):
    """The first SCF iteration from the start vectors psi: uniform density, one set of source problems."""
    rho = torch.full(e.grid, 2.0 * n_occ / e.omega, dtype=torch.float64, device="cuda")
    e.v = e.vloc + e.hartree_xc(rho)[0]
    eps, psi, _ = e.ritz(_orthonormal(psi))
    occ, _ = _fermi(eps, 2.0 * n_occ)
    y = _orthonormal(e.solve(eps, psi)[0])
    rho = rho + BETA_MIX * (e.density(y, occ) - rho)
    e.v = e.vloc + e.hartree_xc(rho)[0]
    eps, psi, hpsi = e.ritz(y)
    occ, mts = _fermi(eps, 2.0 * n_occ)
    rho = e.density(psi, occ)
    _, eh, exc = e.hartree_xc(rho)
    t = dict(kinetic=float((occ[:, None] * e.kin * psi.abs() ** 2).sum()), nonlocal_=0.0,
             local=e.omega / e.n * float((e.vloc * rho).sum()), hartree=eh, xc=exc, ewald=e.ewald())
    if e.beta is not None:
        t["nonlocal_"] = float((occ * (e.dvec[:, None] * (e.beta.conj() @ psi.T).abs() ** 2)).sum())
    t["total"] = sum(t.values()) + mts
    order = ["ewald", "hartree", "kinetic", "local", "nonlocal_", "total", "xc"]
    res = torch.linalg.vector_norm(hpsi - eps[:, None] * psi, dim=1)[:n_occ].max()
    return dict(energy=torch.tensor([t[k] for k in order], dtype=torch.float64), resid=res, eps=eps[None], rho=rho,
                psi=None)  # the phases of eigenvectors are the eigensolver's own


def exact(case, seed):
    out = []
    i = 0
    for lat, pos, d, ecut, kpts in _problems(case, seed):
        grid = _grid(lat, ecut, kpts)
        for k in kpts:
            kin = _sphere(lat, ecut, k)[2]
            given = _rows(case["nb"], kin, seed * 100 + i, case["dtype"])
            psi = given.to(torch.complex128)
            i += 1
            if case["path"] == "orth":
                out.append(_orthonormal(psi))
                continue
            if case["path"] == "adjoint":
                p = _t(pos).to(_real(case)).double().requires_grad_(True)
                v = _v_rest(grid, seed, case["dtype"]).double().requires_grad_(True)
                w = _rows(case["nb"], kin, seed * 100 + 50, case["dtype"]).to(torch.complex128)
                psi.requires_grad_(True)
                e = _Exact(lat, p, d, ecut, k, grid, case["kb"])
                e.v = e.vloc + v
                y = e.h(psi)
                g = torch.autograd.grad(y, (psi, v, p), w)
                out.append(dict(y=y.detach(), g_psi=g[0], g_v=g[1], g_pos=g[2]))
                continue
            e = _Exact(lat, pos, d, ecut, k, grid, case["kb"])
            if case["path"] == "solve":
                x, its = e.solve(_t(_levels(given, kin)), psi)
                out.append(dict(x=x, its=its))
            elif case["path"] == "scf":
                out.append(_exact_scf(e, psi, case["n_occ"]))
            else:
                out.append(e.h(psi))
            del e
    return out if case["path"] == "batch" else out[0]
