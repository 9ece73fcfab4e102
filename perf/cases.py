"""Performance cases: calls a program makes through the public entry points of
paper_1905_01348_gb300, from a 16-orbital exchange to a 432-orbital PT-CN step.

Kinds
  exchange  System.exchange(): W = V_X Psi of the current orbitals (Eq. 3), mixed
            precision or FP64, on the orbital grid or on a coarser Fock grid;
  batch     Batch.exchange(): the same for several small systems in shared launches,
            as the server runs them;
  apply_h   System.apply_h(): H X for a block of vectors (an eigensolver's or a
            propagator's call);
  product   pt_complex_product(): the dense products of ACE and of the PT residual;
  step      System.step(): one whole PT-CN step (Eq. 5, Alg. 1).

Every case carries its sizes as plain numbers: grid n0 n1 n2, cell edges a0 a1 a2
(bohr), cutoff, orbitals. The listed silicon cells are those of the synthetic
package (10.26 bohr and 32 points per cubic cell, 10 Ha, two orbitals per atom).

What a mixed-precision run leaves behind has the 24 bits of the FP32 pair
transforms and tensor-core products it was made with, so the program keeps it as
complex64 / float32; what an FP64 run leaves is kept as it is.
"""
import math

import numpy as np
import torch

import synthetic as syn
import paper_1905_01348_gb300 as pt

DEV = "cuda:0"


def _system(name, kind, reps, n, n_orb, **more):
    edge = syn.SI_CUBIC_CELL_BOHR * reps
    c = dict(name=name, kind=kind, n0=n, n1=n, n2=n, a0=edge, a1=edge, a2=edge, reps=reps, ecut=10.0, n_orb=n_orb,
             precision="mixed", fock=0)
    c.update(more)
    return c


def listed():
    return [
        # One primitive cubic cell, the smallest system served: launches and latency.
        _system("exchange_si8", "exchange", 1, 32, 16),
        # The 2x2x2 supercell, the ordinary size.
        _system("exchange_si64", "exchange", 2, 64, 128),
        # The 3x3x3 supercell: 93,528 pairs at 96^3, the call that bounds a production step.
        _system("exchange_si216", "exchange", 3, 96, 432),
        # Exchange on a coarse (aliasing) Fock grid as the paper uses, part of the bands, a ragged last tile.
        _system("exchange_fock48", "exchange", 3, 96, 101, fock=48),
        # A non-cubic cell in FP64 with a ragged last tile: a reference calculation on a slab.
        dict(name="exchange_fp64_slab", kind="exchange", n0=24, n1=48, n2=32, a0=7.7, a1=15.39, a2=10.26, reps=1,
             ecut=10.0, n_orb=27, precision="fp64", fock=0),
        # Twelve single cells, as the continuous-batching server steps them together.
        _system("batch_si8", "batch", 1, 32, 16, systems=12),
        # H applied to a full block of vectors with the ACE operator.
        _system("apply_h_si64", "apply_h", 2, 64, 128, cols=128, mode="ace"),
        # M = Psi^H W at the 3x3x3 supercell's basis: the long reduction of ACE and the PT residual.
        dict(name="product_overlap_si216", kind="product", op_a=1, op_b=0, m=432, n=432, k=43819),
        # One PT-CN step of each workload (20 SCF iterations: what the density tolerance 1e-6 takes),
        # and of the smallest in FP64, the reference precision. The largest starts from a shorter
        # relaxation, enough for its SCF to be stable.
        _system("step_si8", "step", 1, 32, 16, iters=20, relax=40),
        _system("step_fp64_si8", "step", 1, 32, 16, iters=20, relax=40, precision="fp64"),
        _system("step_si64", "step", 2, 64, 128, iters=20, relax=40),
        _system("step_si216", "step", 3, 96, 432, iters=20, relax=12),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


# Cubic grids and the most orbitals drawn on each.
_CUBIC = {32: 64, 48: 160, 64: 200, 96: 320}
_EDGES = (8, 12, 16, 24, 32, 48, 64)


def draw(rng):
    kind = rng.choice(("exchange", "exchange", "exchange", "exchange", "batch", "apply_h", "product", "product",
                       "step", "step"))
    if kind == "product":
        op_a, op_b = rng.choice(((1, 0), (1, 0), (0, 0), (0, 1)))
        small = [_log_int(rng, 8, 500) for _ in range(2)]
        basis = _log_int(rng, 500, 60000)
        # a reduction over the basis (A^H B), or a basis-sized left operand times a small factor
        m, n, k = (small[0], small[1], basis) if op_a else (basis, small[0], small[0] if op_b else small[1])
        return dict(kind=kind, op_a=op_a, op_b=op_b, m=m, n=n, k=k)
    prec = rng.choice(("mixed", "mixed", "mixed", "fp64"))
    if kind == "exchange" and prec == "fp64":
        n = [rng.choice(_EDGES) for _ in range(3)]
        while n[0] * n[1] * n[2] > 48 ** 3:
            n = [rng.choice(_EDGES) for _ in range(3)]
        a = [e / 32 * syn.SI_CUBIC_CELL_BOHR * rng.uniform(0.95, 1.05) for e in n]
        c = dict(kind=kind, n0=n[0], n1=n[1], n2=n[2], a0=a[0], a1=a[1], a2=a[2], reps=1,
                 ecut=rng.uniform(6.0, 10.0), precision=prec, fock=0)
        # the orbitals stay a fraction of the basis
        c["n_orb"] = min(_log_int(rng, 3, 64), max(1, _npw(c) // 4))
        return c
    big = {"exchange": 96, "apply_h": 64, "batch": 48, "step": 64}[kind]
    e = rng.choice([v for v in _CUBIC if v <= big])
    if prec == "fp64":
        e = 32
    # the wells of `reps` cubed cells in a cell of the drawn edge
    a = e / 32 * syn.SI_CUBIC_CELL_BOHR * rng.uniform(0.97, 1.03)
    c = dict(kind=kind, n0=e, n1=e, n2=e, a0=a, a1=a, a2=a, reps=max(1, e // 32), ecut=rng.uniform(8.0, 10.0),
             precision=prec, fock=0)
    if kind == "batch":
        c.update(n_orb=_log_int(rng, 3, 24), systems=rng.randint(2, 12))
    elif kind == "step":
        # near the filling of the drawn cell, so that the start relaxes and the SCF converges
        full = 16 * c["reps"] ** 3
        c.update(n_orb=rng.randint(full - full // 8, full), iters=20, relax=40)
    else:
        c["n_orb"] = _log_int(rng, 1, _CUBIC[e])
        if kind == "exchange" and e > 48 and rng.random() < 0.3:
            c["fock"] = {64: 32, 96: 48}[e]
        if kind == "apply_h":
            c.update(cols=_log_int(rng, 1, c["n_orb"]), mode=rng.choice(("ace", "exact", "none")))
    return c


# ---- inputs -------------------------------------------------------------------------


def _normal(shape, seed, salt):
    g = torch.Generator(device=DEV)
    g.manual_seed(1000003 * (seed % (1 << 40)) + salt)
    z = torch.randn(tuple(shape) + (2,), generator=g, device=DEV, dtype=torch.float64)
    return torch.view_as_complex(z)


def _axes(n, a):
    """Integer frequencies of a length-n axis and the wave numbers 2 pi m / a."""
    m = np.arange(n)
    m = np.where(m < (n + 1) // 2, m, m - n)
    return m, 2.0 * np.pi * m / a


def _g2(n, a):
    g = [_axes(n[k], a[k])[1] for k in range(3)]
    return g[0][:, None, None] ** 2 + g[1][None, :, None] ** 2 + g[2][None, None, :] ** 2


def _grid(case):
    return (case["n0"], case["n1"], case["n2"]), (case["a0"], case["a1"], case["a2"])


def _coefficients(case, seed, salt=0):
    """Random smooth start orbitals (not orthonormal), (n_orb, npw) complex128 on the device."""
    n, a = _grid(case)
    g2 = _g2(n, a).reshape(-1)
    g2 = torch.from_numpy(g2[0.5 * g2 <= case["ecut"]]).to(DEV)
    return _normal((case["n_orb"], g2.numel()), seed, salt) * torch.exp(-0.25 * g2)


def _workload(case):
    n, a = _grid(case)
    _, frac = syn.diamond_supercell(case["reps"])
    w = dict(syn.COMMON, n=n, cell=a, atoms=frac, n_orb=case["n_orb"], ecut=case["ecut"],
             precision=case["precision"], fock_mode="ace", relax_iters=case.get("relax", 0),
             scf_fixed_iters=case.get("iters", 0))
    if case["fock"]:
        w["fock_grid"] = (case["fock"],) * 3
    return w


def _product_shapes(case):
    m, n, k = case["m"], case["n"], case["k"]
    # column-major operands as row-major tensors of their transposes
    return ((m, k) if case["op_a"] else (k, m)), ((k, n) if case["op_b"] else (n, k)), (n, m)


def _product_inputs(case, seed):
    sa, sb, _ = _product_shapes(case)
    return _normal(sa, seed, 1).to(torch.complex64), _normal(sb, seed, 2).to(torch.complex64)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "product":
        A, B = _product_inputs(case, seed)
        C = torch.empty(_product_shapes(case)[2], dtype=torch.complex128, device=DEV)
        ws = torch.empty(16 * case["m"] * case["n"] * 16 + 256 if case["op_a"] else 4096, dtype=torch.uint8, device=DEV)
        return dict(case=case, A=A, B=B, C=C, ws=ws, stream=torch.cuda.current_stream().cuda_stream)
    w = _workload(case)
    if kind == "batch":
        systems = []
        for q in range(case["systems"]):
            s = torch.cuda.Stream()
            systems.append(pt.System(w, _coefficients(case, seed, q).cpu().numpy(), stream=s))
        return dict(case=case, batch=pt.Batch(systems), systems=systems)
    state = dict(case=case, system=pt.System(w, _coefficients(case, seed).cpu().numpy()))
    if kind == "apply_h":
        state["X"] = _normal((case["cols"], state["system"].npw), seed, 77)
    return state


def _kept(case, t):
    return t.to(torch.complex64) if case.get("precision", "mixed") == "mixed" else t


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "exchange":
        return _kept(case, state["system"].exchange())
    if kind == "batch":
        return [_kept(case, t) for t in state["batch"].exchange()]
    if kind == "apply_h":
        mode = {"ace": pt.PT_FOCK_ACE, "exact": pt.PT_FOCK_EXACT, "none": pt.PT_FOCK_NONE}[case["mode"]]
        return _kept(case, state["system"].apply_h(state["X"], mode))
    if kind == "product":
        A, B, C, ws = state["A"], state["B"], state["C"], state["ws"]
        pt.pt_complex_product(case["op_a"], case["op_b"], case["m"], case["n"], case["k"], 1.0, A.data_ptr(),
                              A.shape[1], B.data_ptr(), B.shape[1], 0.0, C.data_ptr(), C.shape[1], False,
                              ws.data_ptr(), ws.numel(), state["stream"])
        return _kept(case, C)
    _, info = state["system"].step()
    observables = np.array([info["energy"], *info["dipole"]])
    if case["precision"] == "mixed":
        observables = observables.astype(np.float32)
    return dict(psi=_kept(case, state["system"].orbitals_device()), observables=observables)


# ---- work ---------------------------------------------------------------------------


def _npw(case):
    n, a = _grid(case)
    return int(np.count_nonzero(0.5 * _g2(n, a) <= case["ecut"]))


def _exchange_flops(case):
    points = case["fock"] ** 3 if case["fock"] else case["n0"] * case["n1"] * case["n2"]
    pairs = case["n_orb"] * (case["n_orb"] + 1) / 2
    # two transforms, the product, the kernel and two accumulations per pair
    return pairs * points * (10.0 * math.log2(points) + 6 + 2 + 16)


def work(case):
    """Bytes of the inputs and outputs; flops of the pair transforms, the dense products and the
    orbital transforms of the method (no padding, no retries)."""
    kind = case["kind"]
    if kind == "product":
        m, n, k = case["m"], case["n"], case["k"]
        return dict(bytes=8.0 * (m * k + k * n) + 16.0 * m * n, flops=8.0 * m * n * k)
    npw, ne = _npw(case), case["n_orb"]
    block = 16.0 * npw * ne
    if kind == "exchange":
        return dict(bytes=2 * block, flops=_exchange_flops(case))
    if kind == "batch":
        return dict(bytes=2 * block * case["systems"], flops=_exchange_flops(case) * case["systems"])
    points = case["n0"] * case["n1"] * case["n2"]
    fft = 5.0 * points * math.log2(points)
    if kind == "apply_h":
        cols = case["cols"]
        flops = cols * (2 * fft + 8 * points) + ne * 4.0 * points
        if case["mode"] == "ace":
            flops += 2 * 8.0 * npw * ne * cols
        elif case["mode"] == "exact":
            flops += 2 * cols / (ne + 1) * _exchange_flops(case)
        # the orbitals (they define the density), the vectors and the result; the ACE vectors
        return dict(bytes=block * (2 if case["mode"] == "ace" else 1) + 2 * 16.0 * npw * cols, flops=flops)
    gemm = 8.0 * npw * ne * ne
    per_iter = ne * (2 * fft + 10 * points) + 4 * gemm + 20 * 2 * 16.0 * npw * ne
    return dict(bytes=2 * block, flops=_exchange_flops(case) + case["iters"] * per_iter + 5 * gemm)


# ---- the same in 64 bits --------------------------------------------------------------


class _Reference:
    """Plain torch complex128 evaluation of the method (columns stored as rows)."""

    def __init__(self, case):
        self.case = case
        n, a = _grid(case)
        self.n, self.points = n, n[0] * n[1] * n[2]
        self.vol = a[0] * a[1] * a[2]
        w = _workload(case)
        self.w = w
        g2 = _g2(n, a)
        keep = np.flatnonzero(0.5 * g2.reshape(-1) <= case["ecut"])
        self.idx = torch.from_numpy(keep).to(DEV)
        self.g2 = torch.from_numpy(g2).to(DEV)
        i = np.unravel_index(keep, n)
        g = [_axes(n[k], a[k])[1][i[k]] + w["kick"][k] for k in range(3)]
        self.kin = torch.from_numpy(0.5 * (g[0] ** 2 + g[1] ** 2 + g[2] ** 2)).to(DEV)
        # the Fock grid: the same basis vectors on (possibly) fewer points
        f = (case["fock"],) * 3 if case["fock"] else n
        m = [_axes(n[k], a[k])[0][i[k]] for k in range(3)]
        self.nf = f
        self.idx_f = torch.from_numpy(((m[0] % f[0]) * f[1] + m[1] % f[1]) * f[2] + m[2] % f[2]).to(DEV)
        gf = torch.from_numpy(_g2(f, a)).to(DEV)
        om2 = w["omega"] ** 2
        k = 4.0 * math.pi * -torch.expm1(-gf / (4.0 * om2)) / torch.where(gf > 0, gf, 1.0)
        self.khat = torch.where(gf > 0, k, math.pi / om2)
        self.dv = self.vol / self.points
        self.r = [torch.arange(n[q], device=DEV, dtype=torch.float64) * (a[q] / n[q]) for q in range(3)]
        wells = []
        for q in range(3):
            d = self.r[q][None, :, None] - torch.from_numpy(w["atoms"][:, q] * a[q]).to(DEV)[:, None, None]
            d = d - torch.arange(-3, 4, device=DEV, dtype=torch.float64) * a[q]
            wells.append(torch.exp(-d * d / (2.0 * w["well_sigma"] ** 2)).sum(-1))
        self.vion = -w["well_depth"] * torch.einsum("ai,aj,ak->ijk", *wells)

    def real(self, c, fock=False):
        n, idx = (self.nf, self.idx_f) if fock else (self.n, self.idx)
        points = n[0] * n[1] * n[2]
        grid = torch.zeros((c.shape[0], points), dtype=torch.complex128, device=DEV)
        grid[:, idx] = c
        return torch.fft.ifftn(grid.view(-1, *n), dim=(1, 2, 3)) * (points / math.sqrt(self.vol))

    def basis(self, f, fock=False):
        n, idx = (self.nf, self.idx_f) if fock else (self.n, self.idx)
        points = n[0] * n[1] * n[2]
        return torch.fft.fftn(f, dim=(1, 2, 3)).reshape(-1, points)[:, idx] * (math.sqrt(self.vol) / points)

    def orthonormal(self, c):
        # rows: S_ij = sum_G conj(c_i) c_j = L L^H, rows of c replaced by those of L^{-*} c
        L = torch.linalg.cholesky(c.conj() @ c.T)
        return torch.linalg.solve_triangular(L.conj(), c, upper=False)

    def vx(self, c, x=None):
        """V_X[c] x (x: c itself when not given)."""
        psi = self.real(c, True)
        xs = psi if x is None else self.real(x, True)
        out = torch.zeros_like(xs)
        step = max(1, (1 << 27) // psi[0].numel())
        for i in range(psi.shape[0]):
            for j in range(i if x is None else 0, xs.shape[0], step):
                part = slice(j, min(j + step, xs.shape[0]))
                v = torch.fft.ifftn(self.khat * torch.fft.fftn(psi[i].conj() * xs[part], dim=(1, 2, 3)), dim=(1, 2, 3))
                out[part] += psi[i] * v
                if x is None:
                    first = i + 1 - j if j == i else 0   # the diagonal pair counts once
                    out[i] += (xs[part][first:] * v[first:].conj()).sum(0)
        return -self.w["alpha"] * self.basis(out, True)

    def density(self, c):
        return 2.0 * self.real(c).abs().square().sum(0)

    def vloc(self, rho):
        coulomb = torch.where(self.g2 > 0, 4.0 * math.pi / torch.where(self.g2 > 0, self.g2, 1.0), 0.0)
        self.vh = torch.fft.ifftn(coulomb * torch.fft.fftn(rho)).real
        return self.vion + self.vh - (1.0 - self.w["alpha"]) * (3.0 * rho / math.pi) ** (1.0 / 3.0)

    def local(self, v, x):
        return self.kin * x + self.basis(v * self.real(x))

    def ace(self, c, w):
        L = torch.linalg.cholesky(-(c.conj() @ w.T))
        return torch.linalg.solve_triangular(L.conj(), w, upper=False)

    def ace_apply(self, xi, x):
        return -((x @ xi.conj().T) @ xi)

    def project(self, c, h):
        return h - (h @ c.conj().T) @ c

    def relaxed(self, c):
        w = self.w
        kerker = w.get("relax_mix", 0.5) * self.g2 / (self.g2 + w.get("relax_q0", 1.0) ** 2)
        mix = self.density(c)
        for _ in range(w["relax_iters"]):
            mix = mix + torch.fft.ifftn(kerker * torch.fft.fftn(self.density(c) - mix)).real
            r = self.project(c, self.local(self.vloc(mix), c))
            c = self.orthonormal(c - w.get("relax_tau", 1.0) * r / (1.0 + self.kin))
        return c

    def step(self, c):
        w = self.w
        wx = self.vx(c)
        xi = self.ace(c, wx)
        half = 0.5j * w["dt"]
        start = c - half * self.project(c, self.local(self.vloc(self.density(c)), c) + wx)
        x, dx, dr, x_old, r_old = start, [], [], None, None
        for _ in range(case_iters(self.case)):
            h = self.local(self.vloc(self.density(x)), x) + self.ace_apply(xi, x)
            r = start - x - half * self.project(x, h)
            if x_old is not None:
                dx, dr = (dx + [x - x_old])[-w["anderson_dim"]:], (dr + [r - r_old])[-w["anderson_dim"]:]
            x_old, r_old = x, r
            x = x + w["anderson_beta"] * r
            if dx:
                D, X = torch.stack(dr, -1), torch.stack(dx, -1)      # (band, npw, history)
                G = D.mH @ D
                tr = G.diagonal(dim1=1, dim2=2).real.sum(1)
                G = G + 1e-14 * tr[:, None, None] * torch.eye(G.shape[1], device=DEV)
                L, bad = torch.linalg.cholesky_ex(G)
                gamma = torch.cholesky_solve(D.mH @ r[:, :, None], L)
                gamma = torch.where((bad == 0)[:, None, None], gamma, 0.0)
                x = x - ((X + w["anderson_beta"] * D) @ gamma)[:, :, 0]
        return self.orthonormal(x)

    def observables(self, c):
        rho = self.density(c)
        self.vloc(rho)
        w = self.w
        e = 2.0 * (self.kin * c.abs().square()).sum() + self.dv * (self.vion * rho + 0.5 * self.vh * rho).sum()
        e = e - (1.0 - w["alpha"]) * 0.75 * (3.0 / math.pi) ** (1.0 / 3.0) * self.dv * (rho ** (4.0 / 3.0)).sum()
        e = e + (c.conj() * self.vx(c)).sum().real
        d = [-self.dv * (rho.sum([t for t in range(3) if t != q]) * self.r[q]).sum() for q in range(3)]
        return torch.stack([e, *d]).cpu()


def case_iters(case):
    return case["iters"]


def exact(case, seed):
    kind = case["kind"]
    if kind == "product":
        A, B = (t.to(torch.complex128) for t in _product_inputs(case, seed))
        a = A.conj() if case["op_a"] else A.T
        b = B.conj() if case["op_b"] else B.T
        return (a @ b).T.contiguous()
    # FP64 transforms of every pair: beyond some 5e12 flops this takes too long
    if _exchange_flops(case) * case.get("systems", 1) * (3 if kind == "step" else 1) > 5e12:
        return None
    ref = _Reference(case)
    if kind == "batch":
        return [ref.vx(ref.orthonormal(_coefficients(case, seed, q))) for q in range(case["systems"])]
    c = ref.orthonormal(_coefficients(case, seed))
    if kind == "exchange":
        return ref.vx(c)
    if kind == "apply_h":
        x = _normal((case["cols"], c.shape[1]), seed, 77)
        y = ref.local(ref.vloc(ref.density(c)), x)
        if case["mode"] == "exact":
            y = y + ref.vx(c, x)
        elif case["mode"] == "ace":
            y = y + ref.ace_apply(ref.ace(c, ref.vx(c)), x)
        return y
    c = ref.step(ref.relaxed(c))
    return dict(psi=c, observables=ref.observables(c))
