"""Edges of the GPU kernels' tiles and of the rules that choose between them, each against the
FP64 oracle (or, for the dense products, exact complex128 products of the same inputs).

Tolerances are those derived in test_gpu_parity.py (FP64: 1e-10 of the largest value; the
FP32 pair path: 2e-5) and test_gpu_tensor_products.py (1e-5).
"""
import os

import numpy as np
import pytest

import synthetic as syn
from oracle import ptcn as pc

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    import paper_1905_01348_gb300 as p
    from paper_1905_01348_gb300 import build as b
    if not os.path.exists(p._native.LIB_PATH):
        b.build()
    p.load()
    return p


def rel(a, b):
    return float(np.max(np.abs(a - b)) / np.max(np.abs(b)))


def workload(n, n_orb, spacing=0.45, ecut=2.5, **more):
    """A cell of `spacing` bohr per grid point and axis (a per mille apart, to tell the axes apart)."""
    cell = tuple(spacing * k * f for k, f in zip(n, (1.0, 1.001, 0.998)))
    return dict(syn.COMMON, n=n, cell=cell, ecut=ecut, atoms=np.array([[0.1, 0.2, 0.3], [0.6, 0.55, 0.9]]),
                n_orb=n_orb, relax_iters=0, omega=0.3, **more)


def make(w, seed=0):
    model = pc.Model(pc.Params.from_dict(w))
    return model, syn.initial_coefficients(model.grid.g2_basis(), w["n_orb"], seed=seed)


def make_basis(w):
    return len(pc.Model(pc.Params.from_dict(w)).grid.g2_basis())


@pytest.mark.parametrize("precision,tol", [("fp64", 1e-10), ("mixed", 2e-5)])
@pytest.mark.parametrize("n", [(8, 24, 48), (48, 12, 64), (96, 8, 16), (24, 96, 12), (64, 48, 32), (12, 16, 96)])
def test_exchange_line_lengths(pkg, n, precision, tol):
    """Every transform length on every axis of the generic pair kernels, an odd number of pairs."""
    w = workload(n, 5, precision=precision)
    model, C0 = make(w)
    st = model.init_state(C0)
    s = pkg.System(w, C0)
    assert rel(s.exchange().cpu().numpy().T, st.W) < tol
    s.close()


@pytest.mark.parametrize("n,spacing", [((16, 24, 12), 0.9), ((12, 16, 24), 1.1), ((32, 32, 32), 1.0)])
@pytest.mark.parametrize("precision,tol", [("fp64", 1e-10), ("mixed", 2e-5)])
def test_exchange_with_aliasing(pkg, n, spacing, precision, tol):
    """Pair products beyond the grid's frequencies alias: no slab or column may be skipped."""
    w = workload(n, 4, spacing=spacing, precision=precision)
    model, C0 = make(w)
    assert not model.grid.alias_free()
    st = model.init_state(C0)
    s = pkg.System(w, C0)
    assert rel(s.exchange().cpu().numpy().T, st.W) < tol
    s.close()


@pytest.mark.parametrize("edge,n_orb,tile", [(32, 13, 0), (32, 5, 3), (48, 9, 0), (48, 2, 1), (64, 8, 0), (64, 6, 2),
                                             (64, 18, 0), (96, 5, 0)])
def test_exchange_cubic_tiles(pkg, edge, n_orb, tile):
    """The FP32 cubic kernels with full, ragged and diagonal tiles, odd pair counts and small tile edges."""
    w = workload((edge,) * 3, n_orb, spacing=0.33, precision="mixed", pair_tile=tile)
    model, C0 = make(w, seed=3)
    st = model.init_state(C0)
    s = pkg.System(w, C0)
    assert rel(s.exchange().cpu().numpy().T, st.W) < 2e-5
    s.close()


@pytest.mark.parametrize("edge,n_orb", [(64, 126), (96, 27), (96, 29)])
def test_grouped_tiles_add_in_the_same_order(pkg, edge, n_orb):
    """Tiles side by side in a launch (ragged last blocks, empty places) give the sums of one tile at a time."""
    out = []
    for tile in (0, 1):
        w = workload((edge,) * 3, n_orb, precision="mixed", pair_tiles_per_launch=tile)
        C0 = np.random.default_rng(1).standard_normal((n_orb, make_basis(w), 2)).view(np.complex128)[..., 0]
        s = pkg.System(w, C0)
        out.append(s.exchange().clone())
        s.close()
    assert out[0].equal(out[1])


@pytest.mark.parametrize("n_orb", [1, 15, 16, 17, 31, 32, 33, 65])
def test_orthonormalisation_sizes(pkg, n_orb):
    """Overlap, Cholesky panels of 32 columns, the factor's inverse and the triangular product."""
    w = workload((16, 16, 16), n_orb, spacing=0.5, ecut=6.0, precision="fp64", alpha=0.0)
    model, C0 = make(w, seed=5)
    st = model.init_state(C0)
    s = pkg.System(w, C0)
    assert rel(s.orbitals().T, st.Psi) < 1e-10
    s.close()


@pytest.mark.parametrize("depth,iters", [(0, 3), (1, 4), (3, 7)])
def test_anderson_depths(pkg, depth, iters):
    """No history, one entry, and a history that wraps around."""
    w = workload((12, 16, 24), 5, precision="fp64", fock_mode="ace", scf_fixed_iters=iters, anderson_dim=depth, dt=0.5)
    w["relax_iters"] = 3
    model, C0 = make(w, seed=2)
    st, info_o = model.step(model.init_state(C0))
    s = pkg.System(w, C0)
    _, info_g = s.step()
    assert rel(s.orbitals().T, st.Psi) < 1e-10
    assert abs(info_g["energy"] - info_o.energy) < 1e-10 * abs(info_o.energy)
    s.close()


@pytest.mark.parametrize("precision,tol", [("fp64", 1e-10), ("mixed", 1e-4)])
@pytest.mark.parametrize("edge", [32, 48, 64, 96])
def test_local_potential_and_transforms(pkg, edge, precision, tol):
    """H X without exchange (Hartree solve, FP64 transforms) and a step of one orbital (the step's
    transforms in its own precision) on the cubic grids; the step's bound is that of the
    single-orbital parity test."""
    import torch
    w = workload((edge,) * 3, 2, spacing=0.33, precision=precision, fock_mode="ace", scf_fixed_iters=2, dt=0.5)
    w["relax_iters"] = 1
    model, C0 = make(w, seed=7)
    st = model.init_state(C0)
    s = pkg.System(w, C0)
    X = syn.gaussian_vectors((model.grid.npw, 2), seed=1)
    Y = s.apply_h(torch.from_numpy(np.ascontiguousarray(X.T)).to("cuda:0"), pkg.PT_FOCK_NONE).cpu().numpy().T
    assert rel(Y, model.apply_h(st.Psi, X, "none")) < 1e-10
    st, _ = model.step(st)
    s.step()
    assert rel(s.orbitals().T, st.Psi) < tol
    s.close()


@pytest.mark.parametrize("op_a,op_b,M,N,K,scratch", [
    (1, 0, 16, 16, 1647, True), (1, 0, 17, 33, 4099, True), (1, 0, 15, 1, 511, True), (1, 0, 16, 16, 20000, False),
    (0, 0, 1647, 16, 16, True), (0, 1, 301, 31, 31, True), (1, 1, 40, 20, 700, True),
    (1, 0, 64, 64, 3000, True), (1, 0, 73, 74, 3000, True), (1, 0, 128, 128, 13133, True),
    (0, 0, 31, 17, 512, True), (0, 1, 16, 1, 8192, False), (1, 0, 16, 16, 8193, True), (1, 0, 1, 1, 1000, False),
])
def test_product_small_outputs(pkg, op_a, op_b, M, N, K, scratch):
    """Both sides of the rule that sends small outputs to the CUDA cores, with and without split-K."""
    import torch
    a_shape, b_shape = ((K, M) if op_a == 0 else (M, K)), ((N, K) if op_b == 0 else (K, N))
    A, B = (syn.gaussian_vectors(sh, q).astype(np.complex64) for q, sh in enumerate((a_shape, b_shape)))
    C0 = syn.gaussian_vectors((N, M), 2)
    exact = (0.5 - 1j) * ((A.T if op_a == 0 else A.conj()).astype(complex) @ (B.T if op_b == 0 else B.conj())) + 2j * C0.T
    dA, dB, dC = (torch.from_numpy(np.ascontiguousarray(t)).to("cuda:0") for t in (A, B, C0))
    ws = torch.empty((64 << 20) if scratch else 256, dtype=torch.uint8, device="cuda:0")
    pkg.pt_complex_product(op_a, op_b, M, N, K, 0.5 - 1j, dA.data_ptr(), a_shape[1], dB.data_ptr(), b_shape[1], 2j,
                           dC.data_ptr(), M, False, ws.data_ptr(), ws.numel(), torch.cuda.current_stream().cuda_stream)
    assert rel(dC.cpu().numpy().T, exact) < 1e-5


@pytest.mark.parametrize("op_a,op_b,M,N,K", [(0, 0, 1, 1048561, 3), (1, 0, 17, 1048577, 16), (0, 1, 3, 1100001, 5),
                                             (0, 0, 1048577, 2, 9)])
def test_product_long_outputs(pkg, op_a, op_b, M, N, K):
    """Outputs of a few rows or columns whose other edge takes more than 65,535 tiles of 16."""
    import torch
    a_shape, b_shape = ((K, M) if op_a == 0 else (M, K)), ((N, K) if op_b == 0 else (K, N))
    A, B = (syn.gaussian_vectors(sh, q).astype(np.complex64) for q, sh in enumerate((a_shape, b_shape)))
    exact = (A.T if op_a == 0 else A.conj()).astype(complex) @ (B.T if op_b == 0 else B.conj())
    dA, dB = (torch.from_numpy(np.ascontiguousarray(t)).to("cuda:0") for t in (A, B))
    dC = torch.full((N, M), float("nan"), dtype=torch.complex128, device="cuda:0")
    ws = torch.empty(256, dtype=torch.uint8, device="cuda:0")
    pkg.pt_complex_product(op_a, op_b, M, N, K, 1.0, dA.data_ptr(), a_shape[1], dB.data_ptr(), b_shape[1], 0.0,
                           dC.data_ptr(), M, False, ws.data_ptr(), ws.numel(), torch.cuda.current_stream().cuda_stream)
    assert rel(dC.cpu().numpy().T, exact) < 1e-5


@pytest.mark.parametrize("op_a,op_b,M,N,K,scratch", [(1, 0, 32, 300, 20000, True), (0, 1, 2000, 32, 6000, True),
                                                     (1, 0, 16, 16, 70001, True), (1, 1, 40, 40, 33, True),
                                                     (0, 0, 300, 17, 9999, False), (1, 0, 1, 1, 4097, True)])
def test_product_long_reductions(pkg, op_a, op_b, M, N, K, scratch):
    """Small outputs whose reduction takes few to the most chunks, ragged last ones included."""
    import torch
    a_shape, b_shape = ((K, M) if op_a == 0 else (M, K)), ((N, K) if op_b == 0 else (K, N))
    A, B = (syn.gaussian_vectors(sh, q).astype(np.complex64) for q, sh in enumerate((a_shape, b_shape)))
    exact = (A.T if op_a == 0 else A.conj()).astype(complex) @ (B.T if op_b == 0 else B.conj())
    dA, dB = (torch.from_numpy(np.ascontiguousarray(t)).to("cuda:0") for t in (A, B))
    dC = torch.full((N, M), float("nan"), dtype=torch.complex128, device="cuda:0")
    ws = torch.empty((64 << 20) if scratch else 256, dtype=torch.uint8, device="cuda:0")
    pkg.pt_complex_product(op_a, op_b, M, N, K, 1.0, dA.data_ptr(), a_shape[1], dB.data_ptr(), b_shape[1], 0.0,
                           dC.data_ptr(), M, False, ws.data_ptr(), ws.numel(), torch.cuda.current_stream().cuda_stream)
    assert rel(dC.cpu().numpy().T, exact) < 1e-5


@pytest.mark.parametrize("precision,tol", [("fp64", 1e-10), ("mixed", 2e-5)])
@pytest.mark.parametrize("n,n_orb", [((8, 8, 16), 5), ((8, 12, 12), 3), ((12, 12, 8), 9), ((16, 12, 16), 6),
                                     ((16, 16, 96), 2), ((12, 8, 48), 8), ((16, 24, 16), 5), ((64, 96, 12), 5),
                                     ((96, 96, 8), 3)])
def test_exchange_short_lines_and_large_slabs(pkg, n, n_orb, precision, tol):
    """Slabs of two short axes, tiles of few short lines, and slabs that have an SM to themselves."""
    w = workload(n, n_orb, precision=precision)
    model, C0 = make(w, seed=4)
    st = model.init_state(C0)
    s = pkg.System(w, C0)
    assert rel(s.exchange().cpu().numpy().T, st.W) < tol
    s.close()


@pytest.mark.parametrize("edge,n_orb,groups", [(96, 49, 10), (96, 41, 13), (64, 130, 20)])
def test_grouped_tiles_of_odd_block_counts(pkg, edge, n_orb, groups):
    """Tiles side by side where a block has no partner (meetings of two tiles and empty places, a
    diagonal group of one) and, with 41, rounds that take two launch groups: the sums of one tile
    at a time, to the bit, and those of the FP64 kernels."""
    C0 = np.random.default_rng(2).standard_normal((n_orb, make_basis(workload((edge,) * 3, 1)), 2))
    C0 = C0.view(np.complex128)[..., 0]
    out, launches = [], []
    for more in (dict(precision="mixed"), dict(precision="mixed", pair_tiles_per_launch=1), dict(precision="fp64")):
        s = pkg.System(workload((edge,) * 3, n_orb, **more), C0)
        pkg.pt_set_timing(s.handle, True)
        pkg.pt_get_timing(s.handle, reset=True)
        out.append(s.exchange().clone())
        launches.append(pkg.pt_get_timing(s.handle)[2])
        s.close()
    assert launches[0] == groups   # one tile after the other it would be 16, 12 and 36
    assert out[0].equal(out[1])
    assert float((out[0] - out[2]).abs().max() / out[2].abs().max()) < 2e-5


@pytest.mark.parametrize("depth", [7, 11, 16, 20])
@pytest.mark.parametrize("precision,tol", [("fp64", 1e-10), ("mixed", 1e-4)])
def test_anderson_deep_histories(pkg, depth, precision, tol):
    """Every size of the history kernels, filled and wrapped around, in both history precisions."""
    w = workload((12, 16, 24), 5, precision=precision, fock_mode="ace", scf_fixed_iters=depth + 3, anderson_dim=depth,
                 dt=0.5)
    w["relax_iters"] = 3
    model, C0 = make(w, seed=2)
    st, info_o = model.step(model.init_state(C0))
    s = pkg.System(w, C0)
    _, info_g = s.step()
    assert rel(s.orbitals().T, st.Psi) < tol
    assert abs(info_g["energy"] - info_o.energy) < tol * abs(info_o.energy)
    s.close()
