"""The V-cycle's small levels as one launch (levels spread over a cluster,
levels in one block, the product with the coarsest level's inverse) and the
persistent Jacobi-PCG loop, at the sizes where each of their branches begins:
potentials against the FP64 oracle, FP64 bar 1e-10 as in the parity tests."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_1202_6116_gb300 import build as B
from paper_1202_6116_gb300 import pf
from paper_1202_6116_gb300.film import Film

from helpers import mixed_workload, oracle_grid, oracle_params, relerr

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    B.build()
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    pf.lib()


def solve(w, **over):
    f = Film(w, **over)
    st, info = f.solve_potential()
    phi = f.numpy()[1]
    f.close()
    assert st == pf.PF_OK
    return phi, info


@pytest.mark.parametrize("shape,eps,faces", [
    ((16, 16, 1), False, "mixed"),      # one block runs every level; coarsest 1 cell
    ((16, 8, 8), True, "mixed"),        # the finest level spread over the cluster (FP64), with eps
    ((24, 20, 12), False, "mixed"),     # coarsest 3 x 5 x 3: a row per thread
    ((16, 16, 16), False, "periodic"),  # singular: constant vector taken out of the inverse
    ((36, 20, 9), True, "mixed"),       # coarsest 9 x 5 x 9 = 405: a row per warp over the cluster
    ((42, 36, 8), False, "open"),       # coarsest 21 x 9 x 1, singular, rows of no whole vectors
    ((64, 34, 8), False, "mixed"),      # 17 x 1 coarse rows, levels above the launch
    ((8, 8, 37), True, "mixed"),        # a z column is left: 1 x 1 x 37
])
def test_small_levels_match_oracle_fp64(shape, eps, faces):
    w = mixed_workload(*shape, 61, eps=eps).with_(solver="mg", maxit=300, rtol=1e-13)
    if faces != "mixed":
        z8 = np.zeros_like(w.type_lo)
        w = w.with_(type_lo=z8, type_hi=z8, periodic_z=faces == "periodic")
    phio, st, _, _ = O.solve_potential(oracle_grid(w), w.P0, rtol=1e-14)
    assert st == O.OK
    phi, info = solve(w)
    assert relerr(phi, phio) <= 1e-10
    assert info["last_iters"] <= 60


def test_new_electrode_layout_renews_the_inverse():
    """A second layout on the same context: the solve must use its own coarsest operator."""
    w = mixed_workload(36, 20, 9, 62).with_(solver="mg", maxit=300, rtol=1e-13)
    w2 = mixed_workload(36, 20, 9, 63, tol_dirichlet=0.1).with_(solver="mg", maxit=300, rtol=1e-13)
    f = Film(w)
    f.solve_potential()
    f.set_bc(pf.PF_ZLO, w2.type_lo, w2.volt_lo)
    f.set_bc(pf.PF_ZHI, w2.type_hi, w2.volt_hi)
    f.phi.zero_()
    _, info = f.solve_potential()
    phi = f.numpy()[1]
    f.close()
    phio, st, _, _ = O.solve_potential(oracle_grid(w2.with_(P0=w.P0)), w.P0, rtol=1e-14)
    assert st == O.OK and relerr(phi, phio) <= 1e-10
    fresh, info2 = solve(w2.with_(P0=w.P0))
    assert info["last_iters"] == info2["last_iters"]


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("shape,faces", [
    ((1, 1, 1), "mixed"), ((5, 3, 2), "mixed"), ((17, 33, 3), "mixed"),   # a thread per cell, ragged tiles
    ((32, 32, 32), "mixed"), ((24, 16, 12), "periodic"), ((24, 16, 12), "open"),
    ((160, 64, 32), "mixed"),                                             # 16-byte vectors (FP32: 4 cells)
    ((164, 100, 41), "mixed"),                                            # vectors on ragged tiles, several per thread
])
def test_cg_loop_matches_the_two_kernel_iteration(precision, shape, faces):
    """The persistent loop against the same solve with a permittivity field of
    ones, which iterates with one launch per half step: same operator, same
    iteration, sums in another order.  FP64 within 1e-10 of the largest
    potential, FP32 within the solve tolerance times the grid's conditioning
    (1e-4, as in the parity tests)."""
    w = mixed_workload(*shape, 64, precision=precision, rtol=1e-13 if precision == "fp64" else 1e-7)
    if faces != "mixed":
        z8 = np.zeros_like(w.type_lo)
        w = w.with_(type_lo=z8, type_hi=z8, periodic_z=faces == "periodic")
    phi, info = solve(w)
    ref, info_ref = solve(w.with_(eps=np.ones(w.shape)))
    assert relerr(phi, ref) <= (1e-10 if precision == "fp64" else 1e-4)
    assert abs(info["last_iters"] - info_ref["last_iters"]) <= max(2, info_ref["last_iters"] // 50)
    # the whole loop is one launch
    assert info["kernel_launches"] <= 5 < info_ref["kernel_launches"] or shape == (1, 1, 1)


@pytest.mark.parametrize("shape", [(32, 32, 16), (32, 32, 32), (64, 64, 32), (64, 64, 36)])
def test_small_levels_fp32_by_cluster_size(shape):
    """First levels of 16 384 cells (8 blocks) and just above (16), as the finest level and below it: potentials
    within the FP32 parity bar of the oracle."""
    w = mixed_workload(*shape, 65, precision="fp32", rtol=1e-7).with_(solver="mg", maxit=300)
    phio, st, _, _ = O.solve_potential(oracle_grid(w), w.P0, rtol=1e-14)
    assert st == O.OK
    phi, info = solve(w)
    assert relerr(phi, phio) <= 1e-4
    assert info["last_iters"] <= 30


@pytest.mark.parametrize("solver", ["pcg", "mg"])
@pytest.mark.parametrize("shape", [(32, 24, 13), (37, 22, 11), (64, 32, 16)])
def test_patchwork_permittivity_matches_oracle(solver, shape):
    """Blocks of two permittivities: cells whose six neighbours share theirs (no harmonic mean formed) beside cells
    whose neighbours do not, within one warp.  FP64 bar 1e-10 as in the parity tests."""
    if solver == "mg" and shape[0] % 2:
        shape = (40, 24, 12)
    w = mixed_workload(*shape, 66).with_(solver=solver, maxit=3000, rtol=1e-13)
    z, y, x = np.meshgrid(*(np.arange(n) for n in w.shape), indexing="ij")
    w = w.with_(eps=np.where((x // 7 + y // 5 + z // 4) % 2, 30.0, 1.0))
    phio, st, _, _ = O.solve_potential(oracle_grid(w), w.P0, rtol=1e-14)
    assert st == O.OK
    phi, _ = solve(w)
    assert relerr(phi, phio) <= 1e-10


@pytest.mark.parametrize("precision,tol", [("fp64", 1e-12), ("fp32", 1e-5)])
@pytest.mark.parametrize("nz", [8192, 8193])
def test_tall_grids_match_oracle(nz, precision, tol):
    """More than 128 tiles of the largest depth in z (64 planes), and just fewer: the plain rule of the
    tile depth.  Sums over the grid with the bars of the diagnostics' tests."""
    w = mixed_workload(4, 4, nz, 67, precision=precision, amp=0.7)
    f = Film(w)
    f.phi.copy_(0.3 * f.P[0] + 0.1 * f.P[2])
    P, phi = f.numpy()
    d = f.diagnostics(0.3)
    f.close()
    o = O.diagnostics(oracle_grid(w), oracle_params(w), P, phi, 0.3)
    assert d["switched_fraction"] == o["switched_fraction"]
    for k in ("mean_px", "mean_py", "mean_pz"):
        assert abs(d[k] - o[k]) <= tol * np.abs(P).max()
    for k in ("f_landau", "f_grad", "f_elec"):
        assert abs(d[k] - o[k]) <= tol * abs(o[k])
