"""Sums of FP32 fields past the range of a float: a tile's sum of squares can
exceed 3.4e38 while every thread's own fits.  Scaling P, and with it the
potential, by a power of two changes the exponents alone, so the scaled film
solves as the unscaled one up to the order of the sums: potentials within the
FP32 parity bar."""
import numpy as np
import pytest
import torch

from paper_1202_6116_gb300 import build as B
from paper_1202_6116_gb300 import pf
from paper_1202_6116_gb300.film import Film

from helpers import mixed_workload, relerr

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    B.build()
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    pf.lib()


def solve(w, scale):
    f = Film(w, P0=torch.as_tensor(w.P0 * scale))
    st, info = f.solve_potential()
    phi = f.phi.clone()
    f.close()
    return phi, info


@pytest.mark.parametrize("solver,shape,eps", [
    ("pcg", (96, 64, 24), False),        # persistent loop, vectors
    ("pcg", (37, 50, 24), False),        # persistent loop, single cells
    ("pcg", (96, 64, 24), True),         # two kernels an iteration
    ("mg", (96, 64, 24), False),
    ("mg", (32, 32, 32), False),         # every level in the small levels' launch
])
def test_solve_scales_past_the_float_range(solver, shape, eps):
    # |b| up to 3.5e18, its squares 1.2e37 at most; 2048 cells of a tile sum to more than 1e39
    w = mixed_workload(*shape, 95, precision="fp32", eps=eps, volts=False, rtol=1e-6).with_(solver=solver)
    phi, info = solve(w, 1.0)
    big, info_big = solve(w, 2.0 ** 61)
    assert info_big["status"] == pf.PF_OK
    assert abs(info_big["last_iters"] - info["last_iters"]) <= 1
    assert relerr((big.double() * 2.0 ** -61).cpu().numpy(), phi.double().cpu().numpy()) <= 1e-4


def test_mean_polarization_past_the_float_range():
    w = mixed_workload(96, 64, 24, 96, precision="fp32", volts=False)
    P0 = np.zeros_like(w.P0)
    P0[2] = 1.0
    P0[2, :, ::2] = 0.75
    f = Film(w, P0=torch.as_tensor(P0 * 2.0 ** 119))
    d = f.diagnostics()
    f.close()
    assert d["mean_px"] == 0.0 and d["mean_pz"] == 0.875 * 2.0 ** 119
