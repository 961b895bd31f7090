"""Rounding of one TDGL update against the same step in extended precision,
on states whose potential is exactly zero: each component of P depends on the
two coordinates across it, so div P = 0 in every cell of a periodic film."""
import numpy as np
import pytest
import torch

from paper_1202_6116_gb300 import build as B
from paper_1202_6116_gb300 import pf
from paper_1202_6116_gb300 import workloads as W
from paper_1202_6116_gb300.film import Film

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    B.build()
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    pf.lib()


def divergence_free(nx, ny, nz, mean, amp, seed, dtype):
    """mean + amp U[-1, 1] per component, constant along its own axis, representable in dtype."""
    rng = np.random.default_rng(seed)
    u = [rng.uniform(-1, 1, s) for s in ((nz, ny, 1), (nz, 1, nx), (1, ny, nx))]
    return np.stack([np.broadcast_to((m + amp * v).astype(dtype), (nz, ny, nx)) for m, v in zip(mean, u)]).astype(float)


def one_step(P0, precision, **coeffs):
    _, nz, ny, nx = P0.shape
    z8, z = np.zeros((ny, nx), np.int8), np.zeros((ny, nx))
    w = W.Workload("update", nx, ny, nz, P0, z8, z, z8, z, precision=precision, periodic_z=True, rtol=1e-7, **coeffs)
    f = Film(w)
    f.step(1)
    P, phi = f.numpy()
    f.close()
    assert (phi == 0.0).all()
    return P


def landau(P, a1, a11, a12):
    p2 = P * P
    return -(2 * a1 * P + 4 * a11 * P * p2 + 2 * a12 * P * (p2.sum(0) - p2))


@pytest.mark.parametrize("axis", [0, 1, 2])
def test_fp32_landau_force_has_no_bias_at_a_pole(axis):
    """Mean error of the force over thousands of states next to P = 1 along one
    axis, with dt L = 1024 so that the updated P shows the force itself.  One
    value's error is at most a few half-ulps of the terms of size 2 (rms 6e-8),
    plus the rounding of P of size 40 / 1024: its mean over 4096 independent
    values scatters by 1e-9.  A coefficient off by one rounding shifts it by 3e-8."""
    mean = [0.0] * 3
    mean[axis] = 1.0
    n = [64, 64, 64]
    n[axis] = 4                                     # the biased component varies over the other two axes
    P0 = divergence_free(*n, mean, 0.01, 5 + axis, np.float32)
    P = one_step(P0, "fp32", g=0.0, dt=1024.0)
    err = (P[axis] - P0[axis]) / 1024.0 - landau(P0, -1.0, 0.5, 0.8)[axis]
    assert abs(err.mean()) <= 1e-8
    assert np.abs(err).max() <= 5e-7


@pytest.mark.parametrize("dt", [0.3, 0.021, 0.0208, 0.005])
def test_fp64_gradient_term(dt):
    """The gradient term alone, from near the explicit limit (g dt L/dx^2 = 0.15) to a
    usual step: the updated P of size 1 is off by its own rounding (rms 0.29 units
    in the last place) and little more, the increment being 50 times smaller than P."""
    P0 = divergence_free(40, 36, 32, [0.97, 0.97, 0.97], 0.01, 11, np.float64)
    P = one_step(P0, "fp64", a1=0.0, a11=0.0, a12=0.0, g=0.5, dt=dt)
    X = P0.astype(np.longdouble)
    lap = sum(np.roll(X, s, d) - X for d in (1, 2, 3) for s in (1, -1))
    err = (P.astype(np.longdouble) - (X + np.longdouble(dt) * np.longdouble(0.5) * lap)) * 2.0 ** 53
    assert float(np.sqrt((err * err).mean())) <= 0.35


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_adjoint_hessian_has_no_bias_at_a_pole(precision):
    """(lam_out - lam) / dt L = -H(P) lam where P and lam have no divergence
    (psi = 0) and g = 0, dt L = 1024.  Each value of size 4 is off by a few of its
    half-ulps u = 2^-24 or 2^-53 (rms 4 u); the mean over 4096 independent ones
    scatters by u / 16.  Coefficients that do not add up to 12 a11 shift it by 2 u.
    The sensitivities come from the same products."""
    dt = np.float32 if precision == "fp32" else np.float64
    u = 2.0 ** -24 if precision == "fp32" else 2.0 ** -53
    n = (64, 64, 4)
    P0 = divergence_free(*n, [0.0, 0.0, 1.0], 0.01, 21, dt)
    lam0 = divergence_free(*n, [0.0, 0.0, 1.0], 0.01, 22, dt)
    z8, z = np.zeros((64, 64), np.int8), np.zeros((64, 64))
    w = W.Workload("adjoint", *n, P0, z8, z, z8, z, precision=precision, periodic_z=True, rtol=1e-7, g=0.0, dt=1024.0)
    f = Film(w, flags=pf.PF_FLAG_ADJOINT)
    lam = torch.as_tensor(lam0, dtype=f.dtype, device="cuda").contiguous()
    out, grad = torch.empty_like(lam), torch.zeros(4, dtype=torch.float64, device="cuda")
    pf.pf_adjoint_step(f.ctx, lam, out, grad)
    got = out.double().cpu().numpy()
    f.close()
    X, Y = P0.astype(np.longdouble), lam0.astype(np.longdouble)
    p2, pl = X * X, X * Y
    H = Y * (-2 + 6 * p2 + np.longdouble(1.6) * (p2.sum(0) - p2)) + np.longdouble(3.2) * X * (pl.sum(0) - pl)
    # lam_out has size 4096: its own rounding is one part in 1024 of the force's
    err = ((got.astype(np.longdouble) - Y) / 1024 + H)[2]
    assert abs(float(err.mean())) <= u / 2
    assert float(np.abs(err).max()) <= 32 * u
    ref = [-1024 * float((2 * pl).sum()), -1024 * float((4 * p2 * pl).sum()),
           -1024 * float((2 * pl * (p2.sum(0) - p2)).sum()),
           1024 * float((X * sum(np.roll(Y, s, d) - Y for d in (1, 2, 3) for s in (1, -1))).sum())]
    assert np.abs(grad.cpu().numpy() - ref).max() <= 16 * u * max(map(abs, ref))
