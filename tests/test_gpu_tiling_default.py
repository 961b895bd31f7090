"""pf_set_tiling with what pf_get_tiling reports for a new context leaves the
film as it was: every kernel keeps (or gets back) its own planned depth."""
import numpy as np
import pytest
import torch

from paper_1202_6116_gb300 import autotune as AT
from paper_1202_6116_gb300 import build as B
from paper_1202_6116_gb300 import pf
from paper_1202_6116_gb300.film import Film

from helpers import mixed_workload

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    B.build()
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    pf.lib()


def run(w, *tilings):
    """State after three steps, the sums of the diagnostics with it: their last bits follow the tiles."""
    f = Film(w)
    for t in tilings:
        pf.pf_set_tiling(f.ctx, *t)
    f.step(3)
    d = f.diagnostics()
    out = f.P.clone(), f.phi.clone(), d
    t = pf.pf_get_tiling(f.ctx)
    f.close()
    return out, (t.vx, t.tz, t.blocks_per_sm)


def same(a, b):
    return torch.equal(a[0], b[0]) and torch.equal(a[1], b[1]) and a[2] == b[2]


@pytest.mark.parametrize("shape,precision,eps", [((320, 240, 40), "fp64", True), ((256, 256, 64), "fp32", False),
                                                 ((33, 20, 24), "fp64", False)])
def test_setting_the_default_keeps_the_planned_depths(shape, precision, eps):
    w = mixed_workload(*shape, 81, precision=precision, eps=eps, rtol=1e-10 if precision == "fp64" else 1e-6)
    ref, default = run(w)
    assert default[2] == 0
    for sets in ([default], [(default[0], 1 if default[1] > 1 else 2, 0), default], [default + (1,), default]):
        got, now = run(w, *sets)
        assert now == default
        assert same(got, ref)


def test_depths_differ_between_kernels_and_the_tuner_can_keep_them():
    """One depth for every kernel, the default's but with a grid size given, sums in another order than the
    planned depths on one of these films at least: the case that the test above is about exists.  The tuner's
    first row is the default, and applying it changes nothing."""
    differ = 0
    for w in (mixed_workload(320, 240, 40, 82, precision="fp64", eps=True, rtol=1e-6),
              mixed_workload(256, 256, 64, 83, precision="fp32", rtol=1e-5).with_(solver="mg")):
        ref, default = run(w)
        uniform, now = run(w, default[:2] + (64,))
        assert now == default[:2] + (64,)
        differ += not same(uniform, ref)
        res = AT.tune(w, steps=1, warmup=0)
        assert res["table"][0][0] == res["default"] == list(default)
        f = Film(w)
        AT.apply(f, dict(res, vx=default[0], tz=default[1], blocks_per_sm=default[2]))
        f.step(3)
        assert same((f.P, f.phi, f.diagnostics()), ref)
        f.close()
    assert differ


@pytest.mark.parametrize("shape", [(128, 128, 64), (96, 96, 48), (75, 48, 40), (64, 64, 3)])
def test_noisy_steps_do_not_depend_on_the_depth(shape):
    """The update with noise plans its own depth; with the potential held it sums nothing, so that every depth
    gives the same bits."""
    out = []
    for tz in (None, 1, 5, 32):
        f = Film(mixed_workload(*shape, 84, precision="fp32", rtol=1e-5), poisson_every=1000)
        f.set_noise(0.05, 3)
        f.step(1)
        if tz is not None:
            t = pf.pf_get_tiling(f.ctx)
            pf.pf_set_tiling(f.ctx, t.vx, min(tz, shape[2]), 0)
        f.step(4)
        out.append(f.numpy()[0])
        f.close()
    assert all(np.array_equal(o, out[0]) for o in out[1:])
