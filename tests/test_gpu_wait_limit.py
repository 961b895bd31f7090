"""Bounded waits of the persistent CG loop: with a limit of one poll a healthy
solve's waits give up, the call reports PF_ERR_TIMEOUT at once however many
steps it has, and the context goes on afterwards."""
import time

import numpy as np
import pytest
import torch

from paper_1202_6116_gb300 import build as B
from paper_1202_6116_gb300 import pf
from paper_1202_6116_gb300.batch import Batch
from paper_1202_6116_gb300.film import Film

from helpers import mixed_workload

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    B.build()
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    pf.lib()


def restart(f, w):
    f.P.copy_(torch.as_tensor(w.P0, dtype=f.dtype))
    f.phi.zero_()
    pf.pf_bind(f.ctx, f.P, f.phi, f.eps, f.workspace, f.ws_bytes)
    f.set_bc(pf.PF_ZLO, w.type_lo, w.volt_lo)
    f.set_bc(pf.PF_ZHI, w.type_hi, w.volt_hi)


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("how", ["graph", "host", "heun", "solve"])
def test_wait_limit_reports_a_timeout_and_the_context_goes_on(precision, how):
    w = mixed_workload(64, 48, 32, 91, precision=precision, rtol=1e-10 if precision == "fp64" else 1e-6)
    over = {"host": dict(flags=pf.PF_FLAG_NO_GRAPHS), "heun": dict(integrator=pf.PF_HEUN)}.get(how, {})

    def go(f, ok):
        return f.solve_potential(ok) if how == "solve" else f.step(6, ok)

    ref = Film(w, **over)
    go(ref, (pf.PF_OK,))
    want = ref.numpy()
    ref.close()
    f = Film(w, **over)
    pf.pf_set_wait_limit(f.ctx, 1)
    t0 = time.perf_counter()
    st, info = go(f, (pf.PF_ERR_TIMEOUT,))
    assert st == pf.PF_ERR_TIMEOUT and info["status"] == pf.PF_ERR_TIMEOUT
    assert info["nonconverged"] >= 1
    assert time.perf_counter() - t0 < 5.0
    st, _ = go(f, (pf.PF_ERR_TIMEOUT,))                 # and again, from whatever is there
    assert st == pf.PF_ERR_TIMEOUT
    pf.pf_set_wait_limit(f.ctx)
    restart(f, w)
    go(f, (pf.PF_OK,))
    got = f.numpy()
    f.close()
    assert np.array_equal(got[0], want[0]) and np.array_equal(got[1], want[1])


def test_later_solves_of_the_call_end_at_once():
    """200 steps of a batch of which one film's waits give up: none of its solves begins an iteration after the
    first one, and the other film is not touched."""
    ws = [mixed_workload(64, 48, 32, 92 + i, rtol=1e-10) for i in range(2)]
    films = [Film(w) for w in ws]
    b = Batch(films, max_records=1)
    pf.pf_set_wait_limit(films[0].ctx, 1)
    t0 = time.perf_counter()
    st, info = b.step(200, (pf.PF_ERR_TIMEOUT,))
    assert st == pf.PF_ERR_TIMEOUT and time.perf_counter() - t0 < 5.0
    bad, good = b.film_info(0), b.film_info(1)
    assert bad["status"] == pf.PF_ERR_TIMEOUT and bad["nonconverged"] == 200 and bad["total_iters"] == 0
    assert good["status"] == pf.PF_OK and good["nonconverged"] == 0
    got = films[1].numpy()
    b.close()
    for f in films:
        f.close()
    alone = Film(ws[1])
    alone.step(200)
    want = alone.numpy()
    alone.close()
    assert np.array_equal(got[0], want[0]) and np.array_equal(got[1], want[1])
