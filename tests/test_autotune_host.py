"""The autotuner's choice on the host: a candidate has to beat the default by
more than runs differ, and all of them start alike."""
import pytest
import torch

from paper_1202_6116_gb300 import autotune as AT
from paper_1202_6116_gb300 import pf
from paper_1202_6116_gb300 import workloads as W


class FakeFilm:
    calls = []

    def __init__(self, w, device=None):
        self.ctx = None
        self.P, self.phi = torch.zeros(3), torch.zeros(1)

    def solve_potential(self, ok=(pf.PF_OK,)):
        self.calls.append("solve")

    def close(self):
        pass


@pytest.mark.parametrize("gain,chosen", [(0.01, (4, 5, 0)), (0.2, (4, 8, 0))])
def test_default_stays_unless_clearly_beaten(monkeypatch, gain, chosen):
    def timed(f, t, steps, warmup):
        f.calls.append(t)
        return 1.0 - gain if t == (4, 8, 0) else 1.0

    FakeFilm.calls = []
    monkeypatch.setattr(AT, "Film", FakeFilm)
    monkeypatch.setattr(AT, "_CACHE", {})
    monkeypatch.setattr(AT, "time_tiling", timed)
    monkeypatch.setattr(AT.pf, "pf_get_tiling", lambda ctx: pf.pf_tiling(4, 5, 0, 0))
    res = AT.tune(W.film_fp64_grounded(32, 32, 32).with_(precision="fp32"), device="cpu")
    assert (res["vx"], res["tz"], res["blocks_per_sm"]) == chosen
    calls = FakeFilm.calls
    assert calls[1] == (4, 5, 0)                                   # the default first
    assert calls[::2] == ["solve"] * (len(calls) // 2)             # each after a fresh solve
