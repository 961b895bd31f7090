"""Jacobi films in large batches: each film's loop takes another launch form
there (two launches an iteration, or fewer blocks of the persistent loop), and
must give the bits of the film stepped alone."""
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


def films_of(shapes, precision):
    """Films of these shapes in turn with random electrodes; the third of every four is periodic in z, the fourth has
    open faces."""
    out = []
    for i, s in enumerate(shapes):
        w = mixed_workload(*s, 70 + i, precision=precision, rtol=1e-12 if precision == "fp64" else 1e-6)
        if i % 4 >= 2:
            z8 = np.zeros_like(w.type_lo)
            w = w.with_(type_lo=z8, type_hi=z8, periodic_z=i % 4 == 2)
        out.append(w)
    return out


def batch_against_alone(ws, steps):
    films = [Film(w) for w in ws]
    b = Batch(films, max_records=1)
    b.step(steps)
    got = [f.numpy() for f in films]
    infos = [b.film_info(i) for i in range(len(ws))]
    b.close()
    for f in films:
        f.close()
    for w, (P, phi), info in zip(ws, got, infos):
        f = Film(w)
        _, alone = f.step(steps)
        Pa, phia = f.numpy()
        f.close()
        assert np.array_equal(P, Pa) and np.array_equal(phi, phia), w.name
        assert info["total_iters"] == alone["total_iters"]
    return infos


# several tiles per thread group, ragged tiles, blocks not a multiple of eight, one tile only
SMALL = [(32, 32, 32), (33, 20, 27), (64, 48, 12), (16, 16, 5), (40, 72, 19), (48, 48, 16)]


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_large_batch_of_small_jacobi_films_equals_films_alone(precision):
    ws = films_of([SMALL[i % len(SMALL)] for i in range(28)], precision)
    infos = batch_against_alone(ws, 5)
    # two launches an iteration (measured faster once the films' loops do not fit the GPU side by side)
    assert all(i["kernel_launches"] >= 2 * i["total_iters"] for i in infos)


def test_batch_of_32_with_large_jacobi_films_equals_films_alone():
    """FP32 films whose loops fill the GPU by themselves run them on fewer blocks from 32 films on."""
    ws = films_of([(16, 16, 8)] * 27 + [(96, 96, 48), (128, 96, 40), (100, 104, 44), (96, 96, 48), (72, 96, 64)], "fp32")
    infos = batch_against_alone(ws, 4)
    assert all(i["kernel_launches"] < 40 for i in infos[27:])          # one launch a loop


def test_small_batch_keeps_the_persistent_loop():
    ws = films_of([(32, 32, 32)] * 2, "fp32")
    infos = batch_against_alone(ws, 5)
    assert all(i["kernel_launches"] < 40 for i in infos)


@pytest.mark.parametrize("precision,shapes", [
    ("fp32", [(128, 64, 80), (96, 96, 48), (101, 75, 40), (128, 64, 80)]),   # loops that need the whole GPU each
    ("fp32", [(100, 104, 44), (32, 32, 32), (97, 96, 52), (64, 64, 32), (96, 96, 48)]),
    ("fp64", [(96, 96, 48), (75, 101, 50), (96, 80, 56)]),
])
def test_batch_of_few_large_jacobi_films_equals_films_alone(precision, shapes):
    infos = batch_against_alone(films_of(shapes, precision), 4)
    # two launches an iteration, from the third film on that has the GPU to itself
    assert all(i["kernel_launches"] >= 2 * i["total_iters"] for i in infos)
