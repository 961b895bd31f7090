"""What the C ABI does when a launch is refused: the compiled pf_api linked with
a host-only CUDA runtime and launchers whose launches can fail (no GPU)."""
import os
import subprocess

import pytest

from paper_1202_6116_gb300 import build as B

HERE = os.path.dirname(os.path.abspath(__file__))
OK, ERR_CUDA = 0, 2


@pytest.fixture(scope="module")
def fake(tmp_path_factory):
    B.build()
    exe = str(tmp_path_factory.mktemp("fake") / "fake_cuda")
    srcs = [os.path.join(HERE, "fakes", f) for f in ("fake_cuda.cu", "fake_runtime.cpp")]
    for f in ("pf_api", "pf_noalloc"):
        obj = os.path.join(B.OBJ_DIR, f + ".o")
        srcs.append(obj if os.path.exists(obj) else os.path.join(B.CSRC, f + ".cu"))
    r = subprocess.run([B._nvcc(), "-O1", "-std=c++17", "--expt-relaxed-constexpr", "-cudart", "none", "-I" + B.INCLUDE,
                        "-I" + B.CSRC] + B.ARCH + srcs + ["-o", exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr

    def run(*args):
        r = subprocess.run([exe, *args], capture_output=True, text=True, timeout=60)
        assert r.returncode == 0, (r.returncode, r.stderr)
        lines = [ln.split() for ln in r.stdout.splitlines()]
        counts = [{k: int(v) for k, v in (w.split("=") for w in ln[1:])} for ln in lines if ln[0] != "status"]
        return [(int(ln[1]), int(ln[3])) + tuple(counts[2 * i:2 * i + 2])
                for i, ln in enumerate(x for x in lines if x[0] == "status")]
    return run


def test_without_failures(fake):
    for st, _, direct, _ in fake("solve", "pcg", "none"):
        assert st == OK and direct["cg_loop"] == 1 and "cg_p" not in direct
    (st, steps, _, captured), _ = fake("step", "mg", "none")
    assert st == OK and steps == 1 and captured["mg_sub"] >= 1
    for st, _, direct, _ in fake("noalloc", "pcg", "none"):
        assert st == OK and direct["cg_loop"] == 1 and "cg_p" not in direct


def test_refused_loop_iterates_with_two_launches(fake):
    """Solves and host-driven steps clear the refusal, iterate as without the loop and do not try it again."""
    for what in ("solve", "nograph"):
        first, second = fake(what, "pcg", "loop")
        assert first[0] == second[0] == OK
        assert first[2]["cg_loop"] == 1 and first[2]["cg_p"] >= 1 and first[2]["cg_r"] >= 1
        assert "cg_loop" not in second[2] and second[2]["cg_p"] >= 1
    for st, _, direct, _ in fake("noalloc", "pcg", "loop"):       # it keeps nothing between calls
        assert st == OK and direct["cg_p"] >= 1


@pytest.mark.parametrize("what", ["step", "batch"])
def test_refused_loop_in_a_capture(fake, what):
    """The graph is captured once more with the two launches, and steps still run as graphs."""
    first, second = fake(what, "pcg", "loop")
    assert first[0] == second[0] == OK
    assert first[1] == 1 and second[1] == 5
    assert first[3]["cg_p"] >= 1 and first[2]["graph"] == 1
    assert "cg_loop" not in second[3]


@pytest.mark.parametrize("what", ["step", "batch", "nograph", "solve"])
def test_refused_small_levels_are_an_error(fake, what):
    """The V-cycle has no other form of its small levels: no graph is run without them."""
    for st, _, direct, _ in fake(what, "mg", "sub"):
        assert st == ERR_CUDA
        assert "graph" not in direct
