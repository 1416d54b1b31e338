"""The integrate kernels' local walk (LWalker), compiled for the host, against
the oracle's walk: the same voxels in the same order for every segment length,
for short and long pieces, on random, tie-heavy, nearly axis-aligned and very
short rays (Sec. III-B)."""
import os
import subprocess

import numpy as np
import pytest

import oracle

HERE = os.path.dirname(os.path.abspath(__file__))
U = 1 << 16


@pytest.fixture(scope="module")
def checker(tmp_path_factory):
    exe = str(tmp_path_factory.mktemp("piece") / "piece_check")
    subprocess.run(["nvcc", "-gencode", "arch=compute_103a,code=sm_103a", "-std=c++17", "-O2", "-x", "cu",
                    os.path.join(HERE, "host", "piece_check.cu"), "-o", exe], check=True, capture_output=True)
    return exe


def _rays(kind, rng, n):
    if kind == "random":
        a = rng.integers(-100 * U, 100 * U, size=(n, 3))
        return a, a + rng.integers(-300 * U, 300 * U, size=(n, 3))
    if kind == "lattice":  # faces, edges, corners, exact diagonals
        q = U // 4
        a = rng.integers(-40, 40, size=(n, 3)) * q
        return a, a + rng.integers(-200, 200, size=(n, 3)) * q
    if kind == "diagonal":  # within a few units of exact diagonals, from lattice points and off them
        a = rng.integers(-20, 20, size=(n, 3)) * U + rng.integers(0, 2, size=(n, 1)) * rng.integers(0, U, size=(n, 3))
        d = rng.integers(-150, 150, size=(n, 1)) * U
        return a, a + d * rng.choice([-1, 1], size=(n, 3)) + rng.integers(-2, 3, size=(n, 3))
    if kind == "flat":  # one or two axes barely move
        a = rng.integers(-100 * U, 100 * U, size=(n, 3))
        d = rng.integers(-400 * U, 400 * U, size=(n, 3))
        flat = rng.integers(0, 2, size=(n, 3)).astype(bool)
        return a, a + np.where(flat, rng.integers(-3, 4, size=(n, 3)), d)
    a = rng.integers(-3 * U, 3 * U, size=(n, 3))  # short: zero length up to two voxels
    return a, a + rng.integers(-2 * U, 2 * U, size=(n, 3)) * rng.integers(0, 2, size=(n, 3))


@pytest.mark.parametrize("S", [1, 3, 24, 31, 40, 1 << 20])
@pytest.mark.parametrize("kind", ["random", "lattice", "diagonal", "flat", "short"])
def test_piece_walk_matches_oracle(checker, S, kind):
    rng = np.random.default_rng(1000 + S)
    A, B = _rays(kind, rng, 150)
    text = "16 %d %d\n" % (S, len(A)) + "\n".join("%d %d %d %d %d %d" % (*a, *b) for a, b in zip(A, B)) + "\n"
    out = subprocess.run([checker], input=text, capture_output=True, text=True)
    assert out.returncode == 0, out.returncode
    tok = out.stdout.split()
    i = 0
    for a, b in zip(A, B):
        c = int(tok[i])
        got = np.array(tok[i + 1:i + 1 + 3 * c], dtype=np.int64).reshape(c, 3)
        i += 1 + 3 * c
        assert np.array_equal(got, oracle.walk(a, b)), (a, b)
    exact, steps = int(out.stderr.split()[1]), int(out.stderr.split()[3])
    if kind in ("lattice", "diagonal"):
        assert exact > 0             # ties must reach the exact rule
    elif kind == "random":
        assert exact < 0.01 * steps  # and ordinary steps must not
