"""BF16 storage of the Bregman variable: the iterates, bit for bit.

Rounding z to 8 bits makes the last bit of every sum before it matter: where a
sum near a tie rounds the other way, one low-pass coefficient moves by 2^-8 of
itself and, at L = 1, a pixel by up to 2e-3 of the maximum.  FP32 rounding is
therefore no bound for these iterates, and the library keeps one fixed order of
every sum of a BF16-z problem (rank-one PSFs row pass first, masks tap by tap,
the partial sums of norms and inner products) whatever the batch or the launch
geometry.  tests/golden/bf16_iterates.npz holds the iterates of that order; the
comparison is exact.  Inputs are ratios of integers, so they are the same
doubles everywhere.
"""
import math
import os

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

GOLDEN = os.path.join(os.path.dirname(os.path.abspath(__file__)), "golden", "bf16_iterates.npz")


def binomial(p):
    w = np.array([math.comb(p - 1, k) for k in range(p)], dtype=np.float64)
    return np.outer(w, w) / float(int(w.sum()) ** 2)


def disk(p, r2):
    t = np.arange(p) - (p - 1) // 2
    h = (t[:, None] ** 2 + t[None, :] ** 2 <= r2).astype(np.float64)
    return h / h.sum()


def slanted(p):
    """A sparse nonsymmetric PSF along a line."""
    h = np.zeros((p, p))
    for k in range(p):
        h[k, (k + p // 2) // 2] += 2 + k % 3
        h[k, (k + p // 2) // 2 + 1] += 1
    return h / h.sum()


def image(n, k):
    """n x n: a ramp, two rectangles and integer noise, in 1/1024ths."""
    y, x = np.mgrid[0:n, 0:n]
    v = 200 + (300 * x + 150 * y) // n
    v = np.where((y > n // 4) & (y < n // 2) & (x > n // 3), 900 - 40 * k, v)
    v = np.where((y > n // 2) & (x < n // 3), 60 + 20 * k, v)
    return (v + (x * 7919 + y * 104729 + (x * y) * 31 + k) % 23) / 1024.0


# name: n, PSF, bc, preconditioner, alpha, levels, iterations
CASES = {
    "rect_bccb_slanted_l1": (50, slanted(9), "rect", "bccb", 0.5, 1, 4),
    "rect_ns_rank1_l1": (60, binomial(9), "rect", "tikh_ns", 0.05, 1, 4),
    "rect_krylov_disk_l1": (48, disk(7, 9), "rect", "krylov", 0.05, 1, 3),
    "reflective_krylov_rank1_l2": (54, binomial(5), "reflective", "krylov", 0.05, 2, 3),
    "reflective_ns_rank1_l2": (64, binomial(7), "reflective", "tikh_ns", 0.05, 2, 5),
    "reflective_ns_tall_l1": (97, binomial(37), "reflective", "tikh_ns", 0.05, 1, 3),
    "periodic_tikh_slanted_l4": (81, slanted(5), "periodic", "tikh", 0.05, 4, 3),
    "antireflective_rank1_l3": (58, binomial(9), "antireflective", "tikh", 0.05, 3, 3),
    "zero_sym_disk_l1": (70, disk(9, 13), "zero", "sym", 0.3, 1, 4),
}


def iterate(M, name, **kw):
    n, h, bc, precond, alpha, levels, iters = CASES[name]
    g = image(n, len(name))
    ctx = M.Context(h, n, bc, precond, dtype="f32", z_store="bf16", mu=10.0 / 255.0, alpha=alpha, levels=levels,
                    max_iter=iters + 1, stop=False, rect_ns_hybrid=True, **kw)
    ctx.set_data(g.astype(np.float32), 0.4)
    ctx.iterate(iters)
    f = np.asarray(ctx.result())
    ctx.close()
    return f


def batch(M, names, levels):
    """Several cases of one level count advanced together."""
    probs = []
    for name in names:
        n, h, bc, precond, alpha, lev, iters = CASES[name]
        assert lev == levels
        probs.append(dict(psf=h, g=image(n, len(name)).astype(np.float32), delta=0.4, bc=bc, precond=precond,
                          mu=10.0 / 255.0, alpha=alpha, max_iter=iters))
    b = M.Batch(probs, dtype="f32", z_store="bf16", levels=levels, stop=False, rect_ns_hybrid=True)
    b.iterate(max(CASES[name][6] for name in names))
    out = [np.asarray(b.result(i)) for i in range(len(names))]
    b.close()
    return out


@pytest.fixture(scope="module")
def M():
    from paper_1504_07234_gb300.build import build
    build()
    import paper_1504_07234_gb300 as mod
    return mod


@pytest.fixture(scope="module")
def golden():
    return np.load(GOLDEN)


@pytest.mark.parametrize("name", sorted(CASES))
def test_bf16_iterates(M, golden, name):
    assert np.array_equal(iterate(M, name), golden[name])


@pytest.mark.parametrize("shape", range(8))
def test_bf16_iterates_of_every_tile_shape(M, golden, shape):
    for name in ("rect_ns_rank1_l1", "reflective_ns_rank1_l2"):
        assert np.array_equal(iterate(M, name, frame_shape=shape), golden[name])


def test_bf16_iterates_persistent(M, golden):
    for name in ("rect_ns_rank1_l1", "reflective_ns_rank1_l2", "rect_bccb_slanted_l1"):
        assert np.array_equal(iterate(M, name, persistent=1), golden[name])


def test_bf16_iterates_in_a_batch(M, golden):
    """Other problems beside it (two groups, fuller launches) change no bit."""
    names = [k for k in sorted(CASES) if CASES[k][5] == 1]
    for name, f in zip(names * 12, batch(M, names * 12, 1)):
        assert np.array_equal(f, golden[name]), name
