"""FP64 products of the caller's own numbers (pdep_screening_apply) where the
large entries of one factor meet the small ones of the other: accurate relative
to the sum of the products' magnitudes, as FP64 multiply-adds are, and not only
to the factors' largest entries.  The reference is numpy's long double.
"""
import numpy as np
import pytest

import synthetic
from gpu_common import lib_ready, need_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    need_gpu()
    lib_ready()
    import paper_1501_03141_gb300 as pg
    with pg.Context(synthetic.make_system("tiny")) as c:
        yield c


def _check(ctx, val, vec, f, kind="chibar"):
    out = ctx.screening_apply(kind, val, vec, f)
    v, p, x = (np.asarray(a, dtype=np.longdouble) for a in (val, vec, f))
    g = v / (1 - v)
    ref = ((x @ p.T) * g) @ p
    size = ((np.abs(x) @ np.abs(p.T)) * np.abs(g)) @ np.abs(p)
    if kind == "epsinv":
        ref, size = ref + x, size + np.abs(x)
    # Per product, a kept digit sum errs by K 2^-56.8 A B (A, B: the largest
    # magnitudes) with sum |a b| >= 2^-5 A B, a recomputed one by K 2^-53 sum |a b|:
    # K 2^-51.8 either way; K = dim, then n_pdep
    tol = (vec.shape[1] + vec.shape[0]) * 2.0 ** -51
    err = np.abs((out - ref).astype(float))
    assert np.all(err <= tol * size.astype(float)), (err / size.astype(float)).max() / tol


def test_two_entries(ctx):
    dim = ctx.sizes()["n_pdep_dim"]
    vec, f = np.zeros((1, dim)), np.zeros((1, dim))
    vec[0, :2] = 1.0, 2.0 ** -70
    f[0, :2] = 2.0 ** -70, 1.0
    _check(ctx, np.array([-1.0]), vec, f)


# K over one stage, a remainder and several splits of the plane waves; rows past
# a tile; n_pdep short and long for the second product
@pytest.mark.parametrize("n_pdep,n", [(1, 1), (8, 3), (33, 34), (129, 7)])
@pytest.mark.parametrize("decay", [0.0, 15.0, 45.0])
def test_opposite_along_the_plane_waves(ctx, n_pdep, n, decay):
    dim = ctx.sizes()["n_pdep_dim"]
    rng = np.random.default_rng(21)
    w = np.exp(-decay * np.arange(dim) / dim)
    vec = rng.standard_normal((n_pdep, dim)) * w
    f = rng.standard_normal((n, dim)) * w[::-1]
    _check(ctx, -np.linspace(3.0, 0.01, n_pdep), vec, f)


# one vector of each kind in a tile, zeros among them
@pytest.mark.parametrize("kind", ["chibar", "epsinv"])
def test_mixed_tile(ctx, kind):
    dim = ctx.sizes()["n_pdep_dim"]
    rng = np.random.default_rng(22)
    w = np.exp(-50.0 * np.arange(dim) / dim)
    vec, f = rng.standard_normal((3, 20, dim)), rng.standard_normal((4, 5, dim))
    vec = np.concatenate([vec[0] * w, vec[1], vec[2] * w[::-1]])
    f = np.concatenate([f[0] * w, f[1], f[2] * w[::-1], f[3] * 0.0])
    vec[:, rng.integers(0, dim, dim // 3)] = 0.0
    _check(ctx, -np.linspace(3.0, 0.01, 60), vec, f, kind)


# the second product: vectors of falling size, eigenvalues that rise
def test_opposite_along_the_eigenpairs(ctx):
    dim = ctx.sizes()["n_pdep_dim"]
    rng = np.random.default_rng(23)
    scale = np.exp2(-np.arange(40.0))
    vec = rng.standard_normal((40, dim)) * scale[:, None]
    _check(ctx, -np.exp2(-80.0 + 2.0 * np.arange(40)), vec, rng.standard_normal((5, dim)))
