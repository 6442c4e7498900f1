"""Calls that work on the caller's device arrays in place of staged copies: the
same results whatever the arrays' place, alignment and overlap."""
import numpy as np
import pytest
import torch

import synthetic
from gpu_common import lib_ready, need_gpu, rel

pytestmark = pytest.mark.gpu

# the same kernels on the same values; screening sums its K splits by FP64
# atomics in any order: 60 additions of 1.1e-16
TOL_H, TOL_SCREEN = 1e-15, 1e-14


def _dev(x, offset):
    """x on the device, 'offset' doubles past an allocation's start"""
    buf = torch.empty(x.size + offset, dtype=torch.float64, device="cuda")
    v = buf[offset:].view(x.shape)
    v.copy_(torch.from_numpy(x))
    return v


def _forms(f, x, shape):
    """results of f(x, out) over the forms of x and out"""
    yield f(_dev(x, 0), torch.empty(shape, dtype=torch.float64, device="cuda"))
    yield f(_dev(x, 1), _dev(np.zeros(shape), 1))
    yield f(x, torch.empty(shape, dtype=torch.float64, device="cuda"))
    yield f(_dev(x, 0), np.empty(shape))
    if tuple(shape) == x.shape:
        inplace = _dev(x, 0)
        yield f(inplace, inplace)
        rows = torch.empty((x.shape[0] + 1, x.shape[1]), dtype=torch.float64, device="cuda")
        rows[:-1].copy_(torch.from_numpy(x))
        yield f(rows[:-1], rows[1:])


def _np(t):
    return t.cpu().numpy() if isinstance(t, torch.Tensor) else t


@pytest.mark.parametrize("name", ["tiny", "cube48"])
def test_h_and_grid(name):
    need_gpu()
    lib_ready()
    import paper_1501_03141_gb300 as pg
    with pg.Context(synthetic.make_system(name)) as ctx:
        sz = ctx.sizes()
        x = np.random.default_rng(1).standard_normal((3, sz["n_pw"]))
        for prec in (pg.PDEP_FP64, pg.PDEP_MIXED, pg.PDEP_APPLY_DF64):
            ref = ctx.apply_hamiltonian(x, precision=prec)
            for y in _forms(lambda a, o: ctx.apply_hamiltonian(a, precision=prec, out=o), x, x.shape):
                assert rel(_np(y), ref) < TOL_H
        ref = ctx.to_grid(x).reshape(3, -1)
        for y in _forms(lambda a, o: ctx.to_grid(a, out=o), x, (3, sz["n_r"])):
            assert rel(_np(y), ref) < TOL_H


@pytest.mark.parametrize("kind", ["chibar", "epsinv", "wp"])
def test_screening(kind):
    need_gpu()
    lib_ready()
    import paper_1501_03141_gb300 as pg
    with pg.Context(synthetic.make_system("tiny")) as ctx:
        dim = ctx.sizes()["n_pdep_dim"]
        rng = np.random.default_rng(2)
        vec = np.ascontiguousarray(np.linalg.qr(rng.standard_normal((dim, 9)))[0].T)
        val = -rng.uniform(0.1, 2.0, 9)
        f = rng.standard_normal((5, dim))
        ref = ctx.screening_apply(kind, val, vec, f)
        for off in (0, 1):
            v = _dev(vec, off)
            for y in _forms(lambda a, o: ctx.screening_apply(kind, val, v, a, out=o), f, f.shape):
                assert rel(_np(y), ref) < TOL_SCREEN


# Lambda = (1 - B)^{-1} B from the eigenpairs of B, over the sizes where the
# Jacobi solver changes its threads, columns per thread and pairing; its
# eigenpairs are good to some n eps of ||B||, and 1 - B has no eigenvalue below 1
@pytest.mark.parametrize("n", [1, 2, 3, 64, 65, 128, 129, 257, 513, 769])
def test_eigenproblem_sizes(n):
    need_gpu()
    lib_ready()
    import paper_1501_03141_gb300 as pg
    with pg.Context(synthetic.make_system("tiny")) as ctx:
        dim = ctx.sizes()["n_pdep_dim"]
        rng = np.random.default_rng(n)
        phi = np.ascontiguousarray(np.linalg.qr(rng.standard_normal((dim, n)))[0].T)
        B, L = ctx.chi0_imag(phi, [0.3], n_steps=3)
        assert rel(L[0], np.linalg.solve(np.eye(n) - B[0], B[0])) < 1e-11
