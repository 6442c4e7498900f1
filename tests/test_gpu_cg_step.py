"""The CG step's forms agree: a few right-hand sides (a cluster of blocks per
RHS, the projection inside the step, the loop control by the step's last
cluster) against many (projection GEMMs, separate loop control), on row lengths
that take one block to the largest cluster.
"""
import numpy as np
import pytest

from gpu_common import lib_ready, need_gpu, rel

pytestmark = pytest.mark.gpu

# Both solves end at ||b - A x|| <= 1e-10 ||b||, so their solutions differ by at
# most 2e-10 E_max / (eps_{n_ext} - eps_v) of the norm; the spectra of these
# systems (E_max 5 Ha, 20 mHa and more above the deflated states) leave 1e-7.
TOL = 1e-7


def _system(grid, n_occ):
    import synthetic
    if grid == 24:
        return synthetic.make_system("tiny")
    return next(s for s in synthetic.make_batch() if s.grid[0] == grid and s.n_occ == n_occ)


# rows of 799 (one block), 1 935, 3 887, 6 859 and 16 375 coefficients
@pytest.mark.parametrize("grid,n_occ", [(24, 8), (32, 17), (40, 17), (48, 12), (64, 9)])
@pytest.mark.parametrize("prec", ["fp64", "mixed"])
def test_few_against_many(grid, n_occ, prec):
    need_gpu()
    lib_ready()
    import paper_1501_03141_gb300 as pg
    s = _system(grid, n_occ)
    p = pg.PDEP_FP64 if prec == "fp64" else pg.PDEP_MIXED
    with pg.Context(s, precision=p, autotune=0) as ctx:
        n = 1024 // s.n_occ + 1  # more than 1024 right-hand sides
        phi = np.random.default_rng(3).standard_normal((n, ctx.sizes()["n_pdep_dim"]))
        many = ctx.chi0_apply(phi)
        it_many = ctx.stats()["cg_iterations_max"]
        for j in (0, n - 1):
            few = ctx.chi0_apply(phi[j:j + 1])
            assert rel(few[0], many[j]) < TOL
            assert ctx.stats()["cg_iterations_max"] <= it_many + 3
        middle = ctx.chi0_apply(phi[:n - 1])  # at most 1024: loop control in the step
        assert rel(middle, many[:n - 1]) < TOL
