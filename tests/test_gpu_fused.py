"""FP32 H x in one launch (a line per thread, 24^3 .. 48^3): against FP64, on
either side of the item count from which it is used, an odd last vector, more
items than SMs, and spheres below the largest."""

import numpy as np
import pytest

import synthetic
from gpu_common import lib_ready, need_gpu, rel

pytestmark = pytest.mark.gpu

# FP32 line transforms of at most 3 log2(48) rounded steps, with the products
# of the potential and the sums: the 2e-7 the three-launch form is held to
TOL = 2e-7


def _system(n, cell):
    rng = np.random.default_rng(n)
    c, d, w = synthetic.gaussian_wells(rng, 4, cell, (1.0, 3.0), (0.8, 1.5))
    v = synthetic.periodic_gaussian_sum((n,) * 3, cell, c, d, w)
    return synthetic.System(name="t", grid=(n,) * 3, cell=cell, v_r=v, n_occ=2, n_pdep=2, seed=n)


@pytest.mark.parametrize("grid", [24, 32, 40, 48])
@pytest.mark.parametrize("shape", ["cube", "flat", "low"])
def test_fused_h_matches_fp64(grid, shape):
    need_gpu()
    lib_ready()
    import paper_1501_03141_gb300 as pg
    side = 0.42 * grid
    cell = (side, 1.3 * side, 0.8 * side) if shape == "flat" else (side,) * 3
    # "low": three frequencies below the largest sphere on each axis
    ecut = 0.5 * (2 * np.pi / side * (grid / 4 - 3.5)) ** 2 if shape == "low" else 0.0
    s = _system(grid, cell)
    rng = np.random.default_rng(7)
    with pg.Context(s, ecut=ecut) as ctx, pg.Context(s, ecut=ecut, fused_hpsi=0) as plain:
        for n in (1, 76, 77, 152, 153, 311):
            x = rng.standard_normal((n, ctx.sizes()["n_pw"]))
            ref = ctx.apply_hamiltonian(x)
            one = ctx.apply_hamiltonian(x, precision=pg.PDEP_MIXED)
            three = plain.apply_hamiltonian(x, precision=pg.PDEP_MIXED)
            for j in {0, n // 2, max(n - 2, 0), n - 1}:
                assert rel(one[j], ref[j]) < TOL and rel(one[j], three[j]) < 2 * TOL
            assert rel(one, ref) < TOL
