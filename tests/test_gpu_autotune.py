"""What the autotuner waits for and what it times."""
import numpy as np
import pytest

import synthetic
from gpu_common import lib_ready, need_gpu, rel

pytestmark = pytest.mark.gpu


# 256 to 417 RHS of 24^3 (8 occupied states): the CG step adds the projection
# itself, so neither the projection kernels nor the step's block shapes are in
# use, and none may be waited for or chosen
@pytest.mark.parametrize("df_refine", [0, 1, 2])
@pytest.mark.parametrize("n", [32, 40, 52])
def test_loop_without_projection_kernels_is_captured(df_refine, n):
    need_gpu()
    lib_ready()
    import paper_1501_03141_gb300 as pg
    s = synthetic.make_system("tiny")
    with pg.Context(s, precision=pg.PDEP_MIXED, df_refine=df_refine) as ctx:
        phi = np.random.default_rng(7).standard_normal((n, ctx.sizes()["n_pdep_dim"]))
        first = ctx.chi0_apply(phi)
        for _ in range(3):
            again = ctx.chi0_apply(phi)
        st = ctx.stats()
        assert st["graph_launches"] > 0
        assert st["proj_variant"] == -1 and st["cg_variant"] == -1
        assert rel(again, first) < 1e-7 and st["max_cg_residual"] <= 1e-10
        # a loop that does use them times them
        many = ctx.chi0_apply(np.random.default_rng(8).standard_normal((100, phi.shape[1])))
        st = ctx.stats()
        assert st["proj_variant"] >= 0 and st["cg_variant"] >= 0 and np.isfinite(many).all()
