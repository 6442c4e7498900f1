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


# A loop captured while the projection kernels are untimed (fewer than 256 RHS)
# runs the default one, tcgen05 (2): once another system's loop has timed them,
# it is captured again if the choice is another kernel or step shape (0), and
# only then.  The calls before the timing leave it no workspace to grow, which
# would capture every graph again: vectors by the 48^3 system, lists by the
# 24^3 one, whose step adds the projection and times nothing.
def test_graphs_are_keyed_by_the_projection_they_run():
    need_gpu()
    lib_ready()
    import paper_1501_03141_gb300 as pg
    tiny, big = synthetic.make_system("tiny"), synthetic.make_system("cube48")
    mid = next(s for s in synthetic.make_batch() if s.grid[0] == 32 and s.n_occ == 17)
    with pg.Context([tiny, big, mid], precision=pg.PDEP_MIXED, n_deflate=0, fused_hpsi=0) as ctx:
        rng = np.random.default_rng(9)

        def apply(sys, n):
            phi = rng.standard_normal((n, ctx.sizes(sys)["n_pdep_dim"]))
            ctx.chi0_apply(phi, sys=sys)
            return ctx.graph_captures()
        for _ in range(2):
            apply(0, 128)  # 1024 RHS
            apply(1, 3)    # 192 RHS
        before = apply(1, 3)
        st = ctx.stats()
        assert st["proj_variant"] == -1 and st["cg_variant"] == -1
        timed = apply(2, 16)  # 272 RHS
        st = ctx.stats()
        assert st["proj_variant"] >= 0 and st["cg_variant"] >= 0
        after = apply(1, 3)
        print("projection kernel", st["proj_variant"], "step shape", st["cg_variant"], before, timed, after)
        assert (after > timed) == (st["proj_variant"] != 2 or st["cg_variant"] != 0)
