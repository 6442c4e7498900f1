"""kernel_launches counts what ran inside graphs: every launch of a pass of a
while node, those of steps that found nothing to do among them, by the graph it
ran in.  Loops cut short by their caps make the counts exact."""
import numpy as np
import pytest

import synthetic
from gpu_common import lib_ready, need_gpu

pytestmark = pytest.mark.gpu


def _count(ctx, n):
    phi = np.random.default_rng(n).standard_normal((n, ctx.sizes()["n_pdep_dim"]))
    ctx.chi0_apply(phi, allow_unconverged=True)
    st = ctx.stats()
    return st["kernel_launches"], st


# an FP32 pass holds four steps, so one step and four are the same launches
def test_steps_after_the_last_one_are_counted():
    need_gpu()
    lib_ready()
    import paper_1501_03141_gb300 as pg
    got = {}
    for cap in (1, 4, 5, 8):
        with pg.Context(synthetic.make_system("tiny"), precision=pg.PDEP_MIXED, autotune=0,
                        max_refine=2, inner_max_iter=cap) as ctx:
            got[cap], st = _count(ctx, 3)
            assert st["refine_rounds_max"] == 2 and st["cg_iterations_max"] == cap
    assert got[1] == got[4] < got[5] == got[8]


# a call in two chunks runs what its chunks run as calls of their own: more than
# 1024 RHS and then 16, whose steps are other kernels
@pytest.mark.parametrize("prec", ["fp64", "mixed"])
def test_chunks_of_different_steps(prec):
    need_gpu()
    lib_ready()
    import paper_1501_03141_gb300 as pg
    p = pg.PDEP_FP64 if prec == "fp64" else pg.PDEP_MIXED
    with pg.Context(synthetic.make_system("tiny"), precision=p, autotune=0, max_refine=2,
                    inner_max_iter=3, cg_max_iter=3, workspace_limit_bytes=272 << 20) as ctx:
        most = next(n for n in range(129, 300) if _count(ctx, n + 1)[1]["chi0_chunks"] == 2)
        assert _count(ctx, most)[1]["chi0_chunks"] == 1
        assert _count(ctx, most + 2)[0] == _count(ctx, most)[0] + _count(ctx, 2)[0]
