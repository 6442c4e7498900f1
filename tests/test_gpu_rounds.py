"""Refinement rounds inside one graph against the host loop: one round, as many
as are needed, fewer than are needed, and solves that differ in how many they
need."""
import numpy as np
import pytest

import synthetic
from gpu_common import lib_ready, need_gpu, rel

pytestmark = pytest.mark.gpu


# Both end at ||b - A x|| <= 1e-10 ||b||; this system's spectrum leaves 1e-7 of
# the solution (a solve cut short is compared by its status and round count).
@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("kw", [{}, {"max_refine": 1}, {"max_refine": 2}, {"inner_tol": 2e-2}])
@pytest.mark.parametrize("n", [1, 40])
def test_rounds_graph_equals_host_loop(prec, kw, n):
    need_gpu()
    lib_ready()
    import paper_1501_03141_gb300 as pg
    s = synthetic.make_system("tiny")
    p = pg.PDEP_FP64 if prec == "fp64" else pg.PDEP_MIXED
    got = []
    for use_graph in (0, 1):
        with pg.Context(s, precision=p, use_graph=use_graph, autotune=0, **kw) as ctx:
            rng = np.random.default_rng(5)
            phi = rng.standard_normal((n, ctx.sizes()["n_pdep_dim"]))
            w = ctx.chi0_apply(phi, allow_unconverged=True)
            again = ctx.chi0_apply(phi, allow_unconverged=True)
            st = ctx.stats()
            got.append((w, again, st))
    (a, a2, sa), (b, b2, sb) = got
    assert sa["refine_rounds_max"] == sb["refine_rounds_max"] >= 1
    if sa["max_cg_residual"] <= 1e-10:
        assert sb["max_cg_residual"] <= 1e-10
        assert rel(b, a) < 1e-7 and rel(a2, a) < 1e-7 and rel(b2, b) < 1e-7
    else:  # stopped after the first round(s): one FP32 solve's accuracy
        assert sb["max_cg_residual"] > 1e-10 and rel(b, a) < 1e-2


# PDEP_MIXED_BF16 never times the FP32 projection kernels in its CG loops, so its
# refinement rounds are captured while those are untimed; accurate to the same
# residual as above
def test_rounds_graph_bf16_untimed():
    need_gpu()
    lib_ready()
    import paper_1501_03141_gb300 as pg
    s = synthetic.make_system("tiny")
    got = []
    for use_graph in (0, 1):
        with pg.Context(s, precision=pg.PDEP_MIXED_BF16, use_graph=use_graph) as ctx:
            phi = np.random.default_rng(6).standard_normal((160, ctx.sizes()["n_pdep_dim"]))
            for _ in range(3):
                w = ctx.chi0_apply(phi)
            got.append(w)
            assert ctx.stats()["max_cg_residual"] <= 1e-10
    assert rel(got[1], got[0]) < 1e-7
