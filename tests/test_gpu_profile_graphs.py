"""The profile sees the projections and the CG step that run inside graphs: the
same launches' work as the host loop's, which is timed kernel by kernel."""
import numpy as np
import pytest

import synthetic
from gpu_common import lib_ready, need_gpu, rel

pytestmark = pytest.mark.gpu


# 1040 RHS (streamed step) and 480 (a step per cluster, not timed in graphs), with
# either tensor-core kernel; solves cut short by their caps, so that both forms
# do the same steps
@pytest.mark.parametrize("variant", [1, 2])
@pytest.mark.parametrize("n", [60, 130])
def test_graph_profile_equals_host_loop(variant, n):
    need_gpu()
    lib_ready()
    import paper_1501_03141_gb300 as pg
    work, results = {}, {}
    for use_graph in (0, 1):
        with pg.Context(synthetic.make_system("tiny"), precision=pg.PDEP_MIXED, autotune=0,
                        use_graph=use_graph, proj_variant=variant, max_refine=2,
                        inner_max_iter=5) as ctx:
            phi = np.random.default_rng(3).standard_normal((n, ctx.sizes()["n_pdep_dim"]))
            for _ in range(2):  # the first call's later rounds may still grow the workspace
                ctx.chi0_apply(phi, allow_unconverged=True)
            for _ in range(2):  # a second profile starts from nothing
                pg.profile_start()
                results[use_graph] = ctx.chi0_apply(phi, allow_unconverged=True)
                work[use_graph] = pg.profile_stop()["classes"]
            captures = ctx.graph_captures()
            ctx.chi0_apply(phi, allow_unconverged=True)  # the graphs without timers are kept
            assert ctx.graph_captures() == captures
    assert rel(results[1], results[0]) < 1e-7
    for name in ("gemm_tf32x3", "cg_f32") if n == 130 else ("gemm_tf32x3",):
        host, graph = work[0][name], work[1][name]
        assert graph["launches"] == host["launches"] > 0
        assert graph["flops"] == pytest.approx(host["flops"], rel=1e-9)
        assert graph["bytes"] == pytest.approx(host["bytes"], rel=1e-9)
        # the host's events take in what lies between launches, some 10 us each
        assert 0 < graph["ms"] < 2 * host["ms"]
