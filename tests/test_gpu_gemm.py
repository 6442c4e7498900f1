"""FP64 products on the FP16 tensor cores (exact integer digits), through
pdep_screening_apply: out = Phi diag(g) (Phi^T f) is one product over the
plane waves and one over the eigenpairs.  The reference is the same sum in
numpy's long double.
"""
import numpy as np
import pytest

from gpu_common import lib_ready, need_gpu

pytestmark = pytest.mark.gpu

# Each output is a sum of at most 54 split-K partial results, each rounded to
# FP64 once (2^-53 relative), the operands held to 2^-62 of their row's largest
# value: 54 x 2^-53 = 6e-15 of the norm bounds either product.
TOL = 2 * 6e-15


@pytest.fixture(scope="module")
def ctx():
    need_gpu()
    lib_ready()
    import paper_1501_03141_gb300 as pg
    import synthetic
    with pg.Context(synthetic.make_system("tiny")) as c:
        yield c


def _inputs(dim, n_pdep, n, decay, seed):
    rng = np.random.default_rng(seed)
    w = np.exp(-decay * np.arange(dim) / dim)
    vec = np.linalg.qr((rng.standard_normal((n_pdep, dim)) * w).T)[0].T.copy()
    return -np.linspace(3.0, 0.01, n_pdep), vec, rng.standard_normal((n, dim)) * w


def _reference(val, vec, f):
    val, vec, f = (np.asarray(a, dtype=np.longdouble) for a in (val, vec, f))
    return ((f @ vec.T) * (val / (1 - val))) @ vec


# one output, tile edges (32 x 32), remainders, more than one tile; flat
# vectors and ones that fall by 26 orders of magnitude over their length
@pytest.mark.parametrize("n_pdep,n", [(1, 1), (7, 33), (31, 2), (32, 32), (33, 31), (129, 65)])
@pytest.mark.parametrize("decay", [0.0, 60.0])
def test_product_against_long_double(ctx, n_pdep, n, decay):
    val, vec, f = _inputs(ctx.sizes()["n_pdep_dim"], n_pdep, n, decay, 11)
    out = ctx.screening_apply("chibar", val, vec, f)
    ref = _reference(val, vec, f)
    err = np.linalg.norm((out - ref).astype(float)) / np.linalg.norm(ref.astype(float))
    assert err < TOL, err


def test_scales_far_apart(ctx):
    # columns of very different size keep their own relative accuracy; zero
    # and subnormal entries stay harmless
    val, vec, f = _inputs(ctx.sizes()["n_pdep_dim"], 40, 6, 0.0, 12)
    f *= np.array([1.0, 1e-200, 1e200, 0.0, 1e-12, 1e-310])[:, None]
    out, ref = ctx.screening_apply("chibar", val, vec, f), _reference(val, vec, f)
    for j in (0, 1, 2, 4):
        err = np.linalg.norm(((out[j] - ref[j]) / np.abs(ref[j]).max()).astype(float))
        assert err / np.linalg.norm((ref[j] / np.abs(ref[j]).max()).astype(float)) < TOL, (j, err)
    assert np.all(out[3] == 0.0)
    assert np.all(np.abs(out[5]) < 1e-305)


@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_nonfinite_input_stays_in_its_column(ctx, bad):
    val, vec, f = _inputs(ctx.sizes()["n_pdep_dim"], 40, 5, 0.0, 13)
    f[2, 100] = bad
    out = ctx.screening_apply("chibar", val, vec, f)
    good = [0, 1, 3, 4]
    assert not np.any(np.isfinite(out[2]))
    ref = _reference(val, vec, f[good])
    assert np.linalg.norm((out[good] - ref).astype(float)) / np.linalg.norm(ref.astype(float)) < TOL
