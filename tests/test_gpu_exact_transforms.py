"""FP64 transforms by exact digit products on the tensor cores: to_grid and H x
against numpy FFTs in long double, on every grid shape, with odd vector
counts, vectors of very different size in one packed pair, a sphere smaller
than the grid allows, the ends of the exponent range and non-finite input.
"""
import numpy as np
import pytest

from gpu_common import lib_ready, need_gpu

pytestmark = pytest.mark.gpu

GRIDS = [((n, n, n), (n * 10.0 / 24.0,) * 3) for n in (24, 32, 40, 48, 64)]
GRIDS += [((64, 64, 192), (20.0, 20.0, 60.0)), ((40, 24, 24), (17.0, 10.0, 10.0))]
EPS = 2.0 ** -53
# Six passes round at 2^-58 of a pass's largest value, which is below 2^5 of its
# root mean square for these vectors: 6 x 2^-53, and as much for the FP64 numbers
# between the passes and the epilogue's three roundings.
TOL = 12 * EPS
# Seven digits round at 2^-53 of the largest value instead: 6 x 2^-48.
TOL_REFINE = 6 * 2.0 ** -48


class _Sphere:
    def __init__(self, grid, cell, ecut):
        lim = [(n - 1) // 2 for n in grid]
        ns = np.meshgrid(*[np.arange(-m, m + 1) for m in lim], indexing="ij")
        n = np.stack([a.ravel() for a in ns], axis=1)
        g2 = ((2 * np.pi * n / np.asarray(cell)) ** 2).sum(axis=1)
        if not ecut:
            ecut = 0.5 * min(2 * np.pi * ((m - 1) / 4.0) / l for m, l in zip(grid, cell)) ** 2
        half = (0.5 * g2 <= ecut) & ((n[:, 2] > 0) | ((n[:, 2] == 0) & (
            (n[:, 1] > 0) | ((n[:, 1] == 0) & (n[:, 0] > 0)))))
        order = np.lexsort((n[half, 0], n[half, 1], n[half, 2]))
        self.grid, self.n, self.g2 = grid, n[half][order], g2[half][order]

    def to_grid(self, x):
        x = np.asarray(x, dtype=np.longdouble)
        f = np.zeros((x.shape[0],) + self.grid, dtype=np.clongdouble)
        c = (x[:, 0:-1:2] + 1j * x[:, 1:-1:2]) / np.sqrt(np.longdouble(2))
        n = self.n
        f[:, n[:, 0], n[:, 1], n[:, 2]] = c
        f[:, -n[:, 0], -n[:, 1], -n[:, 2]] = c.conj()
        f[:, 0, 0, 0] = x[:, -1]
        return np.fft.ifftn(f, axes=(1, 2, 3), norm="forward").real

    def h(self, v, x):
        f = np.fft.fftn(self.to_grid(x) * v.astype(np.longdouble), axes=(1, 2, 3), norm="forward")
        n, y = self.n, np.empty(x.shape, dtype=np.longdouble)
        c = f[:, n[:, 0], n[:, 1], n[:, 2]] * np.sqrt(np.longdouble(2))
        y[:, 0:-1:2], y[:, 1:-1:2], y[:, -1] = c.real, c.imag, f[:, 0, 0, 0].real
        kin = np.append(np.repeat(0.5 * self.g2, 2), 0.0)
        return y + kin.astype(np.longdouble) * x


def _context(grid, cell, ecut=0.0):
    need_gpu()
    lib_ready()
    import paper_1501_03141_gb300 as pg
    import synthetic
    rng = np.random.default_rng(21)
    c, d, w = synthetic.systems.gaussian_wells(rng, 6, cell, (1.0, 3.0), (0.8, 1.5))
    v = synthetic.systems.periodic_gaussian_sum(grid, cell, c, d, w)
    s = synthetic.systems.System("t", grid, cell, v, 2, 2, 0)
    return pg.Context(s, ecut=ecut, gap_min=0.0, n_deflate=0), _Sphere(grid, cell, ecut), v


def _rel(a, b):
    d = (np.asarray(a, dtype=np.longdouble) - b).reshape(len(b), -1)
    scale = np.abs(b).reshape(len(b), -1).max(axis=1)
    d, b = d / scale[:, None], b.reshape(len(b), -1) / scale[:, None]
    return [float(np.sqrt(float((x * x).sum() / (y * y).sum()))) for x, y in zip(d, b)]


@pytest.mark.parametrize("grid,cell", GRIDS)
@pytest.mark.parametrize("n,decay", [(1, 0.0), (3, 6.0)])
def test_against_long_double(grid, cell, n, decay):
    import paper_1501_03141_gb300 as pg
    ctx, sp, v = _context(grid, cell)
    with ctx:
        rng = np.random.default_rng(n)
        x = rng.standard_normal((n, 2 * len(sp.g2) + 1))
        x *= np.append(np.repeat(np.exp(-decay * sp.g2 / sp.g2.max()), 2), 1.0)
        assert max(_rel(ctx.to_grid(x).reshape((n,) + grid), sp.to_grid(x))) < TOL
        ref = sp.h(v, x)
        assert max(_rel(ctx.apply_hamiltonian(x), ref)) < TOL
        assert max(_rel(ctx.apply_hamiltonian(x, precision=pg.PDEP_APPLY_DF64), ref)) < TOL_REFINE


def test_small_sphere_scales_and_nonfinite():
    grid, cell = (32, 32, 32), (32 * 10.0 / 24.0,) * 3
    ctx, sp, v = _context(grid, cell, ecut=2.0)   # the sphere fills a part of the tables
    with ctx:
        rng = np.random.default_rng(5)
        x = rng.standard_normal((8, 2 * len(sp.g2) + 1))
        # pairs: (1e-9, 1), (1e150, 1e150), (1e-290, 1e-290), (0, 0)
        x *= np.array([1e-9, 1.0, 1e150, 1e150, 1e-290, 1e-290, 0.0, 0.0])[:, None]
        ref, out = sp.h(v, x), ctx.apply_hamiltonian(x)
        err = _rel(out[1:6], ref[1:6])
        assert max(err) < TOL, err
        # the small vector of a pair carries the other one's rounding, as in any
        # transform of a + i b
        assert _rel(out[:1], ref[:1])[0] < 1e9 * TOL
        assert np.all(out[6:] == 0.0)
        x[1, 7], x[4, 3] = np.nan, np.inf
        out = ctx.apply_hamiltonian(x)
        assert not np.any(np.isfinite(out[[1, 4]]))
        assert np.all(np.isfinite(out[[2, 3, 6, 7]]))
        assert max(_rel(out[2:4], ref[2:4])) < TOL
        u = ctx.to_grid(x)
        assert not np.any(np.isfinite(u[[1, 4]])) and np.all(np.isfinite(u[[2, 3, 6, 7]]))
