"""Which tile an FP64 step takes where no shape is registered: the small tiles only where they are the
faster ones (a nozzle of more than some 900 cells, and long or flat plumes, step faster through 32 x 8
tiles).  The totals of a step are summed tile by tile, so their last bits tell the tile."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from synth import cases

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_2504_20742_gb300 as P
    return P


def _totals(P, c, uf, shape):
    P.ct_set_tile_shape(c, 0, shape)
    s = P.Solver(c, uf, precision=0)
    s.init_state(0.5)
    out = []
    for _ in range(4):
        s.step(1, 0.5)
        out.append(s.diagnostics()[1:4].copy())
    P.ct_set_tile_shape(c, 0, -1)
    return np.array(out).view(np.int64)


@pytest.mark.parametrize("nx,nr,tile", [(400, 1, (8, 2)), (912, 1, (8, 2)), (952, 1, (32, 8)), (1600, 1, (32, 8)), (6400, 1, (32, 8)),
                                        (20000, 1, (32, 8)), (96, 40, (8, 2)), (800, 2, (8, 2)), (200, 100, (8, 4)), (300, 68, (8, 4)),
                                        (2000, 8, (32, 8)), (3200, 4, (32, 8)), (5120, 4, (32, 8)), (10240, 2, (32, 8)), (8, 2000, (8, 4))])
def test_default_tile(P, nx, nr, tile):
    c, uf = (cases.nozzle_case(nx=nx), None) if nr == 1 else cases.mixing_layer_case(nx=nx, nr=nr)
    default = _totals(P, c, uf, -1)
    seen = {t: _totals(P, c, uf, [k for k in range(P.ct_tile_shape_count()) if P.ct_tile_shape(k) == t][0])
            for t in ((32, 8), (8, 4), (8, 2))}
    if nr <= 2:
        del seen[(8, 4)]          # up to two rows: the cells, and so the sums, of the 8 x 2 tiles
    assert not any(np.array_equal(a, b) for t, a in seen.items() for u, b in seen.items() if t < u)
    assert np.array_equal(default, seen[tile])
