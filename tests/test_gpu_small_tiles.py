"""The small-grid tiles (8 x 4, 8 x 2) and the 16 x 15 tile, whose slopes are handed out field pair
by field pair: bit for bit the 32 x 8 tile's states at the edges of the tiles, for both geometries
and both precisions, and refused on grids beyond their range."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from synth import cases


@pytest.fixture(scope="module")
def P():
    import paper_2504_20742_gb300 as P
    return P


def _shapes(P, prec):
    return [k for k in range(P.ct_tile_shape_count())
            if P.ct_tile_shape(k) in ((8, 4), (8, 2), (16, 15)) and P.ct_tile_shape_ctas(k, prec)]


def _run(P, c, uf, prec, shape, steps):
    P.ct_set_tile_shape(c, prec, shape)
    s = P.Solver(c, uf, precision=prec)
    s.init_state(0.5)
    s.step(steps, 0.5)
    d = s.diagnostics()
    P.ct_set_tile_shape(c, prec, -1)
    return s.U.clone(), d


@pytest.mark.gpu
@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("nx,nr", [(4, 2), (7, 3), (8, 4), (9, 5), (16, 15), (17, 16), (33, 31), (100, 44), (400, 1), (13, 1)])
def test_same_bits_as_the_default_tile(P, prec, nx, nr):
    if nr == 1:
        c, uf = cases.nozzle_case(nx=nx), None
    else:
        c, uf = cases.mixing_layer_case(nx=nx, nr=nr)
        c = dict(c, wall_len=2.0)
    ref, d0 = _run(P, c, uf, prec, 0, 5)
    assert d0[8] == 0
    bits = torch.int64 if prec == 0 else torch.int32
    for k in _shapes(P, prec) + [-1]:      # -1: the default of this grid
        U, d = _run(P, c, uf, prec, k, 5)
        assert torch.equal(U.view(bits), ref.view(bits)), (k, prec)
        assert d[0] == d0[0] and d[7] == d0[7] and np.array_equal(d[9:23], d0[9:23])
        for q in (1, 2, 3):                # totals: sums in another order, in FP32 within a warp
            assert abs(d[q] - d0[q]) <= (1e-12 if prec == 0 else 1e-5) * abs(d0[q])


@pytest.mark.gpu
@pytest.mark.parametrize("opt", [dict(tables=1), dict(equilibrium=1), dict(phase_change=0), dict(freezing=0), dict(viscous=1, nu_t=0.05),
                                 dict(n_soot=0.0)])
@pytest.mark.parametrize("nx,nr", [(33, 31), (9, 5), (64, 24)])
def test_same_bits_with_the_model_options(P, nx, nr, opt):
    """The source's shares of the small FP64 tiles and the totals in one level (up to 64 tiles) or two."""
    c, uf = cases.mixing_layer_case(nx=nx, nr=nr)
    c = dict(c, **opt)
    ref, d0 = _run(P, c, uf, 0, 0, 5)
    for k in _shapes(P, 0):
        U, d = _run(P, c, uf, 0, k, 5)
        assert torch.equal(U.view(torch.int64), ref.view(torch.int64)), k
        assert d[0] == d0[0] and d[7] == d0[7] and np.array_equal(d[9:25], d0[9:25])
        for q in (1, 2, 3):
            assert abs(d[q] - d0[q]) <= 1e-12 * abs(d0[q])


def test_small_tiles_are_refused_on_large_grids(P):
    c, _ = cases.plume_case(nx=512, nr=128)
    small = [k for k in range(P.ct_tile_shape_count()) if P.ct_tile_shape(k) in ((8, 4), (8, 2))]
    assert len(small) == 2
    for k in small:
        for prec in (P.CT_FP64, P.CT_FP32):
            with pytest.raises(P.ContrailError):
                P.ct_set_tile_shape(c, prec, k)
            P.ct_set_tile_shape(dict(c, nx=64, nr=32), prec, k)
            P.ct_set_tile_shape(dict(c, nx=64, nr=32), prec, -1)
