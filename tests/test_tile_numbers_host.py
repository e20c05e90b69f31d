"""The tile shapes keep their numbers: a caller's program, or a command line, may name one by it."""


def test_numbers_of_the_tile_shapes():
    import paper_2504_20742_gb300 as P
    shapes = [P.ct_tile_shape(k) for k in range(P.ct_tile_shape_count())]
    assert shapes == [(32, 8), (16, 16), (32, 16), (64, 8), (16, 16), (32, 8), (16, 12), (16, 16), (16, 14), (28, 64), (8, 4), (8, 2),
                      (16, 15)]
    assert [P.ct_tile_shape_ctas(k, P.CT_FP64) for k in (6, 7, 8, 12)] == [2, 2, 2, 2]
