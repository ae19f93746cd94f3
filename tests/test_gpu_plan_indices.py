"""A plan's variant indices name the same shapes from version to version (double precision up to
256^2, where the default shape is not the first of the list it was added to)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def T():
    from paper_2304_03306_gb300 import build, ttsh
    build.build()
    ttsh.load_library()
    return ttsh


# index -> (rows per block, points per thread) of the row pass, index -> points of the column pass
ROWS = {1: (1, 8), 2: (1, 4)}
COLS = {1: 4}


@pytest.mark.parametrize("n", [64, 128, 256, 512])
def test_double_indices(T, n):
    d = T.Domain(np.zeros((n, n), np.uint8), n, 20.48 / n, precision=64)
    fresh = d.plan()
    assert (fresh["row_variant"], fresh["col_variant"]) == (0, 0)
    for i, shape in ROWS.items():
        d.set_plan(i, 0)
        p = d.plan()
        assert (p["rows_per_block"], p["row_points_per_thread"]) == shape, i
    for i, points in COLS.items():
        d.set_plan(0, i)
        assert d.plan()["col_points_per_thread"] == points, i
    # every shape is still there
    shapes, points = set(), set()
    for i in range(fresh["n_row_variants"]):
        d.set_plan(i, 0)
        shapes.add((d.plan()["rows_per_block"], d.plan()["row_points_per_thread"]))
    for i in range(fresh["n_col_variants"]):
        d.set_plan(0, i)
        points.add(d.plan()["col_points_per_thread"])
    assert shapes == {(2, 8), (1, 8), (1, 4)} and points == {8, 4}
    d.close()


@pytest.mark.parametrize("n", [64, 128])
def test_autotuner_names_a_shape_by_its_first_index(T, n):
    """A tuned domain of the default shape keeps entry 0, with which a batch steps persistently."""
    for _ in range(4):
        d = T.Domain(np.zeros((n, n), np.uint8), n, 20.48 / n, precision=64)
        plan = d.autotune(iters=4)
        assert plan["row_variant"] != 2 and plan["col_variant"] != 1, plan
        d.close()
