"""fdf_tune times every schedule once: of the sort_tile values, the one that the automatic size
stands for is not timed again."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,n_grid,n_part,tiles", [(1, 32, 4000, 2), (1, 8, 20001, 3), (3, 16, 4000, 2)])
def test_each_bucket_size_is_timed_once(inputs, c1_tables, prec, n_grid, n_part, tiles):
    """Timed runs: the start, sort_cells 5 + 6, steps_per_pass 4, gather_tile 1 (split-state forms) and
    the bucket sizes: 3 beside automatic single cells (39 particles per cell), else 2 (0.1 and 1
    particles per cell: the automatic sizes are 4^3 and 2^3)."""
    from paper_2207_14256_gb300 import build
    from paper_2207_14256_gb300 import fdf as F

    build.build()
    P = F.make_params(inputs.config("c1_32", n_part=n_part, n_grid=n_grid, n_steps=8, precision=prec, seed=7))
    T, keep = F.make_tables(c1_tables)
    tuned, ms, trials = F.fdf_tune(P, T)
    assert trials == 1 + 5 + tiles + 4 + (1 if prec == 3 else 0) + 6
