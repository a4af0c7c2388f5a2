"""The sort's bucket size (fdf_params.sort_tile): 1, 2 and 3 are the caller's cubes of 2, 4 and 8
cells per axis at any density, 0 is the automatic size.  On the host by the footprint, which holds the
histogram of the buckets; on the GPU by runs of every size, whose particles are the same bit for bit.
"""
import numpy as np
import pytest


def test_explicit_sizes_are_kept(inputs):
    from paper_2207_14256_gb300 import fdf

    # one particle per cell: the automatic size is 4^3 cells in the FP64-state form, 2^3 in the split one
    for prec, same in ((1, 2), (2, 2), (3, 1)):
        b = [fdf.fdf_footprint(fdf.make_params(inputs.config("c1_32", n_part=64 ** 3, n_grid=64, precision=prec,
                                                             sort_tile=t))) for t in range(4)]
        hist = [4 * (64 >> t) ** 3 for t in range(4)]
        # within the scans' totals (a thousandth) and the alignment of the two arrays
        for t in (2, 3):
            assert abs((b[1] - b[t]) - (hist[1] - hist[t])) <= hist[1] / 500 + 1024, (prec, t, b)
        assert b[0] == b[same]


@pytest.fixture(scope="module")
def F():
    from paper_2207_14256_gb300 import build
    from paper_2207_14256_gb300 import fdf

    build.build()
    fdf.lib()
    return fdf


@pytest.mark.gpu
@pytest.mark.parametrize("prec", [0, 1, 3])
@pytest.mark.parametrize("n_grid,n_part", [(8, 20001), (32, 5003)])
def test_runs_do_not_depend_on_the_size(F, inputs, c1_tables, prec, n_grid, n_part):
    """39 particles per cell (automatic: single cells) and 0.15 (4^3 cells)."""
    p = inputs.config("c1_32", n_part=n_part, n_grid=n_grid, n_species=2, m_ev=[0.05, 0.2], n_steps=40, precision=prec,
                      sort_cells=1, seed=61)
    got = []
    for t in range(4):
        with F.Run(dict(p, sort_tile=t), c1_tables) as r:
            r.sample()
            r.step(p["n_steps"])
            got.append([r.get(s) for s in range(2)])
    for g in got[1:]:
        for s in range(2):
            for a, b in zip(g[s], got[0][s]):
                assert np.array_equal(a, b)
