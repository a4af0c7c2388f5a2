"""The FP64-state pass's two launch shapes, one block per SM and three (pass_blocks 1 and 3), give
the same results bit for bit: at particle counts around the 32 of a warp's chunk, and where every
warp takes several chunks, so that the work counter hands them out and is set back for the next
pass (three blocks of 8 warps on 152 SMs take 116,736 particles at once)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [1, 2])
@pytest.mark.parametrize("n_part,n_steps", [(1, 100), (31, 100), (32, 100), (33, 100), (257, 200), (300001, 24)])
def test_one_and_three_blocks_per_sm(inputs, c1_tables, prec, n_part, n_steps):
    from paper_2207_14256_gb300 import build
    from paper_2207_14256_gb300 import fdf as F

    build.build()
    p = inputs.config("c1_32", n_part=n_part, n_species=2, m_ev=[0.05, 0.2], n_grid=32, n_steps=n_steps, precision=prec,
                      seed=97)
    got = []
    for pb in (1, 3):
        with F.Run(dict(p, pass_blocks=pb), c1_tables) as r:
            r.sample()
            r.step(n_steps)
            r.step(-4)                     # another pass after the last one's reset
            r.step(4)
            got.append([r.get(s) for s in range(2)])
    for s in range(2):
        for a, b in zip(got[0][s], got[1][s]):
            assert np.array_equal(a, b)
            assert np.isfinite(a).all()
