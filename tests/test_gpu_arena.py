"""A caller's arena of any alignment serves fdf_create: the buffers lie at its first 256-byte boundary,
for kernels that move 32 bytes at once in every form (the plain one in its grid records and its
sort)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [0, 1, 3])
def test_arenas_of_any_alignment(inputs, c1_tables, prec):
    import torch

    from paper_2207_14256_gb300 import build
    from paper_2207_14256_gb300 import fdf as F

    build.build()
    p = inputs.config("c1_32", n_part=3001, n_species=2, m_ev=[0.05, 0.2], n_grid=16, n_steps=20, precision=prec, seed=19)

    def run(arena):
        with F.Run(p, c1_tables, None, arena) as r:
            r.sample()
            r.step(p["n_steps"])
            return [r.get(s) for s in range(2)]

    need = F.fdf_footprint(F.make_params(p))
    room = torch.zeros(need + 1024, dtype=torch.uint8, device="cuda")
    want = run(None)
    for off in (0, 1, 8, 16, 32, 128, 255):
        room.zero_()
        room[off + need:] = 77
        got = run(room[off:off + need])
        assert bool((room[off + need:] == 77).all()) and not bool(room[:off].any())
        for s in range(2):
            for a, b in zip(got[s], want[s]):
                assert np.array_equal(a, b), (off, s)
    with pytest.raises(F.FdfError) as e:
        run(room[16:16 + 65536])           # (the footprint allows for tables larger than these)
    assert e.value.code == F.FDF_ENOMEM
