"""The gather grids that the particle passes read, as the x pass of a run writes them, against the
eight fields that fdf_build_fields returns (another x pass, compared with the oracle elsewhere).

Both x passes run the same stages on the same y-transformed values, so a slot differs by rounding
at most: per stage of a line's log2 N, 4 eps of each value's magnitude on either side, which a
unitary stage passes on in the 2-norm: 8 log2(N) sqrt(N) eps of the packed pair's largest value.
A BF16 grid may round such a difference to the neighbouring value, 2^-7 of it.
"""
import numpy as np
import pytest

import device_checks

pytestmark = pytest.mark.gpu

CELL = {0: ("float64", 64), 1: ("float32", 32), 2: ("bfloat16", 16)}


@pytest.fixture(scope="module")
def F(tmp_path_factory):
    fdf = device_checks.load(tmp_path_factory.mktemp("checks"))
    yield fdf
    device_checks.unload(fdf)


def _grid(F, r, k, N, prec):
    import torch

    g = torch.empty((N ** 3, 8), dtype=getattr(torch, CELL[prec][0]), device="cuda")
    assert F.lib().fdf_check_grid(r.ctx, k, g.data_ptr(), N ** 3 * CELL[prec][1]) == 0, F.fdf_last_error()
    return g


def _close(got, ref, pair, N, prec, what):
    """got and ref of one slot; pair: the largest value of the two slots transformed together."""
    eps = 2.0 ** -53 if prec == 0 else 2.0 ** -24
    bound = 8 * np.log2(N) * np.sqrt(N) * eps * pair
    d = (got.double() - ref).abs()
    if prec == 2:
        d = d - 2.0 ** -7 * ref.abs()
    assert float(d.max()) <= bound, what


@pytest.mark.parametrize("prec", [0, 1, 2])
@pytest.mark.parametrize("N", [8, 16, 32, 64, 128, 256, 512])
def test_gather_grid_is_the_fields(F, inputs, c1_tables, N, prec):
    import torch

    p = inputs.config("c1_32", n_grid=N, box=1000.0 * N / 32, n_part=33, n_steps=40, precision=prec, seed=41,
                      steps_per_pass=1)
    with F.Run(p, c1_tables) as r:
        r.sample()
        for k, slots in ((0, (0, 1, 2, 3, 4, 5, 7)), (1, (0, 1, 2, 3, 4, 5, 6))):
            # step 0's grid has psi in slot 7 (phi_dot + i psi); the steps' have phi_dot alone
            if k:
                r.step(1)
            _, lna = F.fdf_state(r.ctx)
            g = _grid(F, r, k, N, prec)
            ref = F.fdf_build_fields(r.ctx, lna, torch.empty((8, N ** 3), dtype=torch.float64, device="cuda"))
            top = [float(ref[s].abs().max()) for s in range(8)]
            for s in slots:
                pair = max(top[s], top[s ^ 1]) if s != 6 else top[6]
                _close(g[:, s], ref[s], pair, N, prec, (k, s))
            if k:
                _close(g[:, 7], torch.zeros_like(ref[7]), top[6], N, prec, "slot 7 of a step")
            del g, ref


@pytest.mark.parametrize("N", [8, 64, 128])
def test_slot_7_of_the_exact_equations(F, inputs, c1_tables, N):
    """phi + psi; phi from a context whose T_psi is T_phi.  FP64's contract bar, 1e-12."""
    import torch

    p = inputs.config("c1_32", n_grid=N, box=1000.0 * N / 32, n_part=33, n_steps=40, precision=0, seed=43,
                      eom=F.FDF_EOM_EXACT, steps_per_pass=1)

    def fields(r, lna):
        return F.fdf_build_fields(r.ctx, lna, torch.empty((8, N ** 3), dtype=torch.float64, device="cuda"))

    with F.Run(p, c1_tables) as r:
        r.sample()
        r.step(1)
        _, lna = F.fdf_state(r.ctx)
        g, ref = _grid(F, r, 1, N, 0), fields(r, lna)
    with F.Run(p, dict(c1_tables, T_psi=c1_tables["T_phi"])) as r:
        want = ref[7] + fields(r, lna)[7]
    assert float((g[:, 7] - want).abs().max()) <= 1e-12 * float(want.abs().max())
