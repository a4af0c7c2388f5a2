"""The FP64 field build from half spectra, at the grid sizes and slots that no other test builds.

The bars are the contract's, a slot's error relative to its own largest value: 1e-12 in FP64 and
1e-6 in FP32, twice that at 512^3 (27 levels of 2^-24, in quadrature 3.1e-7, and the FP32 unit
Gaussians, wavenumbers and amplitudes, of the same size)."""
import numpy as np
import pytest

import oracle as O

pytestmark = pytest.mark.gpu

TOL64, TOL32 = 1e-12, 2e-6


@pytest.fixture(scope="module")
def F():
    from paper_2207_14256_gb300 import build, fdf

    build.build()
    fdf.lib()
    return fdf


@pytest.mark.parametrize("N", [16, 32, 256])
def test_half_spectrum_fields_match_the_oracle(F, inputs, c1_tables, N):
    p = inputs.config("c1_32", n_grid=N, box=1000.0 * N / 32, precision=0, seed=35, flags=1)
    o = O.Oracle(p, c1_tables)
    lna = o.lna(55)
    with F.Run(p, c1_tables) as r:
        g = r.build_fields(lna)
    ref, _ = o.fields(lna, 0xFF, o.noise())
    for s in range(8):
        assert np.max(np.abs(g[s] - ref[s])) < TOL64 * np.max(np.abs(ref[s])), s


def test_half_spectrum_fields_at_512_match_the_fp32_form(F, inputs, c1_tables):
    """512^3, against the packed FP32 form on the device."""
    import torch

    p = inputs.config("c1_32", n_grid=512, box=16000.0, seed=36)
    lna = O.Oracle(dict(p, n_grid=8), c1_tables).lna(80)
    out = []
    for prec in (0, 1):
        with F.Run(dict(p, precision=prec), c1_tables) as r:
            out.append(F.fdf_build_fields(r.ctx, lna, torch.empty(8, 512 ** 3, dtype=torch.float64, device="cuda")))
    for s in range(8):
        assert (out[0][s] - out[1][s]).abs().max() < (TOL64 + TOL32) * out[0][s].abs().max(), s
