"""The FP64-state pass's integer and FP32 forms on the device, with its own inverse square root
estimate: the bits of the FP64 formulas, for functions alone and for whole runs with the kick's
integrals on the FP32 pipe and in FP64.  What the functions may refuse is derived in
tests/test_wide_math.py: 33 of 65536 roots (and mantissas next to a power of 4), of sums those
that leave their binade, likely only above 2^-7; the bounds are four times that."""
import ctypes as C

import numpy as np
import pytest

import device_checks

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def F(tmp_path_factory):
    fdf = device_checks.load(tmp_path_factory.mktemp("checks"))
    yield fdf
    device_checks.unload(fdf)


@pytest.mark.parametrize("lo,hi", [(1.0, 4.0), (1e-9, 1e13), (1e-30, 1e30)])
def test_functions_have_the_bits_of_fp64(F, lo, hi):
    import torch

    n = 1 << 22
    rng = np.random.default_rng(23)
    u = np.exp(rng.uniform(np.log(lo), np.log(hi), n))
    q = rng.normal(size=n) * np.exp2(rng.integers(-40, 40, n))
    d = (q * np.exp2(-rng.uniform(7.0, 60.0, n)) * rng.choice([-1.0, 1.0], n)).astype(np.float32)
    u[::9] = np.float32(u[::9])                                    # short significands
    d[::97] = 0.0
    dev = [torch.from_numpy(a).cuda() for a in (u, q, d)]
    counts = torch.zeros(12, dtype=torch.int64, device="cuda")
    torch.cuda.synchronize()
    assert F.lib().fdf_check_bits(n, *[t.data_ptr() for t in dev], counts.data_ptr()) == 0, F.fdf_last_error()
    refused, wrong = counts.cpu().numpy().reshape(6, 2).T
    print("refused of %d:" % n, refused)
    assert not wrong.any(), wrong
    assert refused[0] <= 4 * 33 / 65536 * n and refused[1] == 0
    assert refused[3] <= 2.0 ** -7 * n and refused[4] <= 2e-3 * n and refused[5] <= 2e-3 * n


@pytest.mark.parametrize("prec", [1, 2])
@pytest.mark.parametrize("n_steps,order,masses,fast", [
    (200, 1, [0.1, 0.1], 1), (200, 2, [0.02, 0.3], 1), (200, 1, [0.0, 0.06], 1),
    (100, 1, [0.3, 0.3], 2), (120, 1, [0.0, 0.1], 2)])
def test_kick_integrals_have_the_bits_of_fp64(F, inputs, c1_tables, prec, n_steps, order, masses, fast):
    p = inputs.config("c1_32", n_part=20011, n_grid=32, n_species=2, m_ev=masses, n_steps=n_steps, precision=prec,
                      interp_order=order, seed=71)
    got, counts = [], (C.c_int32 * 3)()
    F.lib().fdf_check_kick_fp64(0, counts)
    for fp64 in (0, 1):
        with F.Run(p, c1_tables) as r:
            r.sample()
            r.step(n_steps)
            got.append([r.get(s) for s in range(2)])
        F.lib().fdf_check_kick_fp64(1 - fp64, counts)
        # every pass came with its kick on the FP32 pipe, by fitted polynomials (1) or node sums (2)
        assert counts[fast] == -(-n_steps // 4) and sum(counts) == counts[fast]
    for s in range(2):
        for a, b in zip(*[g[s] for g in got]):
            assert np.array_equal(a, b)
