"""boruta_quantise on repeated values that lie close together (the bisection
over the column): neighbouring floats in one and in several cells of the
bucket map, of both signs, beside spread values and infinities; the numpy
statement of the rank rule, exactly."""
import numpy as np
import pytest

from paper_2605_09950_gb300 import synth

pytestmark = pytest.mark.gpu


def columns(N, rng):
    near = rng.integers(0, 200, N)
    F = [1.0 + near * 2.0**-23, -1.0 - near * 2.0**-23, 1e6 + rng.integers(0, 200, N), 4096.0 + rng.integers(0, 9, N) / 2048,
         np.where(rng.random(N) < 0.5, 1.0 + near * 2.0**-23, -3.0 - near * 2.0**-22),
         np.where(rng.random(N) < 0.5, 1.0 + near * 2.0**-23, rng.standard_normal(N)),
         (1.0 + near * 2.0**-23) * 2.0 ** rng.integers(-3, 4, N), near * 1e-45,
         np.where(rng.random(N) < 0.4, 1.0, 1.0 + rng.integers(0, 2**19, N) * 2.0**-23),
         np.where(rng.random(N) < 0.01, rng.choice([-np.inf, np.inf], N), 1.0 + near * 2.0**-23)]
    return np.stack(F).astype(np.float32)


@pytest.mark.parametrize("N,B", [(4097, 64), (4099, 2), (20_000, 256), (100_003, 255)])
def test_close_values(N, B):
    import torch

    from paper_2605_09950_gb300 import boruta

    F = columns(N, np.random.default_rng(N + B))
    got = boruta.boruta_quantise(torch.from_numpy(F).cuda(), B)
    np.testing.assert_array_equal(got.cpu().numpy(), synth.quantise(F.astype(np.float64), B))


def test_nan_among_close_values_is_refused():
    import torch

    from paper_2605_09950_gb300 import boruta

    F = columns(5000, np.random.default_rng(0))
    F[:, ::7] = np.nan
    with pytest.raises(boruta.BorutaError, match="NaN"):
        boruta.boruta_quantise(torch.from_numpy(F).cuda(), 64)
