"""boruta_quantise at the sizes and value distributions where its paths meet:
sorted columns (4096 values) against bucketed ones, unaligned columns and
strides, repeated values in every share, infinities and denormals; the numpy
statement of the rank rule, exactly."""
import numpy as np
import pytest

from paper_2605_09950_gb300 import synth

pytestmark = pytest.mark.gpu


def columns(N, rng):
    g = rng.standard_normal(N)
    F = [g, np.exp(8 * g), np.full(N, 1.5), np.where(rng.random(N) < 0.9, 2.0, 3.0), np.round(g), -np.abs(g) * 1e-41,
         np.sort(g), np.where(rng.random(N) < 0.6, 0.0, g), rng.integers(0, 70, N) * 1.0,
         1.0 + np.floor(rng.random(N) * 40) * 2.0**-23, np.where(rng.random(N) < 0.01, np.inf, -np.inf)]
    F[0][: min(N, 3)] = [np.inf, -np.inf, 0.0][: min(N, 3)]
    return np.stack(F).astype(np.float32)


@pytest.mark.parametrize("N,B", [(1, 256), (2, 3), (1023, 64), (4096, 256), (4097, 256), (4098, 2), (5000, 255),
                                 (65_537, 256), (200_003, 100)])
@pytest.mark.parametrize("pad", [0, 1])
def test_quantise_sizes(N, B, pad):
    import torch

    from paper_2605_09950_gb300 import boruta

    F = columns(N, np.random.default_rng(N + B))
    wide = torch.zeros((F.shape[0], N + pad), dtype=torch.float32, device="cuda")
    wide[:, pad:] = torch.from_numpy(F).cuda()  # pad = 1: odd stride, columns off 16-byte boundaries
    got = boruta.boruta_quantise(wide[:, pad:], B, N=N)
    np.testing.assert_array_equal(got.cpu().numpy(), synth.quantise(F.astype(np.float64), B))
