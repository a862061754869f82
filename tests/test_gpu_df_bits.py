"""Float pairs of the primitives: within 2^-48 of the double values."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def test_density_keeps_48_bits():
    from paper_2402_05240_gb300 import mhd
    n = (33, 6, 5)
    U = np.abs(np.random.default_rng(3).normal(size=(8,) + n[::-1])) + 0.5
    U[4] += 20.0
    W = mhd.Sim(*n, precision="fp64_df").primitives(torch.from_numpy(U).cuda()).cpu().numpy()
    assert np.max(np.abs(W[0] - U[0]) / U[0]) <= 2.0 ** -48
