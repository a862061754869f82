"""Cells whose operands leave the range of the integer-pipe functions (here:
B_n^2 is subnormal in every cell) are evaluated again with the complete ones."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

import oracle as O  # noqa: E402
from helpers import rel_l1  # noqa: E402
from paper_2402_05240_gb300 import inputs as I  # noqa: E402


@pytest.mark.parametrize("recon", ["pcm", "plmc", "ppmc"])
@pytest.mark.parametrize("n", [(4, 4, 4), (33, 5, 4), (70, 4, 6)])
def test_subnormal_field_energy(recon, n):
    from paper_2402_05240_gb300 import mhd
    box = I.Box(*n)
    x = box.centres()[0]
    one = np.ones(box.shape)
    rho = one * (1 + 0.3 * np.sin(2 * np.pi * (x + 0.13)) + 0.1 * np.sin(6 * np.pi * x))
    vel = (one * 0.4 * np.cos(2 * np.pi * (x + 0.3)), 0 * one, 0 * one)
    pres = one * (1 + 0.2 * np.cos(4 * np.pi * (x + 0.05)))
    U0 = I.assemble(box, rho, vel, pres, (1e-160 * one, 0 * one, 0 * one))
    sim = mhd.Sim(*n, recon=recon)
    U = torch.from_numpy(U0).cuda()
    dts = torch.zeros(3, dtype=torch.float64, device="cuda")
    sim.run(U, 3, dts)
    sim.status()
    ref, _ = O.Oracle(*n, recon=recon).run(U0, 3, dts=dts.cpu().numpy().tolist())
    got = U.cpu().numpy()
    assert np.all(rel_l1(got, ref)[:5] <= 1e-12)
    assert np.array_equal(got[5:], U0[5:])
