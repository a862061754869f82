"""FP64 cells whose transverse field or velocity lies below 1e-154: the
eigensystem, or the whole cell, is evaluated again with the complete functions."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

import oracle as O  # noqa: E402
from helpers import rel_l1  # noqa: E402
from paper_2402_05240_gb300 import inputs as I  # noqa: E402


@pytest.mark.parametrize("recon", ["plmc", "ppmc"])
@pytest.mark.parametrize("kind", ["field", "tail"])
@pytest.mark.parametrize("n", [(33, 5, 4), (70, 6, 5)])
def test_transverse_components(recon, kind, n):
    from paper_2402_05240_gb300 import mhd
    box = I.Box(*n)
    x = box.centres()[0]
    one = np.ones(box.shape)
    rho = one * (1 + 0.3 * np.sin(2 * np.pi * (x + 0.13)) + 0.1 * np.sin(6 * np.pi * x))
    pres = one * (1 + 0.2 * np.cos(4 * np.pi * (x + 0.05)))
    small = 1e-160 * (2 + np.sin(2 * np.pi * x)) if kind == "field" else 10.0 ** (-320 * np.abs(2 * x - 1))
    vt = 0 * one if kind == "field" else one * small
    U0 = I.assemble(box, rho, (one * 0.4 * np.cos(2 * np.pi * (x + 0.3)), vt, 0 * one), pres,
                    (0.3 * one, one * small, 0 * one))
    sim = mhd.Sim(*n, recon=recon)
    U = torch.from_numpy(U0).cuda()
    dts = torch.zeros(3, dtype=torch.float64, device="cuda")
    sim.run(U, 3, dts)
    sim.status()
    ref, _ = O.Oracle(*n, recon=recon).run(U0, 3, dts=dts.cpu().numpy().tolist())
    got = U.cpu().numpy()
    assert np.all(rel_l1(got, ref) <= 1e-12)
