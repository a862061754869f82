"""The one-axis and the three-axis launches of a step are different kernels (for
float the corrector's also in form): grids past the threshold with ragged rows
against the oracle, in every reconstruction and precision, and the two
schedules against each other bit for bit where mhd_init falls back to the
smaller workspace."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

import oracle as O  # noqa: E402
from helpers import rel_l1  # noqa: E402
from paper_2402_05240_gb300 import inputs as I  # noqa: E402

THIN = [(37, 5, 4200), (4, 4, 16500)]  # 16 800 and 16 500 thread blocks


@pytest.fixture(scope="module")
def mhd():
    from paper_2402_05240_gb300 import build
    build.build()
    from paper_2402_05240_gb300 import mhd as m
    return m


def state(n, seed):
    """Turbulent velocities and fields with smooth density and pressure variations."""
    box = I.Box(*n)
    U = I.turbulent_box(box, seed_v=seed, seed_b=seed + 1, kmax=4)
    W = O.Oracle(*n).primitives(U)
    x, y, z = box.centres()
    p = np.random.default_rng(seed + 100).uniform(0, 2 * np.pi, 6)
    t = 2 * np.pi
    rho = W[0] * (1 + 0.2 * np.sin(t * x + p[0]) * np.cos(t * y + p[1]) * np.sin(t * z + p[2]))
    pres = W[4] * (1 + 0.2 * np.cos(t * x + p[3]) * np.sin(t * y + p[4]) * np.cos(t * z + p[5]))
    return I.assemble(box, rho, (W[1], W[2], W[3]), pres, (U[5], U[6], U[7]))


@pytest.mark.parametrize("n", THIN)
@pytest.mark.parametrize("recon", ["pcm", "plm_prim", "plmc", "ppmc"])
@pytest.mark.parametrize("precision,tol", [("fp64", 1e-12), ("fp64_df", 1e-12), ("fp32_bulk", 1e-5)])
def test_one_axis_launches(mhd, n, recon, precision, tol):
    U0 = state(n, 5)
    sim = mhd.Sim(*n, recon=recon, precision=precision, cfl=0.3)
    U = torch.from_numpy(U0).cuda()
    dts = torch.zeros(2, dtype=torch.float64, device="cuda")
    sim.run(U, 2, dts)
    sim.status()
    ref, _ = O.Oracle(*n, recon=recon).run(U0, 2, dts=dts.cpu().numpy().tolist())
    assert np.all(rel_l1(U.cpu().numpy(), ref) <= tol)


@pytest.mark.parametrize("recon,precision,tol", [("plmc", "fp64", 1e-10), ("ppmc", "fp64", 1e-10),
                                                 ("plmc", "fp64_df", 1e-10), ("ppmc", "fp64_df", 1e-10),
                                                 ("ppmc", "fp32_bulk", 1e-3)])
def test_adjoint_one_axis_launches(mhd, recon, precision, tol):
    n = THIN[0]
    U = state(n, 6)
    orc = O.Oracle(*n, recon=recon)
    dt = orc.dt(U, 0.3)
    rng = np.random.default_rng(5)
    dU, g = rng.normal(size=U.shape), rng.normal(size=U.shape)
    _, JdU = orc.step_jvp(U, dU, dt)
    gU = mhd.Sim(*n, recon=recon, precision=precision).adjoint_step(torch.from_numpy(U).cuda(), dt,
                                                                   torch.from_numpy(g).cuda()).cpu().numpy()
    assert abs(float(np.sum(JdU * g)) - float(np.sum(dU * gU))) <= tol * float(np.sum(np.abs(JdU * g)))


@pytest.mark.parametrize("recon", ["plmc", "ppmc"])
@pytest.mark.parametrize("precision", ["fp64", "fp64_df", "fp32_bulk"])
def test_smaller_workspace(mhd, recon, precision):
    """Where the device has room for the one-axis workspace only, mhd_init takes
    it, and the results are the same bits."""
    n = (128, 128, 128)
    U = torch.from_numpy(state(n, 7)).cuda()
    A, B = U.clone(), U.clone()
    sim = mhd.Sim(*n, recon=recon, precision=precision, cfl=0.3)
    sim.run(A, 2)
    torch.cuda.synchronize()
    large = mhd.mhd_workspace_bytes(sim.cfg)
    sim.close()
    words = 28 * (4 if precision == "fp32_bulk" else 8)
    torch.cuda.empty_cache()
    free = torch.cuda.mem_get_info()[0]
    hold = torch.empty(free - (large - words * U[0].numel() // 2), dtype=torch.uint8, device="cuda")
    try:
        assert torch.cuda.mem_get_info()[0] < large
        sim = mhd.Sim(*n, recon=recon, precision=precision, cfl=0.3)
        sim.run(B, 2)
        torch.cuda.synchronize()
        sim.close()
    finally:
        del hold
        torch.cuda.empty_cache()
    assert torch.equal(A, B)
