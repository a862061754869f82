"""The reverse takes the forward's floor decisions: cells whose energy a floor
has just reset recover a pressure that differs from the floor by rounding alone,
and no cotangent may pass through the pressure of a cell that the forward holds
at the floor."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("precision", ["fp64", "fp64_df", "fp32_bulk"])
@pytest.mark.parametrize("p_floor", [1e-20, 1e-6])
@pytest.mark.parametrize("cfl", [False, True])
def test_cells_just_reset(precision, p_floor, cfl):
    from paper_2402_05240_gb300 import mhd
    n, floored = (8, 4, 5), 0
    for seed in range(16):
        # a uniform state keeps itself: all fluxes cancel, so its half step and
        # its next step recover the same pressure
        rng = np.random.default_rng(seed)
        u = np.concatenate([rng.uniform(0.3, 2, 1), rng.normal(size=3), [0.0], rng.normal(size=3)])
        u[4] = 0.1 * (u[1] ** 2 + u[2] ** 2 + u[3] ** 2) / u[0]
        U = torch.from_numpy(np.ascontiguousarray(np.broadcast_to(u[:, None, None, None], (8,) + n[::-1]))).cuda()
        g = torch.from_numpy(rng.normal(size=U.shape)).cuda()
        sim = mhd.Sim(*n, recon="plmc", precision=precision, p_floor=p_floor, cfl=0.3)
        sim.run(U, 1)
        assert sim.floor_count()[1] > 0
        V = U.clone()
        sim.run(V, 1)
        assert float((V[4] - U[4]).abs().max()) <= 4e-16 * float(U[4].max())
        P = sim.primitives(U)[4]
        gU = sim.adjoint_step_cfl(U, g)[0] if cfl else sim.adjoint_step(U, 1e-3, g)
        if bool((P > p_floor * (1 + {"fp64": 0.0, "fp64_df": 1e-13, "fp32_bulk": 1e-7}[precision])).any()):
            continue  # (rounded up: not held at the floor)
        floored += 1
        # the energy's cotangent: none, or the end state's own where P^{n+1} = P_floor to the bit
        ok = (gU[4] == 0) | (gU[4] == g[4])
        assert bool(ok.all()), (seed, float(gU[4].abs().max()))
    assert floored >= 4
