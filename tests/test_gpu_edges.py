"""The general addressing (edge sites and the warps that hold one) and the
wall sites carried by the step kernel, against the oracle on lattices that are
mostly edge: every boundary, odd and even steps, sizes at the edges of warps
and CTAs."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle as O  # noqa: E402
from paper_1110_0270_gb300 import lbm  # noqa: E402
from paper_1110_0270_gb300 import workloads as WL  # noqa: E402

pytestmark = pytest.mark.gpu

# five steps: FP64 reorders the sums of nine populations (2^-53 each); FP32
# rounds about 20 operations a step to 2^-24
TOL = {"fp64": 5 * 40 * 2.0 ** -53, "fp32": 5 * 20 * 2.0 ** -24}


@pytest.mark.parametrize("bc,sizes", [
    ("cavity", [(1, 1), (2, 3), (3, 2), (31, 2), (33, 3), (65, 4), (130, 5)]),
    ("channel", [(1, 2), (2, 2), (33, 3), (129, 4)]),
    ("periodic", [(1, 1), (1, 5), (2, 2), (3, 33), (129, 3)]),
    ("diffusive", [(3, 3), (3, 9), (31, 4), (64, 5), (65, 3), (127, 8), (129, 131)])])
@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("coll", ["lbgk", "elbm"])
def test_edges(bc, sizes, prec, coll):
    for nx, ny in sizes:
        cfg = dict(lattice="D2Q9", nx=nx, ny=ny, bc=bc, lid_u=0.1, collision=coll, precision=prec, beta=0.9,
                   equilibrium="entropic")
        fl = WL.random_fields(ny, nx, 3, 0.02, 0.05)
        f0 = O.init_equilibrium(cfg, fl["rho"], fl["ux"], fl["uy"])
        f0 = f0 * WL.lognormal_factors(f0.shape, 4, 1e-2)
        dt = torch.float64 if prec == "fp64" else torch.float32
        lat = lbm.Lattice(cfg)
        f0 = torch.tensor(f0, dtype=dt, device="cuda")
        lat.set_state(f0)
        f = f0.double().cpu().numpy()
        lat.step(5)
        f = O.step(cfg, f, 5)
        g = lat.get_state(torch.float64).cpu().numpy()
        # ELBM: its root to 1e-15 (FP64), or 2^-24 of alpha (FP32), a step
        tol = TOL[prec] + (0 if coll == "lbgk" else 5 * (1e-14 if prec == "fp64" else 2.0 ** -22))
        assert np.linalg.norm(g - f) < tol * np.linalg.norm(f), (nx, ny)


def test_large_fp64_elbm():
    """Above 2^20 sites ELBM in FP64 takes larger CTAs: a resting lattice with
    noise in the last rows (the ragged last CTA) and beside the side walls, two
    steps (TOL of five steps and the root's 1e-14 each)."""
    nx, ny = 1027, 1025
    cfg = dict(lattice="D2Q9", nx=nx, ny=ny, bc="cavity", lid_u=0.05, collision="elbm", precision="fp64", beta=0.9)
    one = np.ones((ny, nx))
    f0 = O.init_equilibrium(cfg, one, 0 * one, 0 * one)
    f0[:, -3:] *= WL.lognormal_factors(f0[:, -3:].shape, 4, 1e-2)
    f0[:, ::64, :2] *= WL.lognormal_factors(f0[:, ::64, :2].shape, 5, 1e-2)
    lat = lbm.Lattice(cfg)
    lat.set_state(torch.tensor(f0, device="cuda"))
    lat.step(2)
    f = O.step(cfg, f0, 2)
    g = lat.get_state(torch.float64).cpu().numpy()
    assert np.linalg.norm(g - f) < (TOL["fp64"] + 2e-14) * np.linalg.norm(f)
