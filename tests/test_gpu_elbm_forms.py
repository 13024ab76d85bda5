"""The forms of the ELBM solve against the oracle, one step each: the FP32
one near and away from equilibrium, the groups of lanes and the threads' own
FP64 solve (FP32 storage takes each where its range ends), and the D1Q3 FP64
kernel with four lanes per site at the edges of its groups, CTAs and range."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle as O  # noqa: E402
from paper_1110_0270_gb300 import lbm  # noqa: E402
from paper_1110_0270_gb300 import workloads as WL  # noqa: E402

pytestmark = pytest.mark.gpu

# one step in FP32: every population is one rounding of f + alpha beta (f* - f)
# (alpha beta rounded as well: 2^-24 of |alpha beta (f* - f)| <= 2 max(f, f*)),
# the rest population the rounded sum of the others: eight partial sums of at
# most rho, each 2^-24, against |f| >= rho / 3 per site
TOL32 = 2.0 ** -24 * (1 + 4 + 8 * 3)


def one_step(cfg, f0):
    dt = torch.float64 if cfg["precision"] == "fp64" else torch.float32
    lat = lbm.Lattice(cfg)
    lat.set_state(torch.tensor(f0, dtype=dt, device="cuda"))
    lat.step(1)
    f, st = O.step(cfg, f0, 1, stats=True)
    g = lat.get_state(torch.float64).cpu().numpy()
    gs = lat.stats()
    assert gs["diverged"] == 0
    # FP32 storage skips below 1e-15 + 2^-48 rho, the floor of its own rounding
    # (the oracle and FP64 storage: below 1e-15)
    quiet = np.sum(O.delta_s_field(dict(cfg, equilibrium="entropic"), f0) <
                   1e-15 + (0.0 if cfg["precision"] == "fp64" else 2.0 ** -48) * f0.sum(0))
    assert gs["elbm_fallbacks"] == st["elbm_fallbacks"]
    assert gs["elbm_skipped"] == quiet >= st["elbm_skipped"]
    assert gs["elbm_solved"] == f0[0].size - quiet - gs["elbm_fallbacks"]
    return float(np.linalg.norm(g - f) / np.linalg.norm(f))


@pytest.mark.parametrize("lattice,ny,nx", [("D2Q9", 31, 67), ("D1Q3", 1, 1037)])
@pytest.mark.parametrize("u_amp", [0.1, 0.35])
@pytest.mark.parametrize("width", [1e-5, 1e-3, 0.02, 0.1, 0.25, 0.6])
@pytest.mark.parametrize("fallback", ["positivity", "ehrenfest"])
def test_fp32_forms(lattice, ny, nx, u_amp, width, fallback):
    cfg = dict(lattice=lattice, nx=nx, ny=ny, bc="periodic", collision="elbm", precision="fp32", beta=0.93,
               elbm_fallback=fallback)
    fl = WL.random_fields(ny, nx, 3, 0.05, u_amp)
    f0 = O.init_equilibrium(cfg, fl["rho"], fl["ux"], fl["uy"] if lattice == "D2Q9" else None)
    f0 = (f0 * WL.lognormal_factors(f0.shape, 4, width)).astype(np.float32).astype(np.float64)
    assert one_step(cfg, f0) < TOL32


def test_fp32_few_hard_sites_per_warp():
    """Single sites with a nearly empty population in quiet fluid: the groups
    of lanes take them."""
    cfg = dict(lattice="D2Q9", nx=70, ny=9, bc="cavity", lid_u=0.1, collision="elbm", precision="fp32", beta=0.9)
    fl = WL.random_fields(9, 70, 5, 0.01, 0.02)
    f0 = O.init_equilibrium(cfg, fl["rho"], fl["ux"], fl["uy"])
    f0 = f0 * WL.lognormal_factors(f0.shape, 6, 1e-3)
    f0[2, 4, 3] = f0[7, 4, 17] = f0[1, 6, 40] = 1e-9
    assert one_step(cfg, f0.astype(np.float32).astype(np.float64)) < TOL32


@pytest.mark.parametrize("nx", [1, 2, 7, 8, 9, 33, 800, 15999, 16001])
@pytest.mark.parametrize("width", [1e-3, 0.3])
def test_fp64_line(nx, width):
    """FP64 (1e-12: the reordered sums and the solve's own 1e-15)."""
    cfg = dict(lattice="D1Q3", nx=nx, ny=1, bc="ends", collision="elbm", precision="fp64", beta=0.95)
    fl = WL.random_fields(1, nx, 3, 0.05, 0.1)
    f0 = O.init_equilibrium(cfg, fl["rho"], fl["ux"], None)
    assert one_step(cfg, f0 * WL.lognormal_factors(f0.shape, 4, width)) < 1e-12
