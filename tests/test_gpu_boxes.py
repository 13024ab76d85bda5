"""Diffusive boxes (Section 8's wall sites) at the launch shapes where the wall
sites change kernels, against the oracle."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle as O  # noqa: E402
from paper_1110_0270_gb300 import lbm  # noqa: E402
from paper_1110_0270_gb300 import workloads as WL  # noqa: E402

pytestmark = pytest.mark.gpu


def rel_error(cfg, seed, width, steps):
    """||f - oracle|| / ||oracle|| after `steps` steps from a random flow with
    log-normal noise of the given width."""
    ny, nx = cfg["ny"], cfg["nx"]
    fl = WL.random_fields(ny, nx, seed, 0.02, 0.05)
    f0 = O.init_equilibrium(dict(cfg, collision="lbgk"), fl["rho"], fl["ux"], fl["uy"])
    f0 = f0 * WL.lognormal_factors(f0.shape, seed + 1, width)
    dt = torch.float64 if cfg["precision"] == "fp64" else torch.float32
    f0 = torch.tensor(f0, dtype=dt, device="cuda")
    lat = lbm.Lattice(cfg)
    lat.set_state(f0)
    lat.step(steps)
    f = O.step(cfg, f0.double().cpu().numpy(), steps)
    g = lat.get_state(torch.float64).cpu().numpy()
    return float(np.linalg.norm(g - f) / np.linalg.norm(f))


# the largest height the configuration accepts, and heights on either side of
# the one from which the sites' own CTA rows leave no room for the wall sites'
# (65535 rows of CTAs in all: ny / 2 for the sites and 2 (nx + ny - 2) / 256 for
# the wall sites fill them at ny = 129052)
@pytest.mark.parametrize("ny", [129052, 129053, 131069, 131070])
@pytest.mark.parametrize("collision", ["lbgk", "ehrenfest"])
def test_tall_box_fp32(ny, collision):
    cfg = dict(lattice="D2Q9", nx=4, ny=ny, bc="diffusive", lid_u=0.1, collision=collision, precision="fp32",
               beta=0.9, equilibrium="entropic", topk=8, delta=1e-4)
    # three steps of about 20 operations, each 2^-24
    assert rel_error(cfg, 3, 1e-2, 3) < 3 * 20 * 2.0 ** -24


@pytest.mark.parametrize("equilibrium", ["poly", "entropic", "poly_std"])
@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_elbm_walls_are_entropic(precision, equilibrium):
    """ELBM's equilibria are entropic whatever the configuration names, at the
    wall sites too (a fast top wall, where the kinds differ most)."""
    cfg = dict(lattice="D2Q9", nx=37, ny=29, bc="diffusive", lid_u=0.3, collision="elbm", precision=precision,
               beta=0.9, equilibrium=equilibrium)
    # five steps of 40 (20) operations and the root's 1e-14 (2^-22)
    tol = 5 * (40 * 2.0 ** -53 + 1e-14) if precision == "fp64" else 5 * (20 * 2.0 ** -24 + 2.0 ** -22)
    assert rel_error(cfg, 3, 1e-2, 5) < tol


# FP64 ELBM takes CTAs of 64 sites up to 360000 and of 256 above, the wall sites
# behind the others in CTAs of the same size
@pytest.mark.parametrize("nx,ny", [(600, 600), (601, 600), (1030, 1025)])
@pytest.mark.parametrize("bc", ["cavity", "diffusive"])
def test_fp64_elbm_cta_sizes(nx, ny, bc):
    cfg = dict(lattice="D2Q9", nx=nx, ny=ny, bc=bc, lid_u=0.05, collision="elbm", precision="fp64", beta=0.9)
    one = np.ones((ny, nx))
    f0 = O.init_equilibrium(cfg, one, 0 * one, 0 * one)
    # noise where the last CTA and the walls are
    f0[:, -4:] *= WL.lognormal_factors(f0[:, -4:].shape, 4, 1e-2)
    f0[:, ::64, :3] *= WL.lognormal_factors(f0[:, ::64, :3].shape, 5, 1e-2)
    lat = lbm.Lattice(cfg)
    lat.set_state(torch.tensor(f0, device="cuda"))
    lat.step(3)
    g = lat.get_state(torch.float64).cpu().numpy()
    f = O.step(cfg, f0, 3)
    # three steps of 40 operations, each 2^-53, and the root's 1e-14
    assert np.linalg.norm(g - f) < (3 * 40 * 2.0 ** -53 + 3e-14) * np.linalg.norm(f)
