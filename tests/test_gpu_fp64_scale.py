"""FP64 D2Q9 collisions divide by rho through an FP32-seeded reciprocal while rho
lies in 2^-100 ... 2^100 and by a plain division outside: the collisions are
homogeneous in f, so a state scaled by a power of two gives the scaled result on
either side of the seeds' range."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle as O  # noqa: E402
from paper_1110_0270_gb300 import lbm  # noqa: E402
from paper_1110_0270_gb300 import workloads as WL  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("collision", ["lbgk", "mrt", "mrt2"])
@pytest.mark.parametrize("equilibrium", ["poly", "entropic", "poly_std"])
@pytest.mark.parametrize("exponent", [-300, -101, -100, -99, 0, 99, 100, 101, 300])
def test_homogeneous(collision, equilibrium, exponent):
    cfg = dict(lattice="D2Q9", nx=67, ny=31, bc="periodic", collision=collision, precision="fp64", beta=0.9,
               equilibrium=equilibrium)
    fl = WL.random_fields(31, 67, 3, 0.3, 0.1)
    f0 = O.init_equilibrium(dict(cfg, collision="lbgk"), fl["rho"], fl["ux"], fl["uy"])
    f0 = f0 * WL.lognormal_factors(f0.shape, 4, 0.05)
    f = O.step(cfg, f0, 3)
    lat = lbm.Lattice(cfg)
    lat.set_state(torch.tensor(np.ldexp(f0, exponent), device="cuda"))
    lat.step(3)
    assert lat.stats()["diverged"] == 0
    g = np.ldexp(lat.get_state(torch.float64).cpu().numpy(), -exponent)
    # three steps of 40 operations, each 2^-53
    assert np.linalg.norm(g - f) < 3 * 40 * 2.0 ** -53 * np.linalg.norm(f)
