"""The limiters' follow-up work at the sizes where its forms change, one step
against the oracle from a quiet state with a chosen number of far sites."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle as O  # noqa: E402
from paper_1110_0270_gb300 import lbm  # noqa: E402
from paper_1110_0270_gb300 import workloads as WL  # noqa: E402

pytestmark = pytest.mark.gpu


def far_sites(cfg, count, seed=3):
    """Uniform flow with `count` sites perturbed, no two of them neighbours."""
    ny, nx = cfg["ny"], cfg["nx"]
    f = O.init_equilibrium(dict(cfg, collision="lbgk"), np.ones((ny, nx)), np.full((ny, nx), 0.03),
                           np.full((ny, nx), -0.02))
    rng = np.random.default_rng(seed)
    cells = rng.choice((ny // 3) * (nx // 3), size=count, replace=False)
    y, x = 3 * (cells // (nx // 3)) + 1, 3 * (cells % (nx // 3)) + 1
    f[:, y, x] *= np.exp(0.2 * rng.uniform(0.5, 1.0, count) * rng.standard_normal((9, count)))
    return f


def one_step(cfg, f0):
    dt = torch.float64 if cfg["precision"] == "fp64" else torch.float32
    f0 = torch.tensor(f0, dtype=dt, device="cuda")
    lat = lbm.Lattice(cfg)
    lat.set_state(f0)
    lat.step(1)
    f, st = O.step(cfg, f0.double().cpu().numpy(), 1, stats=True)
    g = lat.get_state(torch.float64).cpu().numpy()
    return lat, float(np.linalg.norm(g - f) / np.linalg.norm(f)), st


@pytest.mark.parametrize("count", [0, 1, 16, 17, 31, 32, 33, 256, 257, 600])
@pytest.mark.parametrize("delta0", [0.3, 1e-3])
def test_threshold_forms(count, delta0):
    """One warp up to 32 candidates, the radix descent above (FP64: the
    reordered sums change Delta S_t by its own rounding, 1e-13)."""
    cfg = dict(lattice="D2Q9", nx=90, ny=78, bc="periodic", collision="threshold", precision="fp64", beta=0.9,
               lim_delta0=delta0, delta=1e-7)
    lat, err, st = one_step(cfg, far_sites(cfg, count))
    assert err < 1e-13
    assert lat.stats()["limited_total"] == st["limited_sites"]
