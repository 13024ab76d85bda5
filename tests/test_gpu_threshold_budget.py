"""The threshold limiter (Eqs. EntThresh, entrHom) with no budget or one below
the rounding of its sums: Delta S_0 is the largest Delta S, so every site takes
the LBGK step.  One warp finds it up to 32 candidates, the radix descent above;
FP64, one step against the oracle."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle as O  # noqa: E402
from paper_1110_0270_gb300 import lbm  # noqa: E402
from test_gpu_followups import far_sites, one_step  # noqa: E402

pytestmark = pytest.mark.gpu

BASE = dict(lattice="D2Q9", nx=90, ny=78, bc="periodic", collision="threshold", precision="fp64", delta=1e-7)


# beta = 1: 1 - (2 beta - 1)^2 = 0, so R = 0 for any delta0
@pytest.mark.parametrize("count", [1, 5, 31, 32, 33, 257, 600])
@pytest.mark.parametrize("beta,delta0", [(0.9, 0.0), (1.0, 0.3), (1.0, 0.0)])
def test_no_budget(count, beta, delta0):
    cfg = dict(BASE, beta=beta, lim_delta0=delta0)
    f0 = far_sites(cfg, count)
    lat, err, st = one_step(cfg, f0)
    assert err < 1e-13  # the reordered sums of nine populations
    g = lat.get_state(torch.float64).cpu().numpy()
    f = O.step(dict(cfg, collision="lbgk"), f0, 1)
    assert np.linalg.norm(g - f) < 1e-13 * np.linalg.norm(f)


@pytest.mark.parametrize("count", [3, 4, 7, 32, 41, 300])
def test_budget_below_rounding(count):
    """Equal sites: n v and the running sum of n values v differ by more than R."""
    cfg = dict(BASE, beta=0.9, lim_delta0=1e-25)
    f0 = far_sites(cfg, count)
    rest = f0[:, 0, 0]
    hot = np.any(f0 != rest[:, None, None], axis=0)
    f0[:, hot] = (rest * np.exp(0.2 * np.random.default_rng(7).standard_normal(9)))[:, None]
    assert one_step(cfg, f0)[1] < 1e-13


@pytest.mark.parametrize("precision", ["fp64", "fp32", "fp16_dev"])
@pytest.mark.parametrize("lattice", ["D1Q3", "D2Q9"])
def test_quiet_steps_between_loud_ones(lattice, precision):
    """A step without a screened site leaves no sum behind: a quiet state's steps,
    then a loud state in the same context, against a context that began with it."""
    one = dict(lattice=lattice, nx=90, ny=78 if lattice == "D2Q9" else 1, bc="periodic", collision="threshold",
               precision=precision, beta=0.9, lim_delta0=0.3, delta=1e-5)
    dt = torch.float64 if precision == "fp64" else torch.float32
    ny = one["ny"]
    still = O.init_equilibrium(dict(one, collision="lbgk"), np.ones((ny, 90)), np.zeros((ny, 90)),
                               np.zeros((ny, 90)) if lattice == "D2Q9" else None)
    rng = np.random.default_rng(3)
    loud = still * np.exp(0.05 * rng.standard_normal(still.shape))
    a, b = lbm.Lattice(one), lbm.Lattice(one)
    a.set_state(torch.tensor(still, dtype=dt, device="cuda"))
    a.step(3)
    assert a.stats()["candidates_last"] == a.stats()["screened_last"] == 0
    for lat in (a, b):
        lat.set_state(torch.tensor(loud, dtype=dt, device="cuda"))
        lat.step(2)
    ga, gb = a.get_state(torch.float64).cpu().numpy(), b.get_state(torch.float64).cpu().numpy()
    # the sums' order differs between runs: 2^-24 (2^-53) of S and so of the threshold
    assert np.linalg.norm(ga - gb) <= (1e-13 if precision == "fp64" else 1e-6) * np.linalg.norm(gb)
    assert a.stats()["limited_total"] > 0
    if precision == "fp64":
        assert np.linalg.norm(ga - O.step(one, loud, 2)) < 1e-12 * np.linalg.norm(ga)
