"""D1Q3 runs that take several steps per launch (windows of the line with
halos) against single steps of the same state: the same arithmetic at every
site, so the same bits, at the edges of the windows, of the launches' step
counts and of the range of line lengths."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle as O  # noqa: E402
from paper_1110_0270_gb300 import lbm  # noqa: E402
from paper_1110_0270_gb300 import workloads as WL  # noqa: E402

pytestmark = pytest.mark.gpu


def state(cfg, width):
    fl = WL.random_fields(1, cfg["nx"], 3, 0.05, 0.1)
    f0 = O.init_equilibrium(dict(cfg, collision="lbgk"), fl["rho"], fl["ux"], None)
    f0 = f0 * WL.lognormal_factors(f0.shape, 4, width)
    return torch.tensor(f0, dtype=torch.float64 if cfg["precision"] == "fp64" else torch.float32, device="cuda")


def runs(cfg, f0, n, first=0):
    """The state after n steps: `first` steps and the rest in one call, and one by one."""
    out = []
    for parts in ([first, n - first], [1] * n):
        lat = lbm.Lattice(cfg)
        lat.set_state(f0)
        for k in parts:
            lat.step(k)
        st = lat.stats()
        assert st["diverged"] == 0
        out.append((lat.get_state(f0.dtype), st))
    return out


@pytest.mark.parametrize("nx", [1, 2, 5, 31, 800, 1216, 1217, 1369, 3041, 20000, 35264, 36600])
@pytest.mark.parametrize("bc", ["ends", "periodic"])
@pytest.mark.parametrize("coll,prec", [("lbgk", "fp64"), ("lbgk", "fp32"), ("smooth", "fp64"),
                                       ("double_monotonic", "fp32")])
def test_windows(nx, bc, coll, prec):
    cfg = dict(lattice="D1Q3", nx=nx, ny=1, bc=bc, collision=coll, precision=prec, beta=0.95, lim_alpha=40.0,
               lim_k=1.0, lim_dst=2e-3)
    f0 = state(cfg, 0.02)
    (a, _), (b, _) = runs(cfg, f0, 31)
    assert torch.equal(a, b)


@pytest.mark.parametrize("n,first", [(2, 0), (3, 1), (4, 1), (5, 0), (23, 0), (24, 0), (25, 0), (26, 1), (49, 3),
                                     (128, 0)])
def test_step_counts(n, first):
    cfg = dict(lattice="D1Q3", nx=800, ny=1, bc="ends", collision="lbgk", precision="fp64", beta=0.95)
    (a, _), (b, _) = runs(cfg, state(cfg, 0.02), n, first)
    assert torch.equal(a, b)


@pytest.mark.parametrize("nx", [3, 800, 5000])
def test_elbm_fp32(nx):
    """Same solves, but which form a hard site takes depends on its warp: FP32
    rounding of the two forms' alpha, 20 steps at 2^-23 of f each, twice over."""
    cfg = dict(lattice="D1Q3", nx=nx, ny=1, bc="ends", collision="elbm", precision="fp32", beta=0.9)
    (a, sa), (b, sb) = runs(cfg, state(cfg, 0.05), 20)
    assert float((a - b).norm() / b.norm()) < 2 * 20 * 2.0 ** -23
    n = nx * 20  # every site of every step is counted once
    assert all(s["elbm_solved"] + s["elbm_skipped"] + s["elbm_fallbacks"] == n for s in (sa, sb))


@pytest.mark.parametrize("nx", [1, 2, 3, 4, 5, 31, 800, 1216, 1217])
@pytest.mark.parametrize("bc", ["ends", "periodic"])
def test_elbm_fp64(nx, bc):
    """Windows of eight sites, four lanes each.  A warp's series are as long as
    its largest deviation needs, so a site's last bits depend on its window:
    1e-15 of alpha a step, 20 steps, both runs."""
    cfg = dict(lattice="D1Q3", nx=nx, ny=1, bc=bc, collision="elbm", precision="fp64", beta=0.9)
    (a, sa), (b, sb) = runs(cfg, state(cfg, 0.05), 21)
    assert float((a - b).norm() / b.norm()) < 2 * 20 * 4 * 2.0 ** -52
    assert all(s["elbm_solved"] + s["elbm_skipped"] + s["elbm_fallbacks"] == nx * 21 for s in (sa, sb))


@pytest.mark.parametrize("width", [1e-7, 1e-5, 2e-3, 0.02, 0.05, 0.1, 0.2])
def test_fp64_series(width):
    """One FP64 ELBM step at deviations in every range of the solve's series
    against the oracle (1e-12: reordered sums and the solve's own 1e-15)."""
    cfg = dict(lattice="D1Q3", nx=4001, ny=1, bc="ends", collision="elbm", precision="fp64", beta=0.95)
    f0 = state(cfg, width)
    lat = lbm.Lattice(cfg)
    lat.set_state(f0)
    lat.step(1)
    f = O.step(cfg, f0.cpu().numpy(), 1)
    assert np.linalg.norm(lat.get_state(torch.float64).cpu().numpy() - f) < 1e-12 * np.linalg.norm(f)
