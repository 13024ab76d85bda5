"""ELBM in FP32 and FP64 at the edge of the root's existence: states whose root
comes ever closer to alpha_max, where a population of f + alpha (f* - f) nearly
vanishes, and states just beyond, which have none.  One step against the
oracle, site by site."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle as O  # noqa: E402
from paper_1110_0270_gb300 import lbm  # noqa: E402

pytestmark = pytest.mark.gpu

CX = {3: np.array([-1, 0, 1]), 9: np.array([0, 1, 1, 0, -1, -1, -1, 0, 1])}
CY = {3: np.zeros(3, int), 9: np.array([0, 0, -1, -1, -1, 0, 1, 1, 1])}


def equilibrium(rho, u, Q):
    a = (2.0 * np.sqrt(1.0 + 3.0 * u * u) - 1.0) / 6.0  # [2, sites]
    fac = lambda k, c: np.where(c[:, None] == 0, 1.0 - 2.0 * a[k], a[k] + 0.5 * c[:, None] * u[k])  # noqa: E731
    return rho * fac(0, CX[Q]) * (fac(1, CY[Q]) if Q == 9 else 1.0)


def slack(f, Q):
    """S-decrease at alpha_max, H(alpha_max - 1) / Delta S: a root exists where >= 0."""
    rho = f.sum(0)
    fe = equilibrium(rho, np.stack([(CX[Q][:, None] * f).sum(0), (CY[Q][:, None] * f).sum(0)]) / rho, Q)
    d = (fe - f) / fe
    g = lambda x: np.where(x <= -1, 1.0, (1 + np.maximum(x, -1 + 1e-300)) * np.log1p(np.maximum(x, -1 + 1e-16)) - x)  # noqa: E731
    gm = (fe * g(-d)).sum(0)
    return (fe * g(d / (-d).max(0))).sum(0) / gm - 1.0


def edge_states(Q, n, seed):
    """Up to n noise directions, each scaled to the width where the root
    disappears and brought off it on both sides by relative steps of 1e-1 to
    1e-5; density 1."""
    rng = np.random.default_rng(seed)
    base = equilibrium(np.ones(n), rng.uniform(-0.2, 0.2, (2, n)), Q)
    z = rng.standard_normal((Q, n))
    lo, hi = np.full(n, 0.05), np.full(n, 3.0)
    for _ in range(40):
        m = 0.5 * (lo + hi)
        ok = slack(base * np.exp(m * z), Q) >= 0
        lo, hi = np.where(ok, m, lo), np.where(ok, hi, m)
    keep = np.flatnonzero((lo > 0.06) & (lo < 1.5))
    base, z, lo = base[:, keep], z[:, keep], lo[keep]
    f = np.concatenate([base * np.exp(lo * (1.0 + s * 10.0 ** -k) * z) for k in range(1, 6) for s in (-1.0, 1.0)], 1)
    return f / f.sum(0)


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("fallback", ["positivity", "ehrenfest"])
@pytest.mark.parametrize("Q", [3, 9])
def test_root_next_to_alpha_max(Q, fallback, precision):
    dt = np.float32 if precision == "fp32" else np.float64
    f0 = edge_states(Q, 400, 5).astype(dt).astype(np.float64)
    ny = 1 if Q == 3 else 10
    n = f0.shape[1]
    cfg = dict(lattice=f"D{1 if Q == 3 else 2}Q{Q}", nx=n // ny, ny=ny, bc="periodic", collision="elbm",
               precision=precision, beta=0.93, elbm_fallback=fallback, elbm_max_iter=200)
    f0 = np.ascontiguousarray(f0.reshape(Q, ny, n // ny))
    lat = lbm.Lattice(cfg)
    lat.set_state(torch.tensor(f0.astype(dt), device="cuda"))
    lat.step(1)
    g = lat.get_state(torch.float64).cpu().numpy()
    f, st = O.step(cfg, f0, 1, stats=True)
    assert 0 < st["elbm_fallbacks"] == lat.stats()["elbm_fallbacks"] < n
    # rho = 1; FP32, units of 2^-24 per population: the sum 1, alpha beta's and
    # alpha's rounding (|alpha beta (f* - f)| < 4) 8; the rest population, rho
    # less the others, eight of those and eight sums.  FP64: the same sums and
    # the solve's 1e-15 of alpha.
    tol = 80 * 2.0 ** -24 if precision == "fp32" else 80 * 2.0 ** -53 + 4e-14
    assert np.abs(g - f).max() < tol
