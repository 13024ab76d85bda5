"""The k-largest selection on small lattices at the edges of its paths: counts
of candidates around a CTA's groups, threads and two records per thread, lists
shorter than a CTA, and more candidates than k."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle as O  # noqa: E402
from paper_1110_0270_gb300 import lbm  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("coll", ["ehrenfest", "mrt_limiter", "median"])
@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("nx,ny,n", [(5, 3, 0), (5, 3, 4), (5, 3, 15), (33, 31, 1), (33, 31, 16), (33, 31, 17),
                                     (33, 31, 64), (33, 31, 65), (33, 31, 255), (33, 31, 257), (33, 31, 512),
                                     (33, 31, 513), (33, 31, 1023)])
def test_counts(coll, prec, nx, ny, n):
    rng = np.random.default_rng(n)
    for topk in (9, 2000):
        cfg = dict(lattice="D2Q9", nx=nx, ny=ny, bc="cavity", lid_u=0.05, collision=coll, precision=prec, beta=0.95,
                   topk=topk, delta=1e-3)
        one = np.ones((ny, nx))
        f0 = O.init_equilibrium(dict(cfg, collision="lbgk"), one, 0.02 * one, 0.01 * one)
        hot = rng.permutation(nx * ny)[:n]
        f0.reshape(9, -1)[:, hot] *= 1 + rng.uniform(0.2, 0.5, n) * rng.choice([-1, 1], (9, n))
        dt = torch.float64 if prec == "fp64" else torch.float32
        f0 = torch.tensor(f0, dtype=dt, device="cuda")
        for first in (0, 1):  # the even and the odd step's rewriting
            lat = lbm.Lattice(cfg)
            lat.set_state(f0)
            lat.step(first)
            f = lat.get_state(torch.float64).cpu().numpy()
            lat.step(1)
            g = lat.get_state(torch.float64).cpu().numpy()
            o = O.step(cfg, f, 1)
            # FP64: reordered sums; FP32: about 40 roundings of 2^-24 a population
            assert np.linalg.norm(g - o) < (1e-13 if prec == "fp64" else 40 * 2.0 ** -24) * np.linalg.norm(o), topk
