"""Short calls of lbm_step on a D1Q3 line: two and three steps in FP32 replay the
step graph, longer calls, FP64 and ELBM ones and those inside a stream capture
take the line form; any division of a run into calls gives the same state."""
import pytest

torch = pytest.importorskip("torch")

import oracle as O  # noqa: E402
from paper_1110_0270_gb300 import lbm  # noqa: E402
from paper_1110_0270_gb300 import workloads as WL  # noqa: E402

pytestmark = pytest.mark.gpu

# (on 14000 sites the kernels of a call in FP64 are kept apart at its odd step)
CFGS = [("lbgk", "fp64", "ends", 800), ("lbgk", "fp32", "periodic", 800), ("elbm", "fp64", "ends", 800),
        ("elbm", "fp32", "ends", 800), ("smooth", "fp64", "ends", 14000)]


def start(coll, prec, bc, nx):
    cfg = dict(lattice="D1Q3", nx=nx, ny=1, bc=bc, collision=coll, precision=prec, beta=0.95, lim_alpha=40.0)
    fl = WL.random_fields(1, nx, 3, 0.05, 0.1)
    f0 = O.init_equilibrium(cfg, fl["rho"], fl["ux"], None) * WL.lognormal_factors((3, 1, nx), 4, 1e-2)
    f0 = torch.tensor(f0, dtype=torch.float64 if prec == "fp64" else torch.float32, device="cuda")
    lat = lbm.Lattice(cfg)
    lat.set_state(f0)
    return lat


def difference(a, b):
    a, b = a.get_state(torch.float64), b.get_state(torch.float64)
    return float((a - b).norm() / b.norm())


@pytest.mark.parametrize("coll,prec,bc,nx", CFGS)
@pytest.mark.parametrize("calls", [[2], [3], [1, 2], [1, 3, 2], [2, 2, 3, 1, 2, 4], [3, 3, 5, 2, 7, 1]])
def test_short_calls(coll, prec, bc, nx, calls):
    a, b = start(coll, prec, bc, nx), start(coll, prec, bc, nx)
    for n in calls:
        a.step(n)
    for _ in range(sum(calls)):
        b.step(1)
    # the same arithmetic site by site (ELBM's solves: its 1e-15 or FP32 rounding)
    tol = 0.0 if coll != "elbm" else (1e-12 if prec == "fp64" else 1e-6)
    assert a.stats()["steps"] == b.stats()["steps"] == sum(calls)
    assert difference(a, b) <= tol


@pytest.mark.parametrize("coll,prec,bc,nx", CFGS)
@pytest.mark.parametrize("n", [2, 3, 4, 27])
def test_captured_call(coll, prec, bc, nx, n):
    a, b = start(coll, prec, bc, nx), start(coll, prec, bc, nx)
    f0 = a.get_state(torch.float64 if prec == "fp64" else torch.float32)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        a.set_state(f0)
        a.step(n)
    graph.replay()
    graph.replay()
    b.step(n)
    assert difference(a, b) <= (0.0 if coll != "elbm" else (1e-12 if prec == "fp64" else 1e-6))
