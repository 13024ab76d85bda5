"""The Ehrenfest and MRT-limiter selection on lists around one round of the
selection kernel (16 records a CTA, one CTA per SM), where its second CTA per SM
joins in, on lattices that launch it ahead of the step's end and behind it; one
step against the oracle."""
import pytest

torch = pytest.importorskip("torch")

from test_gpu_followups import far_sites, one_step  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,bc", [(301, 203, "diffusive"), (401, 333, "cavity"), (401, 333, "diffusive"),
                                      (731, 725, "cavity"), (731, 725, "diffusive")])
@pytest.mark.parametrize("collision,precision", [("ehrenfest", "fp32"), ("ehrenfest", "fp64"), ("mrt_limiter", "fp32")])
@pytest.mark.parametrize("rounds,more", [(0, 40), (0, 600), (1, -1), (1, 0), (1, 1), (2, 1)])
def test_lists(nx, ny, bc, collision, precision, rounds, more):
    count = rounds * 16 * torch.cuda.get_device_properties(0).multi_processor_count + more
    count = min(count, (nx // 3 - 1) * (ny // 3 - 1))
    cfg = dict(lattice="D2Q9", nx=nx, ny=ny, bc=bc, lid_u=0.0, collision=collision, precision=precision, beta=0.9,
               topk=64, delta=1e-6)
    # a fluid at rest but for the far sites: nothing else is screened
    f0 = far_sites(cfg, count)
    rest = f0[:, 0, 0].sum()
    w = [4 / 9] + 4 * [1 / 9, 1 / 36]
    quiet = (f0 == f0[:, :1, :1]).all(0)
    for i in range(9):
        f0[i][quiet] = rest * w[i]
    lat, err, st = one_step(cfg, f0)
    gs = lat.stats()
    assert gs["limited_total"] == st["limited_sites"] == min(64, count)
    assert gs["screened_last"] >= gs["candidates_last"] == count
    # one step: the reordered sums of nine populations, FP32 about 20 operations
    assert err < (1e-13 if precision == "fp64" else 20 * 2.0 ** -24)
