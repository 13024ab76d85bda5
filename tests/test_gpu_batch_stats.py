"""The ELBM counters of a batch: every site of every step is counted once as
solved, skipped or without a root, whatever the number of tiles per item."""
import pytest

torch = pytest.importorskip("torch")

import oracle as O  # noqa: E402
from paper_1110_0270_gb300 import lbm  # noqa: E402
from test_gpu_batch import state  # noqa: E402

pytestmark = pytest.mark.gpu

SIZES = [dict(lattice="D2Q9", nx=131, ny=67, bc="cavity", lid_u=0.1), dict(lattice="D2Q9", nx=20, ny=45, bc="periodic"),
         dict(lattice="D1Q3", nx=3001, ny=1, bc="ends")]


@pytest.mark.parametrize("tile_rows", [1, 3, 4, 64])
@pytest.mark.parametrize("precision", ["fp64", "fp32", "fp16_dev"])
def test_every_site_counted(precision, tile_rows):
    steps = 5
    cfgs = [dict(c, collision="elbm", precision=precision, beta=0.9) for c in SIZES]
    b = lbm.Batch(cfgs, opts=dict(tile_rows=tile_rows))
    b.init_uniform(1.0, 0.0, 0.0)
    f0 = [state(c, 20 + i) for i, c in enumerate(cfgs)]
    for i, f in enumerate(f0):
        b.set_state(i, torch.tensor(f, device="cuda"))
    b.step(steps)
    for i, c in enumerate(cfgs):
        st = b.stats(i)
        assert st["elbm_solved"] + st["elbm_skipped"] + st["elbm_fallbacks"] == steps * c["nx"] * c["ny"]
        assert st["elbm_iters_total"] >= st["elbm_iters_max"] >= 1
        if precision == "fp64":
            ref = O.step(c, f0[i], steps, stats=True)[1]
            assert st["elbm_fallbacks"] == ref["elbm_fallbacks"]
