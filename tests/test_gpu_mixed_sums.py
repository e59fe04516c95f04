"""FP32 sums of the mixed-precision step with many tiles a block: members of an
ensemble whose work weight gives them one block each (650 and 36 tiles of 32 x 8
cells on it) against the same members stepped alone (2 tiles a block at most).
The sums only steer the iterations, so the states agree like those of the tile
columns (1e-8 of the field, velocities against the norm of their vector)."""
import numpy as np
import pytest

from paper_2303_10499_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def test_one_block_members_equal_members_alone():
    import torch
    if not torch.cuda.is_available():
        pytest.fail("CUDA device required")
    from paper_2303_10499_gb300 import build as B
    B.build()
    from paper_2303_10499_gb300 import gea as G
    sizes = [(400, 400), (128, 72), (64, 64)]

    def make(i):
        nx, nz = sizes[i]
        grid = W.Grid(nx, nz, 2.5 * nx, 2.5 * nz)
        c = W.Constants(cp=1002.5, dt=0.1, mu=0.3, cs=0.17)
        s = G.Solver(grid, c, mixed=True)
        s.set_conservative(W.random_flow(grid, c, seed=i, uamp=1.0, thamp=0.5).fields)
        return s
    members = [make(i) for i in range(3)]
    e = G.Ensemble(members, weights=[1.0, 1.0, 1e6])
    assert e.blocks()[:2] == [1, 1]
    e.step_async(2)
    torch.cuda.synchronize()
    for i in range(2):
        alone = make(i)
        alone.step(2)
        a, b = members[i].get_full(), alone.get_full()
        assert members[i].stats()["status"] == 0 and members[i].stats()["steps_done"] == 2
        vel = np.hypot(np.linalg.norm(b["u"]), np.linalg.norm(b["w"]))
        for k in ("rho", "T", "pp", "u", "w"):
            scale = vel if k in "uw" else np.linalg.norm(b[k])
            d = np.linalg.norm(a[k] - b[k]) / scale
            print(sizes[i], k, d)
            assert d <= 1e-8, (sizes[i], k, d)
