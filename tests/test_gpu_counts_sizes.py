"""Grain counts at lattice sizes on either side of each step of a warp's share (128 sites up
to 2048), on runs that cross it.  Whole numbers: equal to numpy's."""
import numpy as np
import pytest

from tests.gpu_util import need_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L", [(1116, 1116), (1116, 1118), (1578, 1578), (2000, 1246), (2232, 2232), (2300, 2200), (3156, 3156),
                               (3158, 3158), (4466, 4466)])
@pytest.mark.parametrize("block", [1, 700])
def test_counts(L, block):
    torch, hm = need_gpu()
    N, G = L[0] * L[1], 5000
    rng = np.random.default_rng(N + block)
    q0 = np.repeat(rng.integers(0, G, size=N // block + 1), block)[:N].astype(np.int32)
    q = torch.from_numpy(q0).cuda()
    lat = hm.Lattice(2, L, 4, 256, 1, G)
    lat.hp_bind(q)
    counts = torch.empty(G, dtype=torch.int64, device="cuda")
    alive = torch.empty(1, dtype=torch.int32, device="cuda")
    lat.hp_grain_counts(counts, alive)
    ref = np.bincount(q0, minlength=G)
    np.testing.assert_array_equal(counts.cpu().numpy(), ref)
    assert int(alive.item()) == (ref > 0).sum()
    assert lat.hp_measure()[0].alive == (ref > 0).sum()
    lat.close()
