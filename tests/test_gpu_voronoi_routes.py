"""Tessellations on either side of the rule that chooses between bricks and single sites
(small and large grains, flat and small lattices), from both entry points.  Whole
numbers: equal to the oracle's."""
import numpy as np
import pytest

from tests.gpu_util import need_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dim,L,v", [
    (3, (40, 36, 20), 3), (3, (40, 36, 20), 40), (3, (72, 64, 40), 90), (3, (72, 64, 40), 130), (3, (30, 30, 30), 60),
    (3, (30, 30, 30), 100), (3, (128, 96, 8), 20), (3, (128, 96, 8), 60), (2, (256, 250), 12), (2, (256, 250), 40),
    (2, (300, 200), 11), (2, (300, 200), 60)])
def test_either_route_equals_oracle(oracle, dim, L, v):
    torch, hm = need_gpu()
    N = int(np.prod(L))
    G, seed = N // v, 77 + v
    ref_q, ref_pos = oracle.voronoi(dim, L, G, seed)
    lat = hm.Lattice(dim, L, 8 if dim == 2 else 26, 256, seed, G)
    q = torch.full((N,), -5, dtype=torch.int32, device="cuda")
    m = torch.full((N,), -5, dtype=torch.int32, device="cuda")
    pos = torch.empty(G, dtype=torch.int64, device="cuda")
    lat.hp_bind(q, m)
    for call in (lat.hp_init_voronoi, lat.hp_init_voronoi_static):
        q.fill_(-5)
        m.fill_(-5)
        call(hm.ORIENT_ANGLE, None, pos)
        torch.cuda.synchronize()
        np.testing.assert_array_equal(pos.cpu().numpy(), ref_pos)
        np.testing.assert_array_equal(q.cpu().numpy(), ref_q)
        np.testing.assert_array_equal(m.cpu().numpy(), np.arange(N))
    lat.close()
