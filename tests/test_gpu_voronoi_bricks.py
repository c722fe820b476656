"""The brick-wise nearest-seed assignment where its bounds and lists part: lattices
smaller than a brick and than a run, edges that are no multiple of either, few seeds
(one cell, every seed scanned), many (more than a brick's list holds, so that sites
scan their own rings), axes longer than the 32-bit distances allow, ties between seeds.
Whole numbers: equal to the oracle's."""
import numpy as np
import pytest

from tests.gpu_util import need_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dim,L,G", [
    (3, (2, 2, 2), 1), (3, (6, 10, 4), 3), (3, (34, 18, 10), 7), (3, (66, 42, 22), 1), (3, (66, 42, 22), 2),
    (3, (96, 40, 30), 115_200 // 3), (3, (40, 64, 36), 90), (3, (130, 6, 74), 500), (3, (16, 16, 16), 4096),
    (2, (2, 2), 2), (2, (70, 34), 5), (2, (200, 130), 9000), (2, (500, 66), 40), (2, (36000, 4), 300), (2, (4, 33000), 2)])
def test_bricks_equal_oracle(oracle, dim, L, G):
    torch, hm = need_gpu()
    seed, N = 31 + G, int(np.prod(L))
    ref_q, ref_pos = oracle.voronoi(dim, L, G, seed)
    for mp in (False, True):
        lat = hm.Lattice(dim, L, 8 if dim == 2 else 26, 256, seed, G)
        q = torch.full((N,), -5, dtype=torch.int32, device="cuda")
        m = torch.full((N,), -5, dtype=torch.int32, device="cuda") if mp else None
        pos = torch.empty(G, dtype=torch.int64, device="cuda")
        lat.hp_bind(q, m)
        lat.hp_init_voronoi(hm.ORIENT_ANGLE, None, pos)
        torch.cuda.synchronize()
        np.testing.assert_array_equal(pos.cpu().numpy(), ref_pos)
        np.testing.assert_array_equal(q.cpu().numpy(), ref_q)
        if mp:
            np.testing.assert_array_equal(m.cpu().numpy(), np.arange(N))
        lat.close()
