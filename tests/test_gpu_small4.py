"""The 4-neighbour sweep as it is routed by default, on both sides of the sizes where the
route changes (a cluster, one launch per colour, fused tiles), with a grain and a point
field: bit-exact against the fused kernel."""
import numpy as np
import pytest

from paper_1007_3509_gb300 import synth
from tests.gpu_util import need_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L", [(128, 128), (128, 130), (256, 256), (316, 316), (318, 316), (724, 724), (726, 724)])
@pytest.mark.parametrize("point", [False, True])
@pytest.mark.parametrize("aniso", [False, True])
def test_routes_agree(L, point, aniso):
    torch, hm = need_gpu()
    Q, N = 50, L[0] * L[1]
    rng = np.random.default_rng(N)
    q0 = torch.from_numpy(synth.blocky_lattice(L, Q, 5, block=5).astype(np.int32)).cuda()
    mp0 = torch.from_numpy(rng.permutation(N).astype(np.int32)).cuda()
    table = torch.from_numpy(rng.integers(-60, 60, size=N if point else Q).astype(np.int32)).cuda()
    ang = torch.from_numpy(rng.integers(0, 90000, size=Q).astype(np.int32)).cuda()
    got = []
    for kind in (hm.SWEEP_AUTO, hm.SWEEP_FUSED):
        lat = hm.Lattice(2, L, 4, 256, 9, Q, hm.FIELD_POINT if point else hm.FIELD_GRAIN)
        q, mp = q0.clone(), mp0.clone()
        lat.hp_bind(q, mp if point else None)
        lat.hp_set_field(table)
        lat.hp_set_threshold_table(*hm.hp_build_threshold_table(0.8))
        if aniso:
            J, m = hm.hp_build_read_shockley(1.0, 15.0, 500, 91, 1000, mobility=True)
            lat.hp_set_anisotropy(ang, 90000, 500, J, m)
        lat.hp_set_sweep_kernel(kind)
        lat.hp_sweep(7)
        torch.cuda.synchronize()
        got.append((q.cpu().numpy(), mp.cpu().numpy()))
        lat.close()
    np.testing.assert_array_equal(got[0][0], got[1][0])
    np.testing.assert_array_equal(got[0][1], got[1][1])
