"""The autotuner leaves a lattice on its own route where that beats every variant: one launch
per colour, or one of a cluster, which are none of the variants.  The route shows in the
launches of a call."""
import numpy as np
import pytest

from paper_1007_3509_gb300 import synth
from tests.gpu_util import need_gpu

pytestmark = pytest.mark.gpu

N_MCS = 20


# launches of one call of N_MCS
@pytest.mark.parametrize("L,nbr,point,tables,launches", [
    ((256, 256), 4, False, False, 2 * N_MCS), ((256, 250), 4, True, False, 2 * N_MCS), ((300, 200), 8, False, False, None),
    ((64, 64), 4, False, False, 1), ((128, 128), 8, False, False, 1), ((16, 9000), 8, True, False, 4 * N_MCS),
    ((1024, 1024), 8, False, False, N_MCS), ((128, 128), 4, False, True, 2 * N_MCS), ((256, 256), 8, False, True, N_MCS)])
def test_autotuned_route(oracle, L, nbr, point, tables, launches):
    torch, hm = need_gpu()
    G, seed, kT, N = 30, 77, 0.7, L[0] * L[1]
    rng = np.random.default_rng(N)
    q0 = synth.blocky_lattice(L, G, 4, block=25).astype(np.int32)
    mp0 = rng.permutation(N).astype(np.int32) if point else None
    table = rng.integers(-30, 30, size=N if point else G).astype(np.int32)
    lat = hm.Lattice(2, L, nbr, 256, seed, G, hm.FIELD_POINT if point else hm.FIELD_GRAIN)
    q, m = torch.from_numpy(q0).cuda(), torch.from_numpy(mp0).cuda() if point else None
    lat.hp_bind(q, m)
    lat.hp_set_field(torch.from_numpy(table).cuda())
    lat.hp_set_threshold_table(*hm.hp_build_threshold_table(kT))
    if tables:
        ang = rng.integers(0, 90000, size=G).astype(np.int32)
        J, mob = hm.hp_build_read_shockley(1.0, 15.0, 500, 91, 1000, mobility=True)
        ta = torch.from_numpy(ang).cuda()
        lat.hp_set_anisotropy(ta, 90000, 500, J, mob)
    chosen, ms = lat.hp_sweep_autotune(N_MCS)
    assert 0 <= chosen < hm.hp_sweep_variants(nbr) and ms[chosen] > 0
    assert lat.hp_get_sweep_counter() == 0
    np.testing.assert_array_equal(q.cpu().numpy(), q0)
    if point:
        np.testing.assert_array_equal(m.cpu().numpy(), mp0)
    before = hm.hp_kernel_launches()
    lat.hp_sweep(N_MCS)
    torch.cuda.synchronize()
    if launches is not None:
        assert hm.hp_kernel_launches() - before == launches
    thr, D = oracle.threshold_table(kT)
    b = table[mp0 if point else q0]
    if tables:
        ref = oracle.sweep_aniso(2, L, nbr, seed, 0, N_MCS, thr, D, q0, ang, 90000, 500, J, mob, b, None)[0]
    else:
        ref = oracle.sweep(2, L, nbr, 256, seed, 0, N_MCS, thr, D, q0, b, mp0)[0]
    np.testing.assert_array_equal(q.cpu().numpy(), ref)
    lat.close()
