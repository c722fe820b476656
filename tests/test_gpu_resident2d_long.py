"""The resident 2D sweep where the other tests do not reach: more MCS in a call than one
launch holds, and strips of more lines than a block has warps, so that a warp goes through
several (in an ensemble: a handle by itself sweeps such lattices per colour).  Integer
arithmetic: bit-exact against the oracle."""
import numpy as np
import pytest

from paper_1007_3509_gb300 import synth
from tests.gpu_util import need_gpu

pytestmark = pytest.mark.gpu


def _member(torch, hm, L, nbr, seed, G, table, kT):
    q0 = synth.blocky_lattice(L, G, seed, block=7).astype(np.int32)
    lat = hm.Lattice(2, L, nbr, 256, seed, G, hm.FIELD_GRAIN)
    q = torch.from_numpy(q0).cuda()
    lat.hp_bind(q)
    lat.hp_set_field(torch.from_numpy(table).cuda())
    lat.hp_set_threshold_table(*hm.hp_build_threshold_table(kT))
    return lat, q, q0


@pytest.mark.parametrize("nbr", [4, 8])
@pytest.mark.parametrize("members", [1, 3])
def test_more_mcs_than_a_launch_holds(oracle, nbr, members):
    torch, hm = need_gpu()
    L, G, n, kT = (34, 38), 12, 4096 + 5, 0.9
    table = np.random.default_rng(1).integers(-60, 60, size=G).astype(np.int32)
    lats = [_member(torch, hm, L, nbr, 50 + r, G, table, kT) for r in range(members)]
    for lat, _, _ in lats:
        lat.hp_set_sweep_counter((1 << 32) - 4000)   # the sweep word wraps in the first launch
    before = hm.hp_kernel_launches()
    if members == 1:
        lats[0][0].hp_sweep(n)
    else:
        ens = hm.Ensemble([v[0] for v in lats])
        ens.hp_ensemble_sweep(n)
    torch.cuda.synchronize()
    assert hm.hp_kernel_launches() - before == 2
    thr, D = oracle.threshold_table(kT)
    for r, (lat, q, q0) in enumerate(lats):
        assert lat.hp_get_sweep_counter() == (1 << 32) - 4000 + n
        ref = oracle.sweep(2, L, nbr, 256, 50 + r, (1 << 32) - 4000, 4000, thr, D, q0, table[q0], None)[0]
        ref = oracle.sweep(2, L, nbr, 256, 50 + r, 0, n - 4000, thr, D, ref, table[ref], None)[0]
        np.testing.assert_array_equal(q.cpu().numpy(), ref)
    if members > 1:
        ens.close()
    for v in lats:
        v[0].close()


@pytest.mark.parametrize("nbr", [4, 8])
@pytest.mark.parametrize("L", [(64, 1002), (72, 1000), (130, 618)])
def test_several_lines_to_a_warp(oracle, nbr, L):
    torch, hm = need_gpu()
    G, n = 12, 3
    table = np.random.default_rng(2).integers(-200, 200, size=G).astype(np.int32)
    lats = [_member(torch, hm, L, nbr, 70 + r, G, table, 0.6 + 0.02 * r) for r in range(24)]
    ens = hm.Ensemble([v[0] for v in lats])
    before = hm.hp_kernel_launches()
    ens.hp_ensemble_sweep(n)
    torch.cuda.synchronize()
    assert hm.hp_kernel_launches() - before == 1     # clusters: n launches of tiles otherwise
    for r, (lat, q, q0) in enumerate(lats):
        thr, D = oracle.threshold_table(0.6 + 0.02 * r)
        ref = oracle.sweep(2, L, nbr, 256, 70 + r, 0, n, thr, D, q0, table[q0], None)[0]
        np.testing.assert_array_equal(q.cpu().numpy(), ref)
    ens.close()
    for v in lats:
        v[0].close()
