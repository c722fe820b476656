"""3D lattices with material points on either side of the line between eight and four
warps a window (456 windows a launch): the smallest, ragged widths, the last lattice
below the line and the first beyond it, and ensembles on either side.  Integer arithmetic: bit-exact against the
oracle."""
import numpy as np
import pytest

from paper_1007_3509_gb300 import synth
from tests.gpu_util import need_gpu

pytestmark = pytest.mark.gpu


def _handle(torch, hm, L, mode, seed, G, kT):
    N = int(np.prod(L))
    rng = np.random.default_rng(N)
    q0 = synth.blocky_lattice(L, G, 5, block=4).astype(np.int32)
    mp0 = rng.permutation(N).astype(np.int32)
    n_tab = N if mode == "point" else G
    table = None if mode == "none" else rng.integers(-300, 300, size=n_tab).astype(np.int32)
    lat = hm.Lattice(3, L, 26, 256, seed, G, {"none": hm.FIELD_NONE, "grain": hm.FIELD_GRAIN, "point": hm.FIELD_POINT}[mode])
    q, m = torch.from_numpy(q0).cuda(), torch.from_numpy(mp0).cuda()
    lat.hp_bind(q, m)
    if table is not None:
        lat.hp_set_field(torch.from_numpy(table).cuda())
    lat.hp_set_threshold_table(*hm.hp_build_threshold_table(kT))
    return lat, q, m, q0, mp0, table


@pytest.mark.parametrize("mode", ["none", "grain", "point"])
@pytest.mark.parametrize("L", [(2, 2, 2), (30, 26, 4), (66, 58, 6), (126, 90, 76), (126, 90, 78), (250, 86, 66), (256, 60, 64)])
def test_both_warp_counts_bit_exact(oracle, L, mode):
    torch, hm = need_gpu()
    G, seed, kT = 40, 0xABC0 + L[0], 0.9
    lat, q, m, q0, mp0, table = _handle(torch, hm, L, mode, seed, G, kT)
    lat.hp_sweep(2)
    torch.cuda.synchronize()
    assert hm.hp_sweep_status() == 0
    thr, D = oracle.threshold_table(kT)
    b0 = None if table is None else table[mp0 if mode == "point" else q0]
    rq, _, rm, _ = oracle.sweep(3, L, 26, 256, seed, 0, 2, thr, D, q0, b0, mp0)
    np.testing.assert_array_equal(q.cpu().numpy(), rq)
    np.testing.assert_array_equal(m.cpu().numpy(), rm)
    lat.close()


@pytest.mark.parametrize("mode,mp", [("none", False), ("grain", False), ("none", True), ("grain", True), ("point", True)])
@pytest.mark.parametrize("shapes", [[(34, 30, 6), (64, 28, 4), (2, 2, 2)], [(126, 90, 60), (58, 30, 40), (112, 56, 34)],
                                    [(112, 140, 144), (112, 140, 134)]])
def test_ensembles_bit_exact(oracle, shapes, mode, mp):
    torch, hm = need_gpu()
    kT, members = 0.9, []
    for r, L in enumerate(shapes):
        G, N = 20 + r, int(np.prod(L))
        rng = np.random.default_rng(r)
        q0 = synth.blocky_lattice(L, G, 5 + r, block=4).astype(np.int32)
        mp0 = rng.permutation(N).astype(np.int32) if mp else None
        table = None if mode == "none" else rng.integers(-300, 300, size=N if mode == "point" else G).astype(np.int32)
        lat = hm.Lattice(3, L, 26, 256, 60 + r, G,
                         {"none": hm.FIELD_NONE, "grain": hm.FIELD_GRAIN, "point": hm.FIELD_POINT}[mode])
        q, m = torch.from_numpy(q0).cuda(), torch.from_numpy(mp0).cuda() if mp else None
        lat.hp_bind(q, m)
        if table is not None:
            lat.hp_set_field(torch.from_numpy(table).cuda())
        lat.hp_set_threshold_table(*hm.hp_build_threshold_table(kT))
        members.append((lat, q, m, q0, mp0, table, L, 60 + r))
    ens = hm.Ensemble([v[0] for v in members])
    ens.hp_ensemble_set_variant(11)
    ens.hp_ensemble_sweep(3)
    torch.cuda.synchronize()
    thr, D = oracle.threshold_table(kT)
    for lat, q, m, q0, mp0, table, L, seed in members:
        b0 = None if table is None else table[mp0 if mode == "point" else q0]
        rq, _, rm, _ = oracle.sweep(3, L, 26, 256, seed, 0, 3, thr, D, q0, b0, mp0)
        np.testing.assert_array_equal(q.cpu().numpy(), rq)
        if mp:
            np.testing.assert_array_equal(m.cpu().numpy(), rm)
    ens.close()
    for v in members:
        v[0].close()
