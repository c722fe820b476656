"""2D lattices on the route that their shape chooses (no kernel, no variant set), where the
rules of csrc/routes.h change it.  Integer arithmetic: bit-exact against the oracle."""
import numpy as np
import pytest

from paper_1007_3509_gb300 import synth
from tests.gpu_util import need_gpu

pytestmark = pytest.mark.gpu


def _check(oracle, L, nbr, n, field=True, kT=0.9, sweep0=0, calls=1):
    torch, hm = need_gpu()
    G, seed = 12, 0xBEEF + nbr
    q0 = synth.blocky_lattice(L, G, 4, block=9).astype(np.int32)
    table = np.random.default_rng(7).integers(-200, 200, size=G).astype(np.int32) if field else None
    lat = hm.Lattice(2, L, nbr, 256, seed, G, hm.FIELD_GRAIN if field else hm.FIELD_NONE)
    q = torch.from_numpy(q0).cuda()
    lat.hp_bind(q)
    if field:
        lat.hp_set_field(torch.from_numpy(table).cuda())
    lat.hp_set_threshold_table(*hm.hp_build_threshold_table(kT))
    lat.hp_set_sweep_counter(sweep0)
    launches = hm.hp_kernel_launches()
    for _ in range(calls):
        lat.hp_sweep(n)
    torch.cuda.synchronize()
    launches = hm.hp_kernel_launches() - launches
    assert hm.hp_sweep_status() == 0
    thr, D = oracle.threshold_table(kT)
    ref = oracle.sweep(2, L, nbr, 256, seed, sweep0, n * calls, thr, D, q0, table[q0] if field else None, None)[0]
    np.testing.assert_array_equal(q.cpu().numpy(), ref)
    lat.close()
    return launches


@pytest.mark.parametrize("L,nbr", [((1702, 1702), 8), ((1800, 1800), 8), ((1702, 1702), 4), ((1502, 1502), 8)])
def test_tiles_short_and_tall(oracle, L, nbr):
    _check(oracle, L, nbr, 2)


# launches of one call of n MCS: 1 on a cluster, n times the colours per colour
@pytest.mark.parametrize("L,nbr,launches", [
    ((128, 128), 4, 1), ((256, 64), 4, 1), ((120, 240), 4, 6), ((16, 1024), 4, 6), ((2048, 8), 4, 6), ((8, 2000), 4, 6),
    ((256, 256), 8, 1), ((512, 64), 8, 1), ((64, 512), 8, 1), ((300, 200), 8, 12), ((2000, 30), 8, 12), ((2048, 16), 8, 12),
    ((16, 4000), 8, 12), ((64, 1000), 8, 12)])
@pytest.mark.parametrize("field", [False, True])
def test_small_lattices_by_shape(oracle, L, nbr, launches, field):
    assert _check(oracle, L, nbr, 3, field=field) == launches


# members, launches of one call of 3 MCS: 1 on clusters, 3 of tiles
@pytest.mark.parametrize("shapes,launches", [
    ([(64, 64)] * 5, 1), ([(400, 1000)] + [(64, 64)] * 15, 3), ([(600, 600)] + [(64, 64)] * 7, 3),
    ([(500, 500)] * 24, 1), ([(128, 130), (300, 66), (64, 512)] * 4, 1), ([(72, 64)], 1)])
@pytest.mark.parametrize("nbr", [4, 8])
def test_ensembles_by_shape(oracle, shapes, launches, nbr):
    torch, hm = need_gpu()
    G, n, members = 12, 3, []
    table = np.random.default_rng(7).integers(-200, 200, size=G).astype(np.int32)
    for r, L in enumerate(shapes):
        q0 = synth.blocky_lattice(L, G, r, block=9).astype(np.int32)
        lat = hm.Lattice(2, L, nbr, 256, 40 + r, G, hm.FIELD_GRAIN)
        q = torch.from_numpy(q0).cuda()
        lat.hp_bind(q)
        lat.hp_set_field(torch.from_numpy(table).cuda())
        lat.hp_set_threshold_table(*hm.hp_build_threshold_table(0.5 + 0.02 * r))
        members.append((lat, q, q0, L, 40 + r, 0.5 + 0.02 * r))
    ens = hm.Ensemble([m[0] for m in members])
    ens.hp_ensemble_sweep(n)
    before = hm.hp_kernel_launches()
    ens.hp_ensemble_sweep(n)
    torch.cuda.synchronize()
    assert hm.hp_kernel_launches() - before == launches
    for lat, q, q0, L, seed, kT in members:
        thr, D = oracle.threshold_table(kT)
        ref = oracle.sweep(2, L, nbr, 256, seed, 0, 2 * n, thr, D, q0, table[q0], None)[0]
        np.testing.assert_array_equal(q.cpu().numpy(), ref)
    ens.close()
    for m in members:
        m[0].close()


@pytest.mark.parametrize("L", [(2, 40000), (16, 9000), (64, 2000), (66, 2000), (126, 900)])
@pytest.mark.parametrize("nbr", [4, 8])
@pytest.mark.parametrize("mode", ["none", "grain", "point"])
@pytest.mark.parametrize("tables", [False, True])
def test_narrow_lattices(oracle, L, nbr, mode, tables):
    torch, hm = need_gpu()
    G, n, kT, N = 9, 3, 0.9, L[0] * L[1]
    rng = np.random.default_rng(N)
    q0 = synth.blocky_lattice(L, G, 31, block=3).astype(np.int32)
    ang = rng.integers(0, 90000, size=G).astype(np.int32)
    mp0 = rng.integers(0, N, size=N).astype(np.int32) if mode == "point" else None
    table = None if mode == "none" else rng.integers(-40, 40, size=N if mode == "point" else G).astype(np.int32)
    lat = hm.Lattice(2, L, nbr, 256, 0xA11, G, {"none": hm.FIELD_NONE, "grain": hm.FIELD_GRAIN, "point": hm.FIELD_POINT}[mode])
    q, m = torch.from_numpy(q0).cuda(), None if mp0 is None else torch.from_numpy(mp0).cuda()
    lat.hp_bind(q, m)
    if table is not None:
        lat.hp_set_field(torch.from_numpy(table).cuda())
    lat.hp_set_threshold_table(*hm.hp_build_threshold_table(kT))
    thr, D = oracle.threshold_table(kT)
    b = None if table is None else table[q0 if mode == "grain" else mp0]
    if tables:
        J, mob = hm.hp_build_read_shockley(1.0, 15.0, 500, 91, 1000, mobility=True)
        ta = torch.from_numpy(ang).cuda()
        lat.hp_set_anisotropy(ta, 90000, 500, J, mob)
        rq, _, rm, _ = oracle.sweep_aniso(2, L, nbr, 0xA11, 0, n, thr, D, q0, ang, 90000, 500, J, mob, b, mp0)
    else:
        rq, _, rm, _ = oracle.sweep(2, L, nbr, 256, 0xA11, 0, n, thr, D, q0, b, mp0)
    lat.hp_sweep(n)
    torch.cuda.synchronize()
    np.testing.assert_array_equal(q.cpu().numpy(), rq)
    if mp0 is not None:
        np.testing.assert_array_equal(m.cpu().numpy(), rm)
    lat.close()
