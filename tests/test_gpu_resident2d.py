"""The resident 2D sweep (a lattice kept in a thread-block cluster's shared memory for
the whole call) where its strips, rows and queues part: one CTA and eight, strips of
unequal height, rows shorter and longer than a warp's two runs of 32 columns, edges of
2, dense proposals (a random lattice), a field table or a threshold table too large for
shared memory, several calls, and ensembles of uneven lattices.  Integer arithmetic:
bit-exact against the oracle."""
import numpy as np
import pytest

from paper_1007_3509_gb300 import synth
from tests.gpu_util import need_gpu

pytestmark = pytest.mark.gpu

SHAPES = [(2, 2), (2, 34), (6, 16), (30, 66), (64, 70), (126, 62), (130, 130), (66, 200), (500, 18)]


def _inputs(L, dense, field, G):
    N = L[0] * L[1]
    q0 = synth.random_lattice(L, G, 3) if dense else synth.blocky_lattice(L, G, 4, block=9)
    table = np.random.default_rng(7).integers(-200, 200, size=G).astype(np.int32) if field else None
    return N, q0.astype(np.int32), table


def _handle(torch, hm, L, nbr, G, seed, q0, table, kT):
    lat = hm.Lattice(2, L, nbr, 256, seed, G, hm.FIELD_GRAIN if table is not None else hm.FIELD_NONE)
    q = torch.from_numpy(q0).cuda()
    lat.hp_bind(q)
    if table is not None:
        lat.hp_set_field(torch.from_numpy(table).cuda())
    lat.hp_set_threshold_table(*hm.hp_build_threshold_table(kT))
    return lat, q


@pytest.mark.parametrize("L", SHAPES)
@pytest.mark.parametrize("nbr", [4, 8])
@pytest.mark.parametrize("field", [False, True])
@pytest.mark.parametrize("dense", [False, True])
def test_resident_bit_exact(oracle, L, nbr, field, dense):
    torch, hm = need_gpu()
    G, seed, kT = 12, 0xFEED00000007 + nbr, 0.9
    N, q0, table = _inputs(L, dense, field, G)
    lat, q = _handle(torch, hm, L, nbr, G, seed, q0, table, kT)
    lat.hp_set_sweep_counter((1 << 32) - 3)   # the sweep word wraps during the run
    lat.hp_sweep(4)
    lat.hp_sweep(5)
    torch.cuda.synchronize()
    assert lat.hp_get_sweep_counter() == (1 << 32) + 6
    thr, D = oracle.threshold_table(kT)
    b0 = None if table is None else table[q0]
    ref = q0
    for s0, n in (((1 << 32) - 3, 3), (0, 6)):
        ref, b0, _, _ = oracle.sweep(2, L, nbr, 256, seed, s0, n, thr, D, ref, b0 if table is None else table[ref], None)
    np.testing.assert_array_equal(q.cpu().numpy(), ref)
    lat.close()


def test_tables_larger_than_shared_memory(oracle):
    """G = 60000 energies (240 KB) and a threshold table of kT = 12 (68000 entries)."""
    torch, hm = need_gpu()
    L, G, kT, seed = (96, 64), 60_000, 12.0, 5
    rng = np.random.default_rng(1)
    q0 = rng.integers(0, G, size=L[0] * L[1]).astype(np.int32)
    table = rng.integers(-4000, 4000, size=G).astype(np.int32)
    thr, D = hm.hp_build_threshold_table(kT, cap=1 << 18)
    lat = hm.Lattice(2, L, 8, 256, seed, G, hm.FIELD_GRAIN)
    q = torch.from_numpy(q0).cuda()
    lat.hp_bind(q)
    lat.hp_set_field(torch.from_numpy(table).cuda())
    lat.hp_set_threshold_table(thr, D)
    lat.hp_sweep(5)
    torch.cuda.synchronize()
    ref, _, _, _ = oracle.sweep(2, L, 8, 256, seed, 0, 5, thr, D, q0, table[q0], None)
    np.testing.assert_array_equal(q.cpu().numpy(), ref)
    lat.close()


@pytest.mark.parametrize("nbr", [4, 8])
def test_resident_ensemble(oracle, nbr):
    """65 members (two launches) of uneven size, temperature and counter; the tile
    path of the same ensemble gives the same lattices."""
    torch, hm = need_gpu()
    G, n = 9, 6
    members, refs = [], []
    for r in range(65):
        L = [(64, 64), (40, 98), (128, 16), (22, 30)][r % 4]
        kT, seed = 0.5 + 0.01 * r, 900 + r
        N, q0, table = _inputs(L, r % 3 == 0, True, G)
        lat, q = _handle(torch, hm, L, nbr, G, seed, q0, table, kT)
        lat.hp_set_sweep_counter(r)
        members.append((lat, q))
        thr, D = oracle.threshold_table(kT)
        refs.append((q0, oracle.sweep(2, L, nbr, 256, seed, r, n, thr, D, q0, table[q0], None)[0]))
    ens = hm.Ensemble([m[0] for m in members])
    ens.hp_ensemble_sweep(n)
    torch.cuda.synchronize()
    for (lat, q), (q0, ref) in zip(members, refs):
        np.testing.assert_array_equal(q.cpu().numpy(), ref)
        assert lat.hp_get_sweep_counter() % 65 == (members.index((lat, q)) + n) % 65
        lat.hp_set_spins(torch.from_numpy(q0).cuda())
        lat.hp_set_sweep_counter(lat.hp_get_sweep_counter() - n)
    ens.hp_ensemble_set_variant(0)
    ens.hp_ensemble_sweep(n)
    torch.cuda.synchronize()
    for (lat, q), (_, ref) in zip(members, refs):
        np.testing.assert_array_equal(q.cpu().numpy(), ref)
    chosen, ms = ens.hp_ensemble_autotune(2)
    assert 0 <= chosen < hm.hp_sweep_variants(nbr) and (ms > 0).any()
    for (lat, q), (_, ref) in zip(members, refs):
        np.testing.assert_array_equal(q.cpu().numpy(), ref)
    ens.close()
    for lat, _ in members:
        lat.close()
