"""The lean 3D window kernel where its paths part: how a window is filled (16-byte
copies and boxes, 8-byte copies when Lx % 4 == 2 or the buffer starts on an 8-byte
boundary, single loads when it starts on a 4-byte one), lattices narrower than a
window, and more proposals in a phase than a warp has lanes (a random lattice).
Integer arithmetic: bit-exact against the oracle."""
import numpy as np
import pytest

from paper_1007_3509_gb300 import synth
from tests.gpu_util import need_gpu

pytestmark = pytest.mark.gpu


def _sweep(torch, hm, L, seed, n, kT, q0, mode, table, mp0, shift):
    N = int(np.prod(L))
    lat = hm.Lattice(3, L, 26, 256, seed, int(q0.max()) + 1, mode)
    qb = torch.empty(N + shift, dtype=torch.int32, device="cuda")
    mb = torch.empty(N + shift, dtype=torch.int32, device="cuda")
    q, mp = qb[shift:], mb[shift:]
    q.copy_(torch.from_numpy(q0))
    mp.copy_(torch.from_numpy(mp0))
    lat.hp_bind(q, mp)
    if mode != hm.FIELD_NONE:
        lat.hp_set_field(torch.from_numpy(table).cuda())
    lat.hp_set_threshold_table(*hm.hp_build_threshold_table(kT))
    lat.hp_set_sweep_variant(11)
    lat.hp_sweep(n)
    torch.cuda.synchronize()
    out = q.cpu().numpy(), mp.cpu().numpy()
    lat.close()
    return out


@pytest.mark.parametrize("L,shift", [((250, 62, 6), 0), ((126, 58, 4), 1), ((128, 66, 4), 2), ((62, 34, 4), 0),
                                     ((56, 30, 2), 0), ((2, 4, 6), 0), ((192, 96, 2), 1)])
@pytest.mark.parametrize("mode", [0, 1, 2])
@pytest.mark.parametrize("dense", [False, True])
def test_window_paths_bit_exact(oracle, L, shift, mode, dense):
    torch, hm = need_gpu()
    N, Q, seed, n, kT = int(np.prod(L)), 40, 0xABC0 + shift, 3, 0.8
    q0 = synth.random_lattice(L, Q, 3) if dense else synth.blocky_lattice(L, Q, 4, block=7)
    q0[:Q] = np.arange(Q)[: min(Q, N)] if N >= Q else q0[:Q]
    rng = np.random.default_rng(5)
    mp0 = rng.permutation(N).astype(np.int32)
    G = int(q0.max()) + 1
    table = rng.integers(-300, 300, size=G if mode == 1 else N).astype(np.int32)
    b0 = None if mode == 0 else table[q0] if mode == 1 else table[mp0]
    thr, D = oracle.threshold_table(kT)
    ref_q, _, ref_mp, _ = oracle.sweep(3, L, 26, 256, seed, 0, n, thr, D, q0, b0, mp0)
    q, mp = _sweep(torch, hm, L, seed, n, kT, q0, mode, table, mp0, shift)
    np.testing.assert_array_equal(q, ref_q)
    np.testing.assert_array_equal(mp, ref_mp)
    assert hm.hp_sweep_status() == 0
