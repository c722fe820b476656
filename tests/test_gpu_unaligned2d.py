"""2D sweeps on buffers that start off a 16-byte boundary while the lattice's rows would
allow 16-byte accesses: every fused kernel, with and without misorientation tables.
Integer arithmetic: bit-exact against the oracle."""
import numpy as np
import pytest

from paper_1007_3509_gb300 import synth
from tests.gpu_util import need_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nbr", [4, 8])
@pytest.mark.parametrize("shift", [1, 2, 3])
@pytest.mark.parametrize("variant", [None, 0, 3, 4])
@pytest.mark.parametrize("point,aniso", [(False, False), (True, False), (False, True), (True, True)])
def test_unaligned(oracle, nbr, shift, variant, point, aniso):
    torch, hm = need_gpu()
    L, Q, seed, n = (256, 72), 9, 77, 3
    q0 = synth.blocky_lattice(L, Q, 31, block=3)
    N = q0.size
    rng = np.random.default_rng(5)
    mp0 = rng.integers(0, N, size=N).astype(np.int32)
    table = rng.integers(-40, 40, size=N if point else Q).astype(np.int32)
    b = table[mp0] if point else table[q0]
    lat = hm.Lattice(2, L, nbr, 256, seed, Q, hm.FIELD_POINT if point else hm.FIELD_GRAIN)
    buf, mbuf = (torch.zeros(N + shift, dtype=torch.int32, device="cuda") for _ in range(2))
    q, mp = buf[shift:], mbuf[shift:]
    q.copy_(torch.from_numpy(q0))
    mp.copy_(torch.from_numpy(mp0))
    lat.hp_bind(q, mp if point else None)
    lat.hp_set_field(torch.from_numpy(table).cuda())
    lat.hp_set_threshold_table(*hm.hp_build_threshold_table(0.9))
    thr, D = oracle.threshold_table(0.9)
    if aniso:
        ang = rng.integers(0, 90000, size=Q).astype(np.int32)
        Jtab, mtab = hm.hp_build_read_shockley(1.0, 15.0, 500, 91, 1000, mobility=True)
        ta = torch.from_numpy(ang).cuda()
        lat.hp_set_anisotropy(ta, 90000, 500, Jtab, mtab)
        ref = oracle.sweep_aniso(2, L, nbr, seed, 0, n, thr, D, q0, ang, 90000, 500, Jtab, mtab, b, mp0)
    else:
        ref = oracle.sweep(2, L, nbr, 256, seed, 0, n, thr, D, q0, b, mp0)
    if variant is not None:
        lat.hp_set_sweep_variant(variant)
    lat.hp_sweep(n)
    torch.cuda.synchronize()
    np.testing.assert_array_equal(q.cpu().numpy(), ref[0])
    if point:
        np.testing.assert_array_equal(mp.cpu().numpy(), ref[2])
    lat.close()
