"""Sweeps of several MCS in one call, whose launches overlap on the stream: grids of less
than a wave and of many, 2D and 3D, with and without material points and misorientation
tables, odd and even numbers of MCS, and the same call replayed from a captured graph.
Bit-exact against one call per MCS and, where it is small, against the oracle."""
import numpy as np
import pytest

from paper_1007_3509_gb300 import synth
from tests.gpu_util import need_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dim,L,nbr", [(2, (256, 64), 4), (2, (700, 504), 8), (2, (3360, 2100), 8), (3, (64, 60, 16), 26),
                                       (3, (66, 34, 8), 6), (3, (256, 256, 130), 26), (3, (250, 198, 64), 26)])
@pytest.mark.parametrize("point", [False, True])
@pytest.mark.parametrize("aniso", [False, True])
def test_one_call_and_many(oracle, dim, L, nbr, point, aniso):
    torch, hm = need_gpu()
    Q, seed = 40, 11
    N = int(np.prod(L))
    rng = np.random.default_rng(3)
    q0 = synth.blocky_lattice(L, Q, 5, block=6).astype(np.int32)
    mp0 = rng.permutation(N).astype(np.int32)
    table = rng.integers(-60, 60, size=N if point else Q).astype(np.int32)
    lat = hm.Lattice(dim, L, nbr, 256, seed, Q, hm.FIELD_POINT if point else hm.FIELD_GRAIN)
    q = torch.empty(N, dtype=torch.int32, device="cuda")
    mp = torch.empty(N, dtype=torch.int32, device="cuda") if point else None
    lat.hp_bind(q, mp)
    tt = torch.from_numpy(table).cuda()
    lat.hp_set_field(tt)
    lat.hp_set_threshold_table(*hm.hp_build_threshold_table(0.8))
    if aniso:
        ang = torch.from_numpy(rng.integers(0, 90000, size=Q).astype(np.int32)).cuda()
        J, m = hm.hp_build_read_shockley(1.0, 15.0, 500, 91, 1000, mobility=True)
        lat.hp_set_anisotropy(ang, 90000, 500, J, m)
    elif nbr != 6:
        lat.hp_set_sweep_variant({4: 3, 8: 4, 26: 11}[nbr])
    d0, dm = torch.from_numpy(q0).cuda(), torch.from_numpy(mp0).cuda()

    def start():
        q.copy_(d0)
        if point:
            mp.copy_(dm)
        lat.hp_set_sweep_counter(2)

    def state():
        torch.cuda.synchronize()
        return q.cpu().numpy(), (mp.cpu().numpy() if point else None)

    for n in (5, 8):
        start()
        lat.hp_sweep(n)
        got = state()
        start()
        for _ in range(n):
            lat.hp_sweep(1)
            torch.cuda.synchronize()
        ref = state()
        start()
        graph = torch.cuda.CUDAGraph()
        torch.cuda.synchronize()
        with torch.cuda.graph(graph):
            lat.hp_sweep(n)
        start()
        graph.replay()
        rep = state()
        for a, b, c in zip(got, ref, rep):
            if a is not None:
                np.testing.assert_array_equal(a, b)
                np.testing.assert_array_equal(c, b)
    if N <= 400000 and not aniso:
        thr, D = oracle.threshold_table(0.8)
        want = oracle.sweep(dim, L, nbr, 256, seed, 2, 8, thr, D, q0, table[mp0] if point else table[q0], mp0)
        np.testing.assert_array_equal(got[0], want[0])
    lat.close()
