"""Grain counts and the one-pass measurement where the warp's steps part: lattices
shorter and longer than a warp's 128 sites and its 2048, runs across both, a buffer off
its 16-byte boundary, ids out of range.  Whole numbers: equal to numpy's."""
import numpy as np
import pytest

from tests.gpu_util import need_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L", [(2, 2), (2, 62), (2, 64), (2, 66), (32, 64), (34, 60), (50, 82), (130, 126)])
@pytest.mark.parametrize("shift", [0, 1])
@pytest.mark.parametrize("block", [1, 5, 5000])
def test_counts_and_measure(L, shift, block):
    torch, hm = need_gpu()
    N, G = L[0] * L[1], 300
    rng = np.random.default_rng(N + block)
    q0 = np.repeat(rng.integers(0, G, size=N // block + 1), block)[:N].astype(np.int32)
    buf = torch.zeros(N + shift, dtype=torch.int32, device="cuda")
    q = buf[shift:]
    q.copy_(torch.from_numpy(q0))
    lat = hm.Lattice(2, L, 4, 256, 1, G, hm.FIELD_GRAIN)
    lat.hp_bind(q)
    table = rng.integers(-1000, 1000, size=G).astype(np.int32)
    lat.hp_set_field(torch.from_numpy(table).cuda())
    ang = rng.uniform(0, np.pi / 2, size=G).astype(np.float32)
    counts = torch.empty(G, dtype=torch.int64, device="cuda")
    alive = torch.empty(1, dtype=torch.int32, device="cuda")
    lat.hp_grain_counts(counts, alive)
    ref = np.bincount(q0, minlength=G)
    np.testing.assert_array_equal(counts.cpu().numpy(), ref)
    assert int(alive.item()) == (ref > 0).sum()
    st, hist = lat.hp_measure(hm.ORIENT_ANGLE, torch.from_numpy(ang).cuda())
    bins = np.clip(np.floor(ang.astype(np.float64) * (180.0 / np.pi)).astype(int), 0, 89)
    np.testing.assert_array_equal(hist, np.bincount(bins, weights=ref, minlength=90).astype(np.int64))
    assert st.sites == N and st.alive == (ref > 0).sum() and st.field_sum == int((ref * table.astype(np.int64)).sum())
    q[N - 1] = G
    with pytest.raises(hm.HPError) as e:
        lat.hp_measure(hm.ORIENT_ANGLE, torch.from_numpy(ang).cuda())
    assert e.value.code == hm.HP_ERR_STATE
    lat.close()
