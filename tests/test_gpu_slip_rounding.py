"""The plasticity return map where its FP32 result is nearly a tie: slips a few 2^-47 off the
middle between two FP32 numbers (powers of two among them) commit the number that FP64
arithmetic rounds to.  Without hardening the slip is the quotient (at - g) / k, so that such
slips can be asked for."""
import numpy as np
import pytest

from paper_1007_3509_gb300 import synth
from tests.gpu_util import need_gpu

pytestmark = pytest.mark.gpu


def test_near_ties_without_hardening():
    torch, hm = need_gpu()
    rng = np.random.default_rng(5)
    f = np.exp(rng.uniform(np.log(1e-7), np.log(1e-2), 200_000)).astype(np.float32)
    f[:4000] = np.exp2(rng.integers(-22, -7, 4000)).astype(np.float32)
    f[2000:4000] = np.nextafter(f[2000:4000], np.float32(0))     # the middle below a power of two
    mid = (f.astype(np.float64) + np.nextafter(f, np.float32(1)).astype(np.float64)) / 2
    off = rng.choice([-4, -2, -1, 1, 2, 4], f.size) * 2.0 ** -47
    at, g = np.full(f.size, 2.0, np.float32), np.ones(f.size, np.float32)
    k = np.float64(1) / (mid * (1 + off))
    exact = (at.astype(np.float64) - g) / k
    assert (np.abs(exact - mid) > 2.0 ** -49 * mid).all()        # what FP64 rounds to is beyond doubt
    c = synth.TABLE1
    prm = hm.cp_params(c["C11"], c["C12"], c["C44"], c["tau0"], c["tau0"], c["h0"], c["beta"], 1e-4)
    x = torch.empty(f.size, dtype=torch.float64, device="cuda")
    hm.hp_debug_return_map(prm, torch.from_numpy(at).cuda(), torch.from_numpy(g).cuda(), torch.from_numpy(k).cuda(), x)
    torch.cuda.synchronize()
    got = x.cpu().numpy()
    assert (np.abs(got - exact) <= 2.0 ** -44 * exact).all()
    np.testing.assert_array_equal(got.astype(np.float32), exact.astype(np.float32))
