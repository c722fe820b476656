"""Branches of the Monte Carlo plasticity increment that Table 1 does not reach."""
import numpy as np
import pytest

from paper_1007_3509_gb300 import synth
from tests.gpu_util import need_gpu

pytestmark = pytest.mark.gpu


def test_plasticity_without_hardening_and_with_uniform_choice(oracle):
    """The branches of the increment that Table 1 does not reach: no hardening (taus =
    tau0: the slip is (|tau| - g)/k and g stays), beta = 0 (every candidate equally
    likely) and a point count that is no multiple of a warp, against the FP64 oracle
    away from decision ties (relative stress 1e-5, as for the increment itself)."""
    torch, hm = need_gpu()
    c = dict(synth.TABLE1)
    P, G = 1003, 17
    quat = synth.random_quaternions(G, 11)
    grain = np.random.default_rng(2).integers(0, G, size=P).astype(np.int32)
    for taus, beta in ((c["tau0"], c["beta"]), (c["taus"], 0.0)):
        prm = hm.cp_params(c["C11"], c["C12"], c["C44"], c["tau0"], taus, c["h0"], beta, 1e-4)
        eps, gam, g = (torch.empty(k * P, device="cuda") for k in (6, 1, 1))
        sig = torch.empty(6 * P, device="cuda")
        hm.hp_cp_reset(prm, P, eps, gam, g)
        hm.hp_cp_step(prm, 77, torch.from_numpy(grain).cuda(), torch.from_numpy(quat).cuda(), 0, 6, eps, gam, g, sigma=sig)
        torch.cuda.synchronize()
        por = oracle.cp_params(c["C11"], c["C12"], c["C44"], c["tau0"], taus, c["h0"], beta, 1e-4)
        _, _, ref, near_r, near_t = oracle.mcp_run(por, 77, grain, quat, 0, 6, np.zeros((P, 6)), np.zeros(P))
        ok = (near_r > 1e-5) & (near_t > 1e-5)
        assert ok.mean() > 0.5
        s = sig.view(6, P).cpu().numpy().T
        assert (np.abs(s - ref).max(axis=1)[ok] <= 1e-5 * np.abs(ref).max(axis=1)[ok]).all()
        if taus == c["tau0"]:
            assert (g.cpu().numpy() == np.float32(c["tau0"])).all()
