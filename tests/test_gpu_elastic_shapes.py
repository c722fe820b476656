"""The elastic solve's transforms at the edges of their range: axes of length 1, 2,
4, 8 (one pass, fewer than eight points a thread), 16 and 1024 (passes of unequal
radix, lines across several warps), ragged last blocks, and both ways to start and
to stop, against the FP64 oracle (the tolerance of the oracle comparison of the
solve: 2e-5 of the largest mean strain component)."""
import numpy as np
import pytest

from paper_1007_3509_gb300 import synth
from tests.gpu_util import need_gpu

pytestmark = pytest.mark.gpu

C = synth.TABLE1
E1 = np.array([8e-4, -3e-4, -6e-4, 2e-4, -1e-4, 3e-4])


def _case(shape, G, seed):
    N = int(np.prod(shape))
    rng = np.random.default_rng(seed)
    q = rng.normal(size=(G, 4)).astype(np.float32)
    q /= np.linalg.norm(q, axis=1, keepdims=True)
    return rng.integers(0, G, size=N).astype(np.int32), q, (rng.normal(size=(N, 6)) * 2e-4).astype(np.float32)


@pytest.mark.parametrize("shape", [(1, 8, 4), (2, 4, 8), (4, 2, 1), (8, 1, 2), (16, 4, 2), (1, 1, 8), (8, 1, 1),
                                   (1024, 2, 2), (2, 1024, 2), (2, 4, 1024), (64, 512, 1), (512, 2, 4), (4, 128, 32),
                                   (32, 2, 256)])
@pytest.mark.parametrize("fixed", [False, True])
def test_solve_shapes(shape, fixed):
    """fixed: the iteration count stops the solve (the last update writes the stress)
    and the strain starts from a given field; else the tolerance does, from the mean."""
    torch, hm = need_gpu()
    from oracle import elastic
    grain, quat, epc = _case(shape, 5, sum(shape))
    N = int(np.prod(shape))
    ref_e, ref_s, _, _ = elastic.solve(shape, grain, quat, (C["C11"], C["C12"], C["C44"]), E1,
                                       eps_p=epc.astype(np.float64), tol=1e-11)
    prm = hm.cp_params(C["C11"], C["C12"], C["C44"], C["tau0"], C["taus"], C["h0"], C["beta"], 1e-4)
    eps = torch.from_numpy(np.repeat(E1.astype(np.float32)[:, None], N, axis=1).copy()).cuda().reshape(-1)
    sig = torch.full((6 * N,), float("nan"), device="cuda")
    if not fixed:
        eps.fill_(float("nan"))
    it, _ = hm.hp_elastic_solve(prm, shape, torch.from_numpy(grain).cuda(), torch.from_numpy(quat).cuda(), E1, eps,
                                eps_p=torch.from_numpy(np.ascontiguousarray(epc.T)).cuda(), sigma=sig,
                                tol=1e-30 if fixed else 1e-6, max_iter=40 if fixed else 200, start_from_mean=not fixed)
    torch.cuda.synchronize()
    assert it == 40 if fixed else it < 100
    ge, gs = (v.view(6, N).cpu().numpy().T for v in (eps, sig))
    emax, smax = np.abs(E1).max(), np.abs(ref_s).max()
    assert np.abs(ge - ref_e).max() <= 2e-5 * emax
    assert np.abs(gs - ref_s).max() <= 5e-5 * smax
