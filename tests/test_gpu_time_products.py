"""The FP64 residual's closed-form products with Ub, Qb and the weights, for every number of time functions and
every weight, and la_residual's in-place paths (device buffers, a host buffer, r written over c, a buffer
that is not 32-byte aligned), against the oracle at the parity bounds of the residual (1e-13) and its norm
(1e-12)."""
import dataclasses

import numpy as np
import pytest

from oracle import system
from paper_1111_4363_gb300 import workloads as wl
from tests.helpers import gpu_context, oracle_system, rel_l2

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("weight", ["dual", "literal", "identity"])
@pytest.mark.parametrize("K", range(1, 9))
def test_residual_and_norm(K, weight):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    w = dataclasses.replace(wl.softcore_2d(n=16, levels=1), n=(17, 18, 1), nt=K, sub=(2, 2, 1), coarse_sub=None,
                            weight=weight)
    psi0 = wl.initial_state(w).ravel()
    prob, M, f, W = oracle_system(w, psi0, 0.35)
    c = wl.random_state(M.shape[1], 3)
    ref = system.residual(M, f, c)
    N = system.action_norm(ref, W)
    with gpu_context(w) as ctx:
        host = np.zeros_like(c)
        assert ctx.residual(psi0, 0.35, c, host) == pytest.approx(N, rel=1e-12)
        cd, pd = torch.from_numpy(c.copy()).cuda(), torch.from_numpy(psi0).cuda()
        rd = torch.zeros_like(cd)
        assert ctx.residual(pd, 0.35, cd, rd) == pytest.approx(N, rel=1e-12)
        odd = torch.zeros(len(c) + 1, dtype=torch.complex128, device="cuda")[1:]   # 16 bytes past an allocation
        odd.copy_(cd)
        ro = torch.zeros(len(c) + 1, dtype=torch.complex128, device="cuda")[1:]
        ctx.residual(pd, 0.35, odd, ro)
        ctx.residual(pd, 0.35, cd, cd)
    for r in (host, rd.cpu().numpy(), ro.cpu().numpy(), cd.cpu().numpy()):
        assert rel_l2(r, ref) < 1e-13
