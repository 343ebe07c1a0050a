"""Wide FP64 solves on both sides of the rule that leaves the products of zero blocks out (more CTAs of a colour than
multiprocessors, band at most half of the block rows): a coloured pass from random coefficients against exact local
minimisations of sampled subvolumes from the oracle's system, at the parity bound of FP64 passes (1e-11)."""
import dataclasses

import numpy as np
import pytest

from paper_1111_4363_gb300 import workloads as wl
from tests.helpers import gpu_context, oracle_system, rel_l2

pytestmark = pytest.mark.gpu


def grid(sub, K, blocks):
    n = (sub[0] * blocks[0] - 1, sub[1] * blocks[1] - 1, 1)   # ragged last subvolumes
    return dataclasses.replace(wl.softcore_2d(n=16, levels=1), n=n, sub=sub, nt=K, coarse_sub=None, coarse_nu=None,
                               psi_kind="gaussian", seed=5)


@pytest.mark.parametrize("sub,K,blocks", [((8, 8, 1), 3, (20, 32)), ((8, 8, 1), 3, (20, 16)), ((16, 4, 1), 4, (20, 32)),
                                          ((8, 8, 1), 4, (24, 26))], ids=str)
def test_pass_equals_local_minimisation(sub, K, blocks):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    w = grid(sub, K, blocks)
    psi0 = wl.initial_state(w).ravel()
    prob, M, f, W = oracle_system(w, psi0, 0.35)
    c0 = wl.random_state(M.shape[1], 3)
    grad = M.conj().T @ (W @ (f - M @ c0))
    got = c0.copy()
    with gpu_context(w) as ctx:
        ctx.relax_colour(psi0, 0.35, 3, got)
    nx, ny = w.n[:2]
    Mc, Wr = M.tocsc(), W.tocsr()
    for bx, by in ((1, 1), (blocks[0] - 1, 1), (1, blocks[1] - 1), (blocks[0] - 1, blocks[1] - 1), (5, 9), (11, 7)):
        pts = [y * nx + x for y in range(by * sub[1], min((by + 1) * sub[1], ny))
               for x in range(bx * sub[0], min((bx + 1) * sub[0], nx))]
        idx = (np.array(pts)[:, None] * K + np.arange(K)).ravel()
        MU = Mc[:, idx]
        want = c0[idx] + np.linalg.solve((MU.conj().T @ Wr @ MU).toarray(), grad[idx])
        assert rel_l2(got[idx], want) < 1e-11, (bx, by)
