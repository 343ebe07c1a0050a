"""Galerkin operators of 1D grids around the first level's chunk of 64 coarse points and down to two points: fixed
V-cycles over every level against the oracle's assembled I^T G I."""
import dataclasses

import numpy as np
import pytest

from oracle import multigrid
from oracle.propagate import numpy_coarse_sub, numpy_sub
from paper_1111_4363_gb300 import workloads as wl
from tests.helpers import gpu_context, oracle_system, rel_l2

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,levels", [(4, 2), (126, 2), (128, 3), (132, 3), (392, 4), (64, 6)])
def test_vcycles_over_all_levels_match_the_oracle(n, levels):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    pulse = wl.Pulse(amp=[0.4], omega=[1.3], t_center=[0.0], sigma=[0.0], axis=0)
    w = dataclasses.replace(wl.harmonic_1d(), n=(n, 1, 1), h=(0.25, 1.0, 1.0), nt=2, sub=(2, 1, 1), coarse_sub=(2, 1, 1),
                            levels=levels, nu1=1, nu2=1, coarse_sweeps=2, pulse=pulse, coarse_nu=None,
                            psi_kind="gaussian", seed=3)
    psi0 = wl.initial_state(w).ravel()
    prob, M, f, W = oracle_system(w, psi0, 0.4)
    ref = multigrid.solve_step(M, f, W, prob.shape, prob.K, numpy_sub(w), w.levels, w.nu1, w.nu2, w.coarse_sweeps,
                               ncycles=2, coarse_sub=numpy_coarse_sub(w))[0]
    with gpu_context(w) as ctx:
        c = np.zeros(w.nunknowns, dtype=np.complex128)
        ctx.solve_step(psi0, 0.4, c, ncycles=2)
    assert rel_l2(c, ref) < 1e-11      # the parity bound of every fixed schedule
