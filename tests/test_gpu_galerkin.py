"""Galerkin level operators (la_set_hamiltonian) through fixed V-cycles over every level, against the oracle's
assembled I^T G I: coarse extents below, at and above the contraction's chunk of 8 points, odd coarse
extents, unequal axes and spacings, the laser on every axis, 1D to 3D, up to four levels."""
import dataclasses

import numpy as np
import pytest

from oracle import multigrid
from oracle.propagate import numpy_coarse_sub, numpy_sub
from paper_1111_4363_gb300 import workloads as wl
from tests.helpers import gpu_context, oracle_system, rel_l2

pytestmark = pytest.mark.gpu

CASES = [  # n, h, levels, K, laser axis, field strength
    ((72, 1, 1), (0.25, 1.0, 1.0), 4, 4, 0),      # level extents 72, 36, 18, 9
    ((8, 1, 1), (0.25, 1.0, 1.0), 3, 2, 0),       # down to two points
    ((36, 20, 1), (0.2, 0.35, 1.0), 3, 2, 1),     # 9 x 5 at the coarsest: one full chunk and one point more
    ((64, 8, 1), (0.2, 0.2, 1.0), 4, 2, 0),       # 8 x 1 at the coarsest
    ((8, 12, 20), (0.3, 0.45, 0.25), 3, 2, 2),    # odd extents 3 and 5 at the coarsest
    ((20, 8, 4), (0.3, 0.25, 0.4), 3, 1, 1),      # one point along z at the coarsest
]


@pytest.mark.parametrize("n,h,levels,K,axis", CASES)
def test_vcycles_over_all_levels_match_the_oracle(n, h, levels, K, axis):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    dim = 3 if n[2] > 1 else (2 if n[1] > 1 else 1)
    base = {1: wl.harmonic_1d, 2: wl.softcore_2d, 3: wl.hydrogen_3d}[dim]()
    pulse = wl.Pulse(amp=[0.4], omega=[1.3], t_center=[0.0], sigma=[0.0], axis=axis)
    two = tuple(2 if a < dim else 1 for a in range(3))
    w = dataclasses.replace(base, n=n, h=h, nt=K, sub=two, coarse_sub=two, levels=levels, nu1=1, nu2=1,
                            coarse_sweeps=2, pulse=pulse, coarse_nu=None, psi_kind="gaussian", seed=3)
    psi0 = wl.initial_state(w).ravel()
    prob, M, f, W = oracle_system(w, psi0, 0.4)
    c_ref = multigrid.solve_step(M, f, W, prob.shape, prob.K, numpy_sub(w), w.levels, w.nu1, w.nu2,
                                 w.coarse_sweeps, ncycles=2, coarse_sub=numpy_coarse_sub(w))[0]
    with gpu_context(w) as ctx:
        c = np.zeros(w.nunknowns, dtype=np.complex128)
        ctx.solve_step(psi0, 0.4, c, ncycles=2)
    assert rel_l2(c, c_ref) < 1e-11      # the parity bound of every fixed schedule
