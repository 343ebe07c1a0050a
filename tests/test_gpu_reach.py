"""FP64 subvolume factorisations that stop at the last row a column's point couples to: extents that differ per
axis, time functions that straddle the 16-row blocks, ragged tails, Galerkin subvolumes wider than the box
stencil, and the square form's pivoted LU; coloured passes and V-cycles against the oracle at the parity bound
of every fixed schedule (1e-11)."""
import dataclasses

import numpy as np
import pytest

from oracle import multigrid, relax, system
from oracle.propagate import numpy_coarse_sub, numpy_sub
from paper_1111_4363_gb300 import workloads as wl
from tests.helpers import gpu_context, oracle_system, rel_l2

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()


def case(dim, n, sub, K, **kw):
    base = {1: wl.harmonic_1d, 2: wl.softcore_2d, 3: wl.hydrogen_3d}[dim]()
    kw = dict(dict(levels=1, coarse_sub=None), **kw)
    return dataclasses.replace(base, n=n, sub=sub, nt=K, coarse_nu=None, coarse_sweeps=2, psi_kind="gaussian", seed=4, **kw)


LSQ = [case(2, (12, 7, 1), (5, 3, 1), 5), case(2, (9, 8, 1), (8, 4, 1), 4), case(2, (6, 9, 1), (2, 8, 1), 7),
       case(3, (8, 5, 4), (4, 2, 3), 3), case(1, (37, 1, 1), (16, 1, 1), 7), case(1, (9, 1, 1), (2, 1, 1), 1)]


@pytest.mark.parametrize("w", LSQ, ids=lambda w: f"{w.dim}d_{w.sub}_K{w.nt}")
def test_coloured_passes(w):
    psi0 = wl.initial_state(w).ravel()
    prob, M, f, W = oracle_system(w, psi0, 0.35)
    G, g = (M.conj().T @ W @ M).tocsr(), M.conj().T @ (W @ f)
    R = relax.BlockRelaxation(G, prob.shape, numpy_sub(w), prob.K)
    with gpu_context(w) as ctx:
        for colour in range(1 << w.dim):
            ref = wl.random_state(M.shape[1], 5) * 0.05
            got = ref.copy()
            R.colour_pass(ref, g, colour)
            ctx.relax_colour(psi0, 0.35, colour, got)
            assert rel_l2(got, ref) < 1e-11, colour


@pytest.mark.parametrize("n,sub,K", [((20, 16, 1), (4, 4, 1), 2), ((16, 24, 1), (5, 3, 1), 4), ((8, 12, 8), (3, 2, 3), 2)])
def test_wide_galerkin_subvolumes(n, sub, K):
    w = case(3 if n[2] > 1 else 2, n, sub, K, levels=2, coarse_sub=sub, nu1=1, nu2=1)
    psi0 = wl.initial_state(w).ravel()
    prob, M, f, W = oracle_system(w, psi0, 0.2)
    ref = multigrid.solve_step(M, f, W, prob.shape, prob.K, numpy_sub(w), 2, 1, 1, 2, ncycles=2,
                               coarse_sub=numpy_coarse_sub(w))[0]
    with gpu_context(w) as ctx:
        c = np.zeros(w.nunknowns, dtype=np.complex128)
        ctx.solve_step(psi0, 0.2, c, ncycles=2)
    assert rel_l2(c, ref) < 1e-11


@pytest.mark.parametrize("w", [case(2, (12, 7, 1), (5, 3, 1), 5, local_form="square"),
                               case(3, (6, 5, 4), (2, 2, 3), 8, local_form="square"),
                               case(1, (25, 1, 1), (9, 1, 1), 6, local_form="square"),
                               case(2, (5, 4, 1), (1, 3, 1), 3, local_form="square")],
                         ids=lambda w: f"{w.dim}d_{w.sub}_K{w.nt}")
def test_square_passes(w):
    psi0 = wl.initial_state(w).ravel()
    prob, M, f, W = oracle_system(w, psi0, 0.35)
    R = relax.SquareRelaxation(M, prob.shape, numpy_sub(w), prob.K)
    with gpu_context(w) as ctx:
        for colour in range(2):
            ref = wl.random_state(M.shape[1], 5) * 0.05
            got = ref.copy()
            R.colour_pass(ref, f, colour)
            ctx.relax_colour(psi0, 0.35, colour, got)
            assert rel_l2(got, ref) < 1e-11, colour
