"""The complex64 factorisation of subvolumes of at most 32 unknowns (stored as the inverse of L) and the solves
with it: one coloured pass in mixed precision from c = 0 against the oracle's exact block minimisation, for both
size classes, time functions that leave padding rows, single points per time function and ragged tails; and
mixed V-cycles on Galerkin levels of such subvolumes, which must converge to the direct solution.

Tolerance of a pass: as for the larger factors, 8 sqrt(n) cond(G_UU) u with u = 2^-24 (assembly, elimination and
two mat-vecs with the inverse are backward stable up to sums of n rounded terms)."""
import dataclasses

import numpy as np
import pytest

from oracle import relax, system
from oracle.propagate import numpy_sub
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
    return dataclasses.replace(base, n=n, sub=sub, nt=K, coarse_nu=None, psi_kind="gaussian", seed=2, **kw)


CASES = [case(2, (9, 7, 1), (4, 2, 1), 4), case(2, (5, 8, 1), (2, 2, 1), 4), case(2, (7, 6, 1), (2, 2, 1), 6),
         case(1, (50, 1, 1), (16, 1, 1), 2), case(1, (70, 1, 1), (32, 1, 1), 1), case(1, (6, 1, 1), (2, 1, 1), 8),
         case(1, (13, 1, 1), (4, 1, 1), 8), case(3, (5, 4, 3), (2, 2, 2), 3), case(2, (11, 7, 1), (5, 3, 1), 2),
         case(2, (5, 5, 1), (2, 2, 1), 1), case(1, (11, 1, 1), (3, 1, 1), 5), case(1, (9, 1, 1), (4, 1, 1), 7),
         case(2, (120, 120, 1), (2, 2, 1), 4)]     # the last: enough matrices for four warps per CTA


@pytest.mark.parametrize("w", CASES, ids=lambda w: f"{w.dim}d_{w.n}_{w.sub}_K{w.nt}")
def test_mixed_pass(w):
    psi0 = wl.initial_state(w).ravel()
    prob, M, f, W = oracle_system(w, psi0, 0.35)
    G, g = (M.conj().T @ W @ M).tocsr(), M.conj().T @ (W @ f)
    R = relax.BlockRelaxation(G, prob.shape, numpy_sub(w), prob.K)
    some = [(col, idx) for col, idx, _ in R.blocks][:: max(1, len(R.blocks) // 40)]
    cond = max(np.linalg.cond(G[idx][:, idx].toarray()) for _, idx in some)
    n = max(len(idx) for _, idx, _ in R.blocks)
    tol = 8.0 * np.sqrt(n) * cond * 2.0 ** -24
    assert tol < 0.1
    with gpu_context(w, precision=1) as ctx:
        for colour in range(1 << w.dim):
            ref = np.zeros(M.shape[1], dtype=np.complex128)
            R.colour_pass(ref, g, colour)
            got = np.zeros_like(ref)
            ctx.relax_colour(psi0, 0.35, colour, got)
            assert np.linalg.norm(got - ref) <= tol * np.linalg.norm(ref), colour


@pytest.mark.parametrize("w", [case(2, (24, 16, 1), (4, 4, 1), 4, levels=3, coarse_sub=(2, 2, 1)),
                               case(2, (20, 12, 1), (4, 2, 1), 3, levels=3, coarse_sub=(2, 2, 1)),
                               case(3, (8, 12, 8), (2, 2, 2), 4, levels=2, coarse_sub=(2, 2, 2)),
                               case(1, (72, 1, 1), (8, 1, 1), 4, levels=3, coarse_sub=(4, 1, 1))],
                         ids=lambda w: f"{w.dim}d_{w.n}_K{w.nt}")
def test_mixed_cycles_converge(w):
    """Refined to N/N(0) <= 1e-22 the coefficients equal the direct solution to 1e-9, in as many cycles as FP64
    takes (one more allowed for the rounding of the last one)."""
    psi0 = wl.initial_state(w).ravel()
    prob, M, f, W = oracle_system(w, psi0, 0.0)
    cd = system.direct_solve(M, f)
    cycles = []
    for precision in (0, 1):
        with gpu_context(w, precision=precision, tol=1e-22, max_cycles=80) as ctx:
            c = np.zeros(M.shape[1], dtype=np.complex128)
            _, (cyc, _, _, rel) = ctx.solve_step(psi0, 0.0, c)
            assert rel <= 1e-22 and rel_l2(c, cd) < 1e-9
            cycles.append(cyc)
    assert cycles[1] <= cycles[0] + 1
