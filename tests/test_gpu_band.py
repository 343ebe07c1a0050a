"""The complex64 banded factorisation of finest-level subvolumes of more than 128 unknowns: one coloured
pass in mixed precision from c = 0 against the oracle's exact block minimisation, at window widths 4 and 8,
bands from 1 to 8, time functions that do and do not divide 16, and ragged tails.

Tolerance: the pass solves G_UU delta = rhs with a factor rounded to complex64 (unit roundoff u = 2^-24); the
relative error of delta is at most about cond(G_UU) times the backward error of assembly, factorisation and
the two substitutions, each a sum of up to n rounded terms, sqrt(n) u for independent roundings.  The bound is
8 sqrt(n) cond u with the largest condition number of the pass's blocks."""
import dataclasses

import numpy as np
import pytest

from oracle import relax
from oracle.propagate import numpy_sub
from paper_1111_4363_gb300 import workloads as wl
from tests.helpers import gpu_context, oracle_system

pytestmark = pytest.mark.gpu


def case(dim, n, sub, K):
    base = {1: wl.harmonic_1d, 2: wl.softcore_2d, 3: wl.hydrogen_3d}[dim]()
    return dataclasses.replace(base, n=n, sub=sub, nt=K, levels=1, coarse_sub=None, coarse_nu=None,
                               psi_kind="gaussian", seed=2)


CASES = {
    "3d_4x4x4_K4": case(3, (8, 4, 8), (4, 4, 4), 4),               # band 8
    "3d_4x4x4_K4_ragged": case(3, (7, 5, 6), (4, 4, 4), 4),        # tails of 3, 1 and 2 points
    "3d_4x4x4_K3": case(3, (8, 4, 6), (4, 4, 4), 3),               # 192 unknowns, K does not divide 16
    "2d_8x8_K4": case(2, (16, 13, 1), (8, 8, 1), 4),               # band 4
    "2d_8x8_K3": case(2, (8, 16, 1), (8, 8, 1), 3),                # 192 unknowns
    "2d_5x9_K3": case(2, (11, 20, 1), (5, 9, 1), 3),               # odd extents, tails of 1 and 2 points
    "1d_32_K8": case(1, (80, 1, 1), (32, 1, 1), 8),                # band 1, tail of 16 points
    "1d_64_K3": case(1, (100, 1, 1), (64, 1, 1), 3),               # band 1
}


@pytest.mark.parametrize("name", list(CASES))
def test_mixed_pass_of_wide_subvolumes(name):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    w = CASES[name]
    psi0 = wl.initial_state(w).ravel()
    prob, M, f, W = oracle_system(w, psi0, 0.35)
    G = (M.conj().T @ W @ M).tocsr()
    g = M.conj().T @ (W @ f)
    R = relax.BlockRelaxation(G, prob.shape, numpy_sub(w), prob.K)
    with gpu_context(w, precision=1) as ctx:
        for colour in range(1 << w.dim):
            ref = np.zeros(M.shape[1], dtype=np.complex128)
            R.colour_pass(ref, g, colour)
            got = np.zeros_like(ref)
            ctx.relax_colour(psi0, 0.35, colour, got)
            touched = np.nonzero(ref)[0]
            if len(touched) == 0:
                assert not got.any()
                continue
            cond, nmax = 1.0, 1
            for col, idx, _ in R.blocks:
                if col == colour:
                    cond, nmax = max(cond, np.linalg.cond(G[idx][:, idx].toarray())), max(nmax, len(idx))
            tol = 8.0 * np.sqrt(nmax) * cond * 2.0 ** -24
            err = np.linalg.norm(got - ref) / np.linalg.norm(ref)
            assert err < tol < 0.1, (colour, err, tol)
