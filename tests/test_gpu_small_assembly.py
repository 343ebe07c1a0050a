"""H^2 of a point pair in the complex64 factorisation of at most 32 unknowns is formed in FP64 and rounded once.

Neighbouring points whose diagonal entries D = dsum + V0 nearly cancel have (H^2)_pq = -w (D_p + D_q), which a sum of
rounded diagonals loses.  One time function, no field, V0 alternating between +-10^4, and a source whose normal
residual is nonzero at the subvolume's first point only: then the second point's correction is -G_10 / G_11 times the
first's up to terms of order w^2 / D^2, and keeps the relative accuracy of G_10.

Tolerance: 64 u, u = 2^-24, for the fewer than 64 rounded operations between that entry and the result; a sum of
rounded diagonals is off by up to D u / |D_p + D_q| = 2e-3."""
import dataclasses

import numpy as np
import pytest

from paper_1111_4363_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sub", [2, 3, 16, 17, 20, 32])
def test_cancelling_diagonals_keep_their_sum(sub):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from oracle import system
    from paper_1111_4363_gb300 import binding as B
    n = 3 * sub
    w = dataclasses.replace(wl.harmonic_1d(), n=(n, 1, 1), h=(0.5, 1.0, 1.0), nt=1, dt=0.5, sub=(sub, 1, 1), levels=1,
                            coarse_sub=None, coarse_nu=None, pulse=None)
    V0 = (-1.0) ** np.arange(n) * 1e4 + np.random.default_rng(7).uniform(0.1, 0.3, n) - 4.0   # D = V0 + 4
    psi0 = np.zeros(n, dtype=np.complex128)
    psi0[sub - 2] = 1.0
    prob = dataclasses.replace(system.Problem.from_workload(w), V0=V0)
    M, f, W = system.assemble(prob, 0.0, psi0, w.weight)
    G, g = (M.conj().T @ W @ M).toarray(), M.conj().T @ (W @ f)
    U = np.arange(sub, 2 * sub)
    assert g[U][0] != 0 and not g[U][1:].any()
    want = np.linalg.solve(G[np.ix_(U, U)], g[U])
    got = np.zeros(n, dtype=np.complex128)
    with B.Context(B.config_from_workload(w, precision=1)) as ctx:
        ctx.set_hamiltonian(V0, None)
        ctx.relax_colour(psi0, 0.0, 1, got)
    tol = 64 * 2.0 ** -24
    assert abs(got[U][0] - want[0]) <= tol * abs(want[0])
    assert abs(got[U][1] - want[1]) <= tol * abs(want[1])
