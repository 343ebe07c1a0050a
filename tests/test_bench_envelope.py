"""bench.py's flop count inside a factor's envelope, on the CPU: against the nonzeros and the multiply-adds of actual
factorisations of the oracle's subvolume matrices, and dense local algebra where the reach covers the subvolume."""
import dataclasses

import numpy as np
import pytest

from oracle import relax, system
from oracle.propagate import numpy_sub
from paper_1111_4363_gb300 import workloads as wl
from tests.helpers import oracle_system
from tests.test_bench_contract import bench, fake_profile  # noqa: F401


@pytest.mark.parametrize("n,K", [(96, 6), (24, 4), (7, 1), (128, 8)])
def test_dense_where_the_reach_covers_the_subvolume(bench, n, K):
    fac, sol = bench.envelope_flops(n, K, n, False)
    assert fac == pytest.approx(4.0 / 3.0 * (n ** 3 - n)) and sol == 8.0 * n * n
    fac, sol = bench.envelope_flops(n, K, n, True)
    assert abs(fac - 8.0 / 3.0 * n ** 3) <= 4.0 * n and sol == 8.0 * n * n


@pytest.mark.parametrize("dim,sub,K", [(2, (4, 4, 1), 6), (2, (5, 3, 1), 3), (3, (3, 2, 3), 2), (1, (9, 1, 1), 4)])
def test_envelope_of_the_oracles_factors(bench, dim, sub, K):
    """Every entry of L lies inside, its first and last ones at the bound, so nothing outside is counted and no entry
    is left out; the multiply-adds are those of a right-looking elimination over the envelope."""
    base = {1: wl.harmonic_1d, 2: wl.softcore_2d, 3: wl.hydrogen_3d}[dim]()
    n = tuple(3 * sub[a] if a < dim else 1 for a in range(3))
    w = dataclasses.replace(base, n=n, sub=sub, nt=K, levels=1, coarse_sub=None, coarse_nu=None)
    prob, M, f, W = oracle_system(w, wl.initial_state(w).ravel(), 0.3)
    R = relax.BlockRelaxation((M.conj().T @ W @ M).tocsr(), prob.shape, numpy_sub(w), K)
    idx = next(i for _, i, _ in R.blocks if len(i) == int(np.prod(sub[:dim])) * K)
    Lf = np.linalg.cholesky((M.conj().T @ W @ M).tocsr()[idx][:, idx].toarray())
    m, reach = len(idx), bench.factor_reach(w)
    rows, cols = np.nonzero(np.abs(Lf) > 1e-12 * np.abs(Lf).max())
    assert (rows // K - cols // K).max() == reach
    below = [sum(1 for r in range(j + 1, m) if r // K - j // K <= reach) for j in range(m)]
    fac, sol = bench.envelope_flops(m, K, reach, False)
    assert fac == 4.0 * sum(b * (b + 1) for b in below) and sol == 16.0 * sum(below) + 8.0 * m


def test_square_envelope_holds_under_row_swaps(bench):
    """Pivoted LU of a subvolume matrix: no entry of U beyond the count's last column, none of L beyond its last row."""
    import scipy.linalg as sla
    w = dataclasses.replace(bench.workload("2d-square"), n=(12, 12, 1), nt=4)
    prob = system.Problem.from_workload(w)
    M, f, W = system.assemble(prob, 0.2, wl.initial_state(w).ravel(), w.weight)
    pts = [12 * (4 + y) + 4 + x for y in range(4) for x in range(4)]
    idx = np.concatenate([np.arange(4 * p, 4 * p + 4) for p in pts])
    m, K, reach = len(idx), 4, bench.factor_reach(w)
    assert reach == 4
    last = [min(m - 1, (j // K + reach + 1) * K - 1) for j in range(m)]
    A = M[idx][:, idx].toarray()
    P, L, U = sla.lu(A)
    assert all(not np.any(U[j, last[last[j]] + 1:]) for j in range(m))
    assert all(np.count_nonzero(L[j + 1:, j]) <= last[j] - j for j in range(m))
    fac, _ = bench.envelope_flops(m, K, reach, True)
    assert fac == sum(8.0 * (last[j] - j) * (last[last[j]] - j + 1) for j in range(m))


def test_rooflines_count_the_envelope(bench):  # noqa: F811
    w = bench.workload("2d")
    dense = 4096 * 4.0 / 3.0 * 96 ** 3
    r = bench.dominant_roofline(fake_profile(flops_factor=dense), w, 0, ms_total=20.0, traffic_ok=False)
    e = bench.envelope_roofline(r, w, 0)
    ratio = bench.envelope_flops(96, 6, 8, False)[0] / bench.envelope_flops(96, 6, 96, False)[0]
    assert 0.3 < ratio < 0.9
    assert e["achieved"] == pytest.approx(r["achieved"] * ratio, abs=1e-4)
    assert e["algorithmic_flops"] == pytest.approx(dense * ratio) and e["kernel"] == r["kernel"]
    # wider and complex64 factors: the library's own counts
    w3 = bench.workload("3d")
    r3 = bench.dominant_roofline(fake_profile(), w3, 1, ms_total=20.0, traffic_ok=False)
    assert bench.envelope_roofline(r3, w3, 1) is r3
