"""The kernel names of bench.py's rooflines follow the library's dispatch (CPU): the band against the restatement that
is pinned on the oracle's own factors, and one workload per kernel."""
import dataclasses

import pytest

from paper_1111_4363_gb300 import workloads as wl
from tests.test_bench_contract import bench, fake_profile  # noqa: F401
from tests.test_oracle_band import band_blocks


@pytest.mark.parametrize("dim,sub,K", [(3, (4, 4, 4), 4), (3, (4, 4, 4), 3), (2, (8, 8, 1), 4), (3, (8, 4, 2), 4),
                                       (3, (4, 4, 3), 5), (2, (4, 4, 1), 6), (1, (32, 1, 1), 8), (2, (16, 4, 1), 4)])
def test_band(bench, dim, sub, K):  # noqa: F811
    base = {1: wl.harmonic_1d, 2: wl.softcore_2d, 3: wl.hydrogen_3d}[dim]()
    w = dataclasses.replace(base, sub=sub, nt=K)
    pts = 1
    for a in range(dim):
        pts *= sub[a]
    nblk = -(-pts * K // 16)
    assert bench.band_blocks(w) == min(max(band_blocks(dim, sub, K, nblk), 1), nblk - 1)


def test_names(bench):  # noqa: F811
    w2, w3 = bench.workload("2d"), bench.workload("3d")
    small = dataclasses.replace(w2, sub=(4, 2, 1), nt=4)
    dense = dataclasses.replace(w3, sub=(8, 4, 2), nt=4)       # band 15
    assert bench.finest_kernels(w2, 0) == ("k_factor", "k_sweep_fine")
    assert bench.finest_kernels(w2, 1) == ("k_factor_blk", "k_sweep_fine")
    assert bench.finest_kernels(small, 1) == ("k_factor_small", "k_sweep_small")
    assert bench.finest_kernels(w3, 0) == ("k_factor_wide", "k_sweep_fine")
    assert bench.finest_kernels(w3, 1) == ("k_factor_band", "k_sweep_super")
    assert bench.finest_kernels(dense, 1) == ("k_factor_wide", "k_sweep_fine")
    assert bench.finest_kernels(bench.workload("2d-square"), 0) == ("k_factor_square", "k_sweep_square")
    r = bench.finest_roofline(fake_profile(), w3, 1, ms_total=20.0, traffic_ok=False)
    assert r["kernel"] == "k_factor_band (finest level)"
    r = bench.finest_roofline(fake_profile(ms_sweep=40.0), small, 1, ms_total=60.0, traffic_ok=False)
    assert r["kernel"] == "k_sweep_small (one sweep, all colours)"
