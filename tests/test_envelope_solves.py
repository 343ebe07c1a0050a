"""Two-warp triangular solves inside the envelope and over whole rows: the library's rule between them on the host, and
both on the GPU, FP64 passes of many subvolumes against exact local minimisations from the oracle's system (1e-11), and
mixed V-cycles with coarse subvolumes of 33 to 128 unknowns, which must converge to the direct solution."""
import dataclasses
import os
import shutil
import subprocess

import numpy as np
import pytest

from oracle import system
from paper_1111_4363_gb300 import workloads as wl
from tests.helpers import gpu_context, oracle_system, rel_l2

CSRC = os.path.join(os.path.dirname(os.path.abspath(__file__)), "..", "paper_1111_4363_gb300", "csrc")

PROGRAM = r"""
#include <stdio.h>
#include "la_internal.cuh"
int main() {
  for (int npts = 1; npts <= 32; ++npts)
    for (int reach = 0; reach < npts; ++reach)
      for (int nb = 1; nb <= 8; ++nb)
        for (unsigned ctas = 1; ctas < 2000; ctas += 455)
          for (int fp64 = 0; fp64 < 2; ++fp64)
            printf("%d %d %d %u %d %d\n", npts, reach, nb, ctas, fp64,
                   (int)la::solve_inside_envelope(reach, npts, nb, ctas, fp64 != 0));
  return 0;
}
"""


def test_rule_on_the_host(tmp_path):
    """No bounds where they leave nothing out, never fewer with a shorter reach, and the measured points of the rule."""
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    src, exe = tmp_path / "rule.cu", tmp_path / "rule"
    src.write_text(PROGRAM)
    subprocess.run([nvcc, "-O1", "-std=c++17", "-gencode", "arch=compute_103a,code=sm_103a", "-I", CSRC, str(src),
                    "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    table = {tuple(int(v) for v in ln.split()[:5]): int(ln.split()[5]) for ln in out.stdout.splitlines()}
    for (npts, reach, nb, ctas, fp64), inside in table.items():
        if inside:
            assert nb > 1 and (npts == 1 or reach < npts - 1)
            assert reach == 0 or table[(npts, reach - 1, nb, ctas, fp64)]
    few, many = 1, 456 + 455
    assert table[(16, 8, 6, many, 1)] and table[(16, 8, 6, few, 1)] and not table[(16, 8, 2, few, 1)]
    assert not table[(8, 6, 2, many, 1)] and not table[(16, 12, 8, many, 1)]
    assert table[(16, 2, 8, few, 0)] and not table[(16, 10, 6, many, 0)] and not table[(8, 7, 4, few, 0)]


@pytest.mark.gpu
@pytest.mark.parametrize("sub,K,blocks", [((4, 4, 1), 6, (46, 46)), ((4, 4, 1), 6, (6, 6)), ((4, 2, 1), 4, (44, 48)),
                                          ((3, 3, 1), 2, (50, 44)), ((5, 5, 1), 3, (6, 6))], ids=str)
def test_fp64_passes(sub, K, blocks):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    n = (sub[0] * blocks[0] - 1, sub[1] * blocks[1] - 1, 1)   # ragged last subvolumes
    w = dataclasses.replace(wl.softcore_2d(n=16, levels=1), n=n, sub=sub, nt=K, coarse_sub=None, coarse_nu=None,
                            psi_kind="gaussian", seed=5)
    psi0 = wl.initial_state(w).ravel()
    prob, M, f, W = oracle_system(w, psi0, 0.35)
    c0 = wl.random_state(M.shape[1], 3)
    grad = M.conj().T @ (W @ (f - M @ c0))
    got = c0.copy()
    with gpu_context(w) as ctx:
        ctx.relax_colour(psi0, 0.35, 3, got)
    Mc, Wr = M.tocsc(), W.tocsr()
    last = tuple(b - 1 if b % 2 == 0 else b - 2 for b in blocks)
    for bx, by in ((1, 1), (last[0], 1), (1, last[1]), last, (3, 5)):
        pts = [y * n[0] + x for y in range(by * sub[1], min((by + 1) * sub[1], n[1]))
               for x in range(bx * sub[0], min((bx + 1) * sub[0], n[0]))]
        idx = (np.array(pts)[:, None] * K + np.arange(K)).ravel()
        MU = Mc[:, idx]
        want = c0[idx] + np.linalg.solve((MU.conj().T @ Wr @ MU).toarray(), grad[idx])
        assert rel_l2(got[idx], want) < 1e-11, (bx, by)


@pytest.mark.gpu
@pytest.mark.parametrize("dim,n,csub,K", [(2, (32, 24, 1), (4, 4, 1), 4), (2, (24, 32, 1), (4, 4, 1), 7),
                                          (1, (96, 1, 1), (16, 1, 1), 8), (1, (64, 1, 1), (8, 1, 1), 6),
                                          (3, (8, 8, 8), (2, 2, 2), 6)])
def test_mixed_coarse_sweeps(dim, n, csub, K):
    """Refined to N/N(0) <= 1e-22 the coefficients equal the direct solution to 1e-9, in as many cycles as FP64 takes
    (one more allowed for the rounding of the last one)."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    base = {1: wl.harmonic_1d, 2: wl.softcore_2d, 3: wl.hydrogen_3d}[dim]()
    w = dataclasses.replace(base, n=n, sub=tuple(4 if a < dim else 1 for a in range(3)) if dim < 3 else (2, 2, 2), nt=K,
                            levels=2, coarse_sub=csub, coarse_nu=None, nu1=1, nu2=1, coarse_sweeps=2,
                            psi_kind="gaussian", seed=2)
    psi0 = wl.initial_state(w).ravel()
    prob, M, f, W = oracle_system(w, psi0, 0.0)
    cd = system.direct_solve(M, f)
    cycles = []
    for precision in (0, 1):
        with gpu_context(w, precision=precision, tol=1e-22, max_cycles=120) as ctx:
            c = np.zeros(M.shape[1], dtype=np.complex128)
            _, (cyc, _, _, rel) = ctx.solve_step(psi0, 0.0, c)
            assert rel <= 1e-22 and rel_l2(c, cd) < 1e-9
            cycles.append(cyc)
    assert cycles[1] <= cycles[0] + 1
