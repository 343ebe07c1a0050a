"""Kernels launched with programmatic stream serialisation begin before their predecessor has finished.

- On the CPU, from the sources: a kernel (or device function) that waits for its predecessor inside
  (overlap_wait) declares no pointer to what a predecessor writes __restrict__, and reads none by __ldg; only the
  factors, the stencils and the time matrices, which are final before a chain of such launches begins, may be.
- On the GPU: a propagation by la_step (overlapped launches, directly and as a captured graph) and the same one by
  la_step_batch (plain launches in a conditional graph body) give the same bits, for odd K and for every kernel
  of the chain, repeatedly."""
import dataclasses
import glob
import os
import re

import numpy as np
import pytest

from paper_1111_4363_gb300 import workloads as wl

CSRC = os.path.join(os.path.dirname(os.path.abspath(__file__)), "..", "paper_1111_4363_gb300", "csrc")
FINAL = {"factors", "sigma", "tm"}


def functions(text):
    """(name, parameter list, body) of the kernels and device functions of a source file."""
    for m in re.finditer(r"(?:__global__|__device__)[^;{}]*?\b(\w+)\s*\(((?:[^()]|\([^()]*\))*)\)\s*(?:const\s*)?\{", text):
        depth, i = 1, m.end()
        while depth:
            depth += {"{": 1, "}": -1}.get(text[i], 0)
            i += 1
        name = m.group(1)
        if name == "__launch_bounds__":
            continue
        yield name, m.group(2), text[m.end():i]


def test_pointers_of_overlapped_kernels_promise_nothing():
    text = "\n".join(re.sub(r"//[^\n]*", "", open(f).read())
                     for f in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))))
    text = re.sub(r"__launch_bounds__\((?:[^()]|\([^()]*\))*\)", "", text)
    fns = list(functions(text))
    waits = {n for n, _, b in fns if "overlap_wait()" in b and n != "overlap_wait"}
    waits |= {n for n, _, b in fns if any(re.search(rf"\b{w}\b\s*[<(]", b) for w in waits)}
    for expected in ("k_restrict_tile", "k_prolong_add", "k_sweep_fine", "k_sweep_super", "k_sweep_small", "sweep_rhs",
                     "k_sweep_coarse", "k_gresid_tiles", "coarse_rhs"):
        assert expected in waits
    # every kernel that is launched overlapped waits
    launched = set(re.findall(r"launch_overlapped\([^;]*?\b(k_\w+)", text))
    launched |= set(re.findall(r"auto kern = (k_(?:sweep|gresid)\w+)", text)) - {"k_sweep_square"}
    assert launched and launched <= waits
    for name, params, body in fns:
        if name not in waits:
            continue
        bad = [p for p in re.findall(r"__restrict__\s+(\w+)", params) if p not in FINAL]
        assert not bad, (name, bad)
        assert not re.search(r"__ldg\(\s*(?:f|yx|c|ev|ec|ef|gvec|sf)\b", body), name


def grid(dim, n, sub, K, levels):
    base = {1: wl.harmonic_1d, 2: wl.softcore_2d, 3: wl.hydrogen_3d}[dim]()
    return dataclasses.replace(base, n=n, sub=sub, nt=K, levels=levels, coarse_nu=None, psi_kind="gaussian", seed=4,
                               coarse_sub=tuple(2 if a < dim else 1 for a in range(3)) if levels > 1 else None,
                               nu1=1, nu2=1, coarse_sweeps=1, trial=3, tol=1e-10, max_cycles=60)


GRIDS = [grid(2, (40, 28, 1), (4, 4, 1), 3, 3),      # k_sweep_fine (48 unknowns), k_sweep_coarse
         grid(2, (28, 20, 1), (4, 2, 1), 3, 3),      # k_sweep_small
         grid(3, (12, 16, 8), (4, 4, 4), 3, 3),      # k_sweep_super (192 unknowns)
         grid(3, (8, 12, 8), (2, 2, 2), 5, 2),
         grid(1, (96, 1, 1), (8, 1, 1), 7, 3)]


@pytest.mark.gpu
@pytest.mark.parametrize("w", GRIDS, ids=lambda w: f"{w.dim}d_{w.n}_K{w.nt}_L{w.levels}")
def test_overlapped_steps_equal_plain_ones(w):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_1111_4363_gb300 import binding as B
    from tests.helpers import gpu_context
    psi0 = torch.from_numpy(wl.initial_state(w).ravel()).cuda()
    with gpu_context(w, precision=1) as plain:
        want = psi0.clone()
        B.step_batch([plain], [want], 3, [0.0])
    for _ in range(8):
        with gpu_context(w, precision=1) as ctx:
            psi = psi0.clone()
            ctx.step(psi, 3, 0.0)
            assert torch.equal(torch.view_as_real(psi), torch.view_as_real(want))
    assert np.isfinite(want.cpu().numpy()).all()
