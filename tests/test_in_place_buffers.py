"""Which caller buffers la_residual's kernel uses in place, on the host: the library's own predicate, compiled from
its header with nvcc, on pointer attributes of every kind.  Only aligned memory of the context's device
qualifies; another GPU's memory, host, managed and unregistered memory go through a copy."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.abspath(__file__)), "..", "paper_1111_4363_gb300", "csrc")

PROGRAM = r"""
#include <stdio.h>
#include "la_internal.cuh"

int main() {
  const cudaMemoryType types[4] = {cudaMemoryTypeUnregistered, cudaMemoryTypeHost, cudaMemoryTypeDevice,
                                   cudaMemoryTypeManaged};
  for (cudaMemoryType t : types)
    for (int owner = 0; owner < 3; ++owner)
      for (int device = 0; device < 3; ++device)
        for (int offset = 0; offset < 64; offset += 8) {
          cudaPointerAttributes a = {};
          a.type = t;
          a.device = owner;
          const void* p = reinterpret_cast<const void*>((uintptr_t)0x7f0000000000ull + offset);
          printf("%d %d %d %d %d\n", (int)(t == cudaMemoryTypeDevice), owner, device, offset,
                 (int)la::usable_in_place(a, device, p));
        }
  return 0;
}
"""


def test_only_aligned_memory_of_the_contexts_device(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    src, exe = tmp_path / "in_place.cu", tmp_path / "in_place"
    src.write_text(PROGRAM)
    subprocess.run([nvcc, "-O1", "-std=c++17", "-gencode", "arch=compute_103a,code=sm_103a", "-I", CSRC, str(src),
                    "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert out.returncode == 0
    rows = [tuple(int(v) for v in ln.split()) for ln in out.stdout.splitlines()]
    assert len(rows) == 4 * 3 * 3 * 8
    for is_device, owner, device, offset, got in rows:
        assert got == int(is_device and owner == device and offset % 32 == 0), (is_device, owner, device, offset)


def test_la_residual_asks_the_predicate():
    """The entry point decides by the predicate and the context's own device, not by "some device pointer"."""
    text = open(os.path.join(CSRC, "la_api.cu")).read()
    body = text[text.index('extern "C" la_status la_residual('):]
    body = body[:body.index('\nextern "C"')]
    assert "usable_in_place(a, c->device, p)" in body and "is_device_ptr(p)" not in body


@pytest.mark.gpu
@pytest.mark.parametrize("shift", [-64, -2, 2, 64])
def test_residual_over_part_of_its_coefficients(shift):
    """r written into a buffer that overlaps part of c: the same residual as into one of its own."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_1111_4363_gb300 import workloads as wl
    from tests.helpers import gpu_context, variant
    w = variant(wl.softcore_2d(n=32, levels=1), n=(23, 18, 1), nt=4, sub=(2, 2, 1), coarse_sub=None)
    psi0 = torch.from_numpy(wl.initial_state(w).ravel()).cuda()
    n = w.npoints * w.nt
    c = torch.from_numpy(wl.random_state(n, 3)).cuda()
    with gpu_context(w) as ctx:
        want = torch.empty_like(c)
        N = ctx.residual(psi0, 0.35, c, want)
        buf = torch.zeros(n + 128, dtype=torch.complex128, device="cuda")
        cin, r = buf[64:64 + n], buf[64 + shift:64 + shift + n]
        cin.copy_(c)
        assert ctx.residual(psi0, 0.35, cin, r) == N
        assert torch.equal(r, want)
