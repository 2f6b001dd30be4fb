"""Checkpoint copies: which are made by a kernel (copy_route.h), and both routes' bytes.

A kernel reaches memory of its own device only, the copy engine that of another
device (and it refuses what is no device memory), so the kernel is for buffers on
the handle's device: shown by the rule itself, compiled for the host, since no
second device is used here. On the GPU: a state below and one above the size
up to which the kernel copies, saved, overwritten by steps and loaded again.
"""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2306_07603_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include "copy_route.h"
using namespace ifd;
static bool route(std::uintptr_t at, std::int64_t bytes, bool here) {
  void *p = reinterpret_cast<void *>(at);
  return copy_by_kernel({{p, p, p}, {p, p, p}, {bytes, bytes, 8}}, here);
}
int main() {
  const std::int64_t half = COPY_MOST / 2;
  std::printf("%d%d%d%d%d%d%d\n", route(4096, 1024, true), route(4096, 1024, false),
              route(4096, half - 8, true), route(4096, half - 8, false), route(4096, half, true),
              route(4104, 1024, true), route(4096, 1028, true));
}
"""


def test_a_kernel_copies_only_memory_of_its_device(tmp_path):
    if shutil.which("g++") is None:
        pytest.skip("no host compiler")
    (tmp_path / "route.cpp").write_text(PROGRAM)
    exe = str(tmp_path / "route")
    subprocess.run(["g++", "-std=c++17", "-I", CSRC, "-o", exe, str(tmp_path / "route.cpp")],
                   check=True)
    assert subprocess.check_output([exe], text=True).strip() == "1010000"


@pytest.mark.gpu
@pytest.mark.parametrize("nx,ny,kernels", [(65, 47, 1), (1025, 900, 0)])
def test_saved_state_comes_back(nx, ny, kernels):
    import torch

    from paper_2306_07603_gb300 import capi
    from paper_2306_07603_gb300.solver import Solver, cavity
    s = Solver([cavity(nx, ny, 400.0, 0.75, theta_deg=60.0)])
    s.step(2)
    words = capi.ifdlbm_state_bytes(s.h) // 8
    assert (words * 8 <= 64 << 20) == bool(kernels)
    first, again = (torch.zeros(words, dtype=torch.float64, device="cuda") for _ in range(2))
    torch.cuda.synchronize()
    before = capi.ifdlbm_launch_count()
    capi.ifdlbm_save_state_dev(s.h, first)
    assert capi.ifdlbm_launch_count() - before == kernels
    want = s.get_state(0)[0]
    s.step(3)
    capi.ifdlbm_load_state_dev(s.h, first)
    capi.ifdlbm_save_state_dev(s.h, again)
    got = s.get_state(0)[0]
    s.close()
    assert torch.equal(first, again) and (got == want).all()


@pytest.mark.gpu
def test_copies_can_be_captured():
    """Looking the buffer's device up is no stream operation: a capture records the copies."""
    import torch

    from paper_2306_07603_gb300 import capi
    from paper_2306_07603_gb300.solver import Solver, cavity
    s = Solver([cavity(65, 47, 400.0, 0.75)])
    a, b = (torch.zeros(capi.ifdlbm_state_bytes(s.h) // 8, dtype=torch.float64, device="cuda")
            for _ in range(2))
    s.step(2)
    capi.ifdlbm_save_state_dev(s.h, a)
    s.sync()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=s.stream):
        capi.ifdlbm_load_state_dev(s.h, a)
        capi.ifdlbm_save_state_dev(s.h, b)
    assert not torch.equal(a, b)
    with torch.cuda.stream(s.stream):
        graph.replay()
    s.sync()
    s.close()
    assert torch.equal(a, b)
