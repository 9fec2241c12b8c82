"""Which outputs pm_instance_tables writes by a kernel (csrc/pm_reach.h): the rule compiled on the host, with pointer
attributes made up for it (no GPU), and on a GPU the outputs that it sends the other way."""
import os
import subprocess

import numpy as np
import pytest

import oracle

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include <cstdio>
#include <initializer_list>
#include "pm_reach.h"
int main()
{
    const cudaMemoryType types[] = {cudaMemoryTypeUnregistered, cudaMemoryTypeHost, cudaMemoryTypeDevice,
                                    cudaMemoryTypeManaged};
    for (cudaMemoryType t : types)
        for (int device : {0, 1})
            for (uintptr_t at : {0x1000, 0x1001, 0x1002}) {
                cudaPointerAttributes a{};
                a.type = t;
                a.device = device;
                std::printf("%d", pm_kernel_may_store(a, reinterpret_cast<void *>(at), 1) ? 1 : 0);
            }
    std::printf("\n");
}
"""


def test_rule_on_the_host(tmp_path):
    src, exe = tmp_path / "reach.cpp", tmp_path / "reach"
    src.write_text(PROGRAM)
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    subprocess.run(["g++", "-std=c++17", f"-I{cuda}/include", f"-I{ROOT}/paper_1610_10061_gb300/csrc", str(src), "-o",
                    str(exe)], check=True, capture_output=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.strip()
    # neither pageable nor pinned host memory, device memory of device 1 only, managed memory; even addresses
    assert out == "000000" + "000000" + "000101" + "101101"


@pytest.mark.gpu
@pytest.mark.parametrize("cumulative", [False, True])
def test_outputs_at_odd_addresses_and_in_host_memory(cumulative):
    torch = pytest.importorskip("torch")
    from paper_1610_10061_gb300 import build
    build.build()
    from paper_1610_10061_gb300 import pm
    n, m, p = 37, 70, 4
    d = np.random.default_rng(3).integers(0, 5000, size=(n, m)).astype(np.int32)
    pi, delta = oracle.tables(d, p)
    L = m - p + 1
    inst = pm.Instance(d, p, cumulative=cumulative)
    raw = [torch.zeros(n * L * size + 16, dtype=torch.uint8, device="cuda") for size in (2, 4)]
    for at in (0, 1, 2, 3):
        pm.pm_instance_tables(inst.handle, raw[0][at:], raw[1][at:])
        got = [r.cpu().numpy()[at:] for r in raw]
        np.testing.assert_array_equal(got[0][:n * L * 2].copy().view(np.uint16).reshape(n, L), pi)
        np.testing.assert_array_equal(got[1][:n * L * 4].copy().view(np.int32).reshape(n, L), delta)
    host = [torch.zeros(n, L, dtype=t).pin_memory() for t in (torch.int16, torch.int32)]
    pm.pm_instance_tables(inst.handle, host[0], host[1])
    np.testing.assert_array_equal(host[0].numpy().view(np.uint16), pi)
    np.testing.assert_array_equal(host[1].numpy(), delta)
    inst.close()
