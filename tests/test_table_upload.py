"""Table uploads are complete before they count as done."""
import os
import subprocess
import sys

import pytest

from paper_1405_2255_gb300 import build

CSRC = os.path.join(os.path.dirname(os.path.abspath(build.__file__)), "csrc")

HOST = r"""
#include <cuda_runtime.h>
static int calls = 0, synced_at = 0, init_at = 0;
static unsigned long long* done_word = nullptr;
static unsigned long long done_at_sync = ~0ull;
static cudaError_t fake_sync(cudaStream_t) { synced_at = ++calls; done_at_sync = *done_word; return cudaSuccess; }
static cudaError_t fake_device(int* d) { *d = 3; return cudaSuccess; }
#define cudaStreamSynchronize fake_sync
#define cudaGetDevice fake_device
#include "common.cuh"
int main() {
    gb3::DeviceOnce o;
    done_word = &o.done;
    int runs = 0;
    for (int k = 0; k < 2; ++k) gb3::once_per_device(o, [&] { ++runs; init_at = ++calls; });
    if (runs != 1 || init_at != 1) return 1;      // once
    if (synced_at != 2) return 2;                 // the copies are waited for
    if (done_at_sync != 0 || o.done != 8) return 3;  // before the device counts as done
    return 0;
}
"""


def test_upload_waits_before_done(tmp_path):
    """once_per_device with the runtime's calls replaced by host functions (no GPU)."""
    src, exe = tmp_path / "once.cu", tmp_path / "once"
    src.write_text(HOST)
    subprocess.run([build.nvcc(), "-std=c++17", "-I", CSRC, "-o", str(exe), str(src)], check=True, capture_output=True)
    assert subprocess.run([str(exe)]).returncode == 0


FIRST = r"""
import numpy as np, torch
from paper_1405_2255_gb300 import gb3fmm as g, inputs
x, mu = (torch.from_numpy(a).to("cuda:0") for a in inputs.plummer(3000, 3))
s = torch.cuda.Stream()
torch.cuda.synchronize()
with torch.cuda.stream(s):
    for prm in (dict(precision=0, p=14), dict(precision=1, p=14), dict(precision=1, p=12, m2l_rot=0)):
        c = g.Context(eps=1e-4, leaf_size=16, p2p_c=0.0, **prm)
        a, b = (c.fmm_evaluate_active(x, mu, tidal=True) for _ in range(2))
        s.synchronize()
        assert all(torch.equal(u, v) for u, v in zip(a, b)), prm
        c.close()
"""


@pytest.mark.gpu
def test_first_evaluation_of_a_process():
    """The first call, which uploads the tables, gives the bits of the second."""
    root = os.path.dirname(os.path.dirname(CSRC))
    subprocess.run([sys.executable, "-c", FIRST], check=True, cwd=root, timeout=300)
