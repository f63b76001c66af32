"""The scratch of afqmc_apply_flips is kept between calls and bounded: device memory in use, in a process of its
own (the pool lives as long as the process)."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

pytest.importorskip("paper_2506_09611_gb300.afqmc")

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = r"""
import torch
from paper_2506_09611_gb300 import afqmc

MB = 1 << 20


def used():
    torch.cuda.synchronize()
    free, total = torch.cuda.mem_get_info()
    return total - free


G = (torch.eye(4096, device="cuda") * 0.5).repeat(2, 1, 1)
small = (torch.eye(64, device="cuda") * 0.5).repeat(2, 1, 1)
sites = torch.arange(128, dtype=torch.int32, device="cuda")
delta = torch.full((256,), 1e-3, dtype=torch.float64, device="cuda")
st, side = torch.cuda.current_stream(), torch.cuda.Stream()  # (torch's streams take device memory: before u0)


def run(fn, A, m, stream=st):
    N = A.shape[1]
    fn("fp32", N, N, A[0].data_ptr(), A[1].data_ptr(), sites.data_ptr(), delta.data_ptr(), m, stream)


for m in (1, 33, 65):  # every kernel loaded
    run(afqmc.afqmc_apply_flips_noalloc, small, min(m, 64))
    run(afqmc.afqmc_apply_flips_noalloc, G, m)
u0 = used()
run(afqmc.afqmc_apply_flips, small, 4)
u1 = used()
assert u1 - u0 >= 16 * MB, (u0, u1)  # kept: the next call maps nothing
for _ in range(3):
    run(afqmc.afqmc_apply_flips, small, 4)
    assert used() == u1
run(afqmc.afqmc_apply_flips, G, 128, side)
run(afqmc.afqmc_apply_flips, G, 128)
assert used() - u0 <= 40 * MB, (u0, used())  # bounded: one 32 MB block and change
print("ok")
"""


def test_scratch_is_kept_and_bounded():
    r = subprocess.run([sys.executable, "-c", CHILD], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and r.stdout.strip().endswith("ok"), r.stdout + r.stderr
