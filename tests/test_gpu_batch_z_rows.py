"""The z-in-shared-memory limit that a batched solve reports is the one it ran with.

A schedule may name a few more rows than the kernel's own shared memory leaves; the
launch takes what is left.  What is reported has to fit an SM together with the
system's 1 KB per CTA and the kernel's static part, of which its two matrix
descriptors (eight buckets of more than 64 bytes each) are more than 1,024 bytes."""
import re

import numpy as np
import pytest
import torch

from gpu_helpers import dev, lib
from paper_2307_03914_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ug,side,size", [("fp32", 126, 4), ("fp64", 90, 8)])
def test_reported_rows_fit(ug, side, size):
    B = lib()
    A, off = W.block_diagonal([W.convdiff2d(side, side)] * 3)
    Ad, Pd = B.DeviceCSR.from_host(A), B.DeviceCSR.from_host(A, with_values=False)
    Ah = B.matrix_create(Ad)
    M, _ = B.bspai_build(Ad, Pd, 0.3)
    ro = dev(off.astype(np.int32))
    BM, _ = B.bspai_bucket_batched(M, ro, 2.0 ** -16, ["fp64", "fp32"])
    b = dev(np.random.default_rng(1).uniform(-1, 1, A.n))

    def solve(z):
        B.batch_schedule_force(128, z_shared_rows=z)
        try:
            x = torch.zeros_like(b)
            return B.gmres_ir_solve_batched(Ah, ro, 1, b, BM, M, x, ug, ug, 1e-4, B.opts(kmax=6, i_max=1)), x
        finally:
            B.batch_schedule_force(None)

    with pytest.raises(B.BspaiError) as e:
        solve(1 << 24)
    most = int(re.search(r"exceeds the (\d+) rows", str(e.value)).group(1))
    assert most <= side * side  # the systems are larger: every limit below takes effect
    fit, x_fit = solve(-1)
    named, x_named = solve(most)
    assert named["z_shared_rows"] == fit["z_shared_rows"] and torch.equal(x_named, x_fit)
    assert most - 1100 * 4 // size <= fit["z_shared_rows"] <= most
    sms = torch.cuda.get_device_properties(0)
    per_cta = 14000 * 4 // size  # a quarter of an SM: the CTAs per SM that 128 threads of 128 registers allow
    assert fit["z_shared_rows"] > per_cta * 0.9
    assert fit["z_shared_rows"] * size + 1024 + 1024 <= sms.shared_memory_per_multiprocessor // 4
    assert solve(64)[0]["z_shared_rows"] == 64
