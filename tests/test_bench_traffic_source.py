"""The bench's solver hash is that of the file the kernel it ran comes from."""
import hashlib
import os

import pytest

import bench


@pytest.mark.parametrize("kernel,unit", [("k_solve_mg", "gfm_mg.cu"), ("k_solve_mixed", "gfm_solve.cu"),
                                         ("k_solve_batched", "gfm_solve.cu")])
def test_hash_follows_the_kernel(kernel, unit):
    with open(os.path.join(bench.ROOT, "paper_1804_01130_gb300", "csrc", unit), "rb") as fh:
        assert bench._traffic_record("no such workload", kernel)[1] == hashlib.sha256(fh.read()).hexdigest()[:16]
