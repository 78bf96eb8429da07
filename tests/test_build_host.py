"""Kernel families of build.py (no GPU needed): what a profile's source hash
covers."""
import os

from paper_1304_5546_gb300 import build as B


def test_every_stage_kernel_source_is_in_a_family():
    names = [n for n in os.listdir(B.CSRC)
             if n.startswith("kernels") and not n.startswith("kernels_batch")]
    assert {"kernels_er.cuh", "kernels_f64.cuh", "kernels.cuh"} <= set(names)
    for n in names:
        assert any(pick(n) for pick in B.KERNEL_FAMILIES.values()), n
    hashes = {f: B.kernel_source_hash(f) for f in B.KERNEL_FAMILIES}
    assert len(set(hashes.values())) == len(hashes)
