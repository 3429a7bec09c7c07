"""The hash that ties a committed profile to its kernel's sources covers every
file that decides the kernel's traffic."""
import os
import shutil

import pytest

import bench

# what a kernel's loop and its launch shape are written in
NEEDED = {
    "chain_kernel": {"wq4_chain.cu", "wq4_items.cuh", "wq4_device.cuh"},
    "stage_kernel": {"wq4_stage.cu", "wq4_tiles.cuh", "wq4_items.cuh", "wq4_tc.cuh", "wq4_device.cuh", "wq4_bgemv.cu"},
    "gemv_kernels": {"wq4_gemv.cu", "wq4_bgemv.cu", "wq4_tiles.cuh", "wq4_items.cuh", "wq4_tc.cuh", "wq4_device.cuh"},
    "paged_attn_kernel": {"wq4_attn.cu", "wq4_device.cuh"},
    "gemm_kernel": {"wq4_gemm.cu", "wq4_tc.cuh", "wq4_device.cuh"},
}


@pytest.mark.parametrize("kernel", sorted(bench.KERNEL_SOURCES))
def test_a_change_of_any_source_changes_the_hash(kernel, tmp_path, monkeypatch):
    assert NEEDED[kernel] <= set(bench.kernel_files(kernel))
    base = bench.source_sha(kernel)
    copy = tmp_path / "csrc"
    shutil.copytree(bench.CSRC, copy)
    monkeypatch.setattr(bench, "CSRC", str(copy))
    assert bench.source_sha(kernel) == base
    for f in NEEDED[kernel]:
        text = (copy / f).read_text()
        (copy / f).write_text(text + "\n// changed\n")
        assert bench.source_sha(kernel) != base, f
        (copy / f).write_text(text)
    assert bench.source_sha(kernel) == base


def test_every_profile_with_a_hash_names_a_known_kernel():
    d = os.path.join(bench.ROOT, "profiles")
    for name in os.listdir(d):
        if "source_sha:" in open(os.path.join(d, name)).read():
            assert any(name.startswith(k) for k in bench.KERNEL_SOURCES), name
