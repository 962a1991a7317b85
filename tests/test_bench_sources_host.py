"""Which sources a recorded DRAM figure depends on: the kernel's file and every header beside
it that it is built from."""

import pytest

pytest.importorskip("torch")

import bench  # noqa: E402


@pytest.mark.parametrize("kernel, want", [
    ("k_step", {"kernels.cu", "internal.hpp", "launch.cuh", "philox.cuh"}),
    ("k_deliver_slices", {"slices.cu", "internal.hpp", "philox.cuh", "stream.cuh"}),
    ("k_deliver_blocked_8", {"blocked.cu", "internal.hpp", "launch.cuh", "philox.cuh", "stream.cuh"}),
    ("k_resident", {"resident.cu", "internal.hpp", "philox.cuh", "stream.cuh"}),
    ("k_deliver_regions", {"resident.cu", "internal.hpp", "philox.cuh", "stream.cuh"}),
])
def test_every_included_header_counts(kernel, want):
    assert set(bench._kernel_sources(kernel)) == want


def test_kernels_without_a_record():
    assert bench._kernel_sources("k_update") is None and bench._recorded_traffic("k_update") is None
