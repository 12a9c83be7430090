"""The bench line reports DRAM traffic only for the launch that was captured:
the record is dropped when the kernel, its launch, the cut of its items or the
constants of the cut change, and comments do not matter."""
import pytest

import bench

NNZ = bench.SPMV_TRAFFIC["near_nnz"]
KERNELS = {"k_near_spmv": {"total_ms": 64.9, "launches": 1020, "avg_us": 63.6}}


def _reported():
    return bench.roofline(KERNELS, {"near_nnz": NNZ}, 20480, {"hbm_gbs": 6805.5}, "measured")["traffic"]


def test_traffic_of_the_present_launch():
    assert _reported() == bench.SPMV_TRAFFIC["items_bytes"]
    # captured bytes lie just above the algorithmic ones
    assert 1.0 < _reported() / (8 * NNZ + 16 * 20480) < 1.02


@pytest.mark.parametrize("name,old,new,kept", [
    ("bem_capi.cu", "row_ptr[M.n] > 2500 * M.n ? 8 : 4", "row_ptr[M.n] > 2500 * M.n ? 8 : 6", False),
    ("bem_capi.cu", "kSpmvMinEntries = 4096", "kSpmvMinEntries = 8192", False),
    ("bem_capi.cu", "kSpmvItemEntries = 65536", "kSpmvItemEntries = 32768", False),
    ("bem_kernels.cuh", "kSpmvThreads = 128", "kSpmvThreads = 256", False),
    ("bem_capi.cu", "// One right-hand side:", "// For one right-hand side:", True),
])
def test_a_changed_cut_drops_the_record(monkeypatch, name, old, new, kept):
    read = bench._csrc
    assert read(name).count(old) == 1
    monkeypatch.setattr(bench, "_csrc", lambda f: read(f).replace(old, new) if f == name else read(f))
    assert _reported() == (bench.SPMV_TRAFFIC["items_bytes"] if kept else None)
