"""Which segment heights the split variants report: the one-warp walk's depend on the
lattices, so that its variant has none to report and says so; the benchmark names its
kernel and its line of the profile by that."""
import pytest

import bench


@pytest.fixture(scope="module")
def hlb():
    from paper_1812_10375_gb300 import build
    build.build()
    from paper_1812_10375_gb300 import hlb
    return hlb


def test_segment_rows_of_the_variants(hlb):
    rows, kinds = hlb.variant_energy_rows(), hlb.variant_kinds()
    split = [r for r, k in zip(rows, kinds) if k == bench.KIND_SPLIT]
    assert split == [hlb.HLB_ROWS_BY_SIZE, 64, 64, 96, 96, 0]
    assert all(r == -1 for r, k in zip(rows, kinds) if k != bench.KIND_SPLIT)
    assert bench.ROWS_BY_SIZE == hlb.HLB_ROWS_BY_SIZE not in (-1, 0) and hlb.HLB_ROWS_BY_SIZE < 0


def test_benchmark_names_the_kernel(hlb):
    names = [bench.kernel_name((64, 24, 256), bench.KIND_SPLIT, r) for r in hlb.variant_energy_rows()[:6]]
    assert names == ["k_flow_batch+" + k for k in ["k_energy_pair_batch"] + ["k_energy_walk_batch"] * 4
                     + ["k_energy_batch"]]
    assert bench.variant_key((64, 24, 256), bench.KIND_SPLIT, hlb.HLB_ROWS_BY_SIZE) == "64x24x256_pair"
