"""Which pass kernel the bench names comes from lowd_info, and the field that tells the wavefronts from
the one-CTA sweeps sits where the struct had padding: the other fields keep their places."""
import bench
from paper_2307_15969_gb300 import lowd


def test_info_layout():
    f = lowd.lowd_info
    assert f.stars.offset == 72 and f.wavefront_blocks.offset == 76
    assert f.star_edges.offset == 80 and __import__("ctypes").sizeof(f) == 88


def test_bench_names_the_kernel_that_ran():
    assert bench._pass_kernel({"wavefront_blocks": 72, "sweep_kernel": 1}) == "k_sweep_systolic"
    assert bench._pass_kernel({"wavefront_blocks": 2, "sweep_kernel": 2}) == "k_sweep_systolic"
    assert bench._pass_kernel({"wavefront_blocks": 0, "sweep_kernel": 1}) == "k_sweep_tma"
    assert bench._pass_kernel({"wavefront_blocks": 0, "sweep_kernel": 5}) == "k_sweep_flow"
    assert bench._sweep_record("k_sweep_flow") is None and bench._traffic_per_pass("k_sweep_vec") is None
