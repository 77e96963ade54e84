"""The split mode's roofline counts as digit products only the GEMM flops that ran on the tensor cores, and a
batch is not labelled with a pipeline that its large Swaps may not take."""

import bench
from test_bench_line import args, fake_report, line_for

BIG, SMALL = [(1024, 1024, 512, 9, 0, 0, 0)] * 3, [(128, 64, 64, 7, 0, 0, 0)] * 5


def tensor_kernel(reps, **over):
    roof = line_for(reps, 35.0, prec="bf16_split", **over)["roofline"]
    return [k for k in [roof] + roof["other_kernels"] if k["kernel"].startswith("oz_gemm_kernel")][0]


def test_only_the_flops_on_the_tensor_cores_count():
    full = 9.0e12 * 36 / 9.0 / 1e12
    assert abs(tensor_kernel([fake_report(svd_trace=BIG)])["achieved"] - full) <= 1e-9 * full
    small = tensor_kernel([fake_report(svd_trace=SMALL)])
    assert small["achieved"] == 0.0 and small["tensor_core_flop_share"] == 0.0
    both = tensor_kernel([fake_report(svd_trace=BIG + SMALL)])
    assert 0.99 < both["tensor_core_flop_share"] < 1.0
    assert abs(both["achieved"] - both["tensor_core_flop_share"] * full) <= 1e-9 * full
    # every GEMM is on the tensor cores with split_digits set; nothing is known without a trace
    assert tensor_kernel([fake_report(svd_trace=SMALL)], split_digits=8)["tensor_core_flop_share"] == 1.0
    assert tensor_kernel([fake_report()])["tensor_core_flop_share"] == 1.0


def test_a_batch_is_not_labelled_preconditioned_alone():
    one, many = (bench.config(args(batch=b))["svd"] for b in (1, 8))
    assert "float32 passes" not in one and "3 float32 passes" in many
