"""The benchmark's launch counts and operation counts follow what a step
launches: where the solve takes the curl there are eight kernels, not ten, and
the solve's operations include it; digit products are not counted on the FP64
unit."""
import bench


def test_launches_follow_the_kernel_times():
    ten = {k: (1.0, 6) for k in ("curl", "zsynth", "product", "zanalysis", "solve")}
    eight = {k: v for k, v in ten.items() if k != "curl"}
    assert bench.launches_per_step(ten, 3) == 10
    assert bench.launches_per_step(eight, 3) == 8
    assert bench.launches_per_step(dict(eight, curl=(0.0, 0)), 3) == 8


def test_costs_leave_out_digit_products():
    small = dict(N=32, K=16, M=16)
    points = 32 * 31 * 16
    alone = bench.kernel_costs(small, 0)
    fused = bench.kernel_costs(small, 0, curl_in_solve=True, split=True)
    assert alone["curl"]["flops"] == 30 * points
    assert fused["solve"]["flops"] - alone["solve"]["flops"] == 102 * points
    assert fused["solve"]["bytes"] - alone["solve"]["bytes"] == 16 * 6 * points
    assert alone["zsynth"]["flops"] == 0 and alone["product"]["flops"] == 9 * 32 * 48 * 48
    assert bench.kernel_costs(small, 1)["zsynth"]["flops"] > 0
    # per row: 150 operations beside the substitutions, 78 where the stencils are digits
    per = lambda N, split=False: bench.kernel_costs(dict(N=N, K=4, M=4), 1, split=split)["solve"]["flops"]
    assert per(64, split=True) - per(64) == 72 * 64 * 7 * 4
    assert per(63, split=True) == per(63)
