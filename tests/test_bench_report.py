"""The benchmark's report counts one launch's tensor-core work alike wherever it states it."""
import bench


def test_tensor_ceiling_of_the_step_is_the_sum_of_its_kernels():
    stats = [{"launches": 40, "tensor_flops": 40 * 7.5e10}, {"launches": 20},
             {"launches": 20, "tensor_flops": 20 * 3.0e10}, {"launches": 20, "tensor_flops": 0}]
    for peaks in ({"bf16_tflops_sustained": 1718.4}, {}):
        rows = [bench.tensor_roofline(s, 0.1, peaks) for s in stats]
        assert rows[1] is None and rows[3] is None
        step = 2 * rows[0]["t_ceil_ms"] + rows[2]["t_ceil_ms"]  # 20 steps
        assert abs(bench.tensor_ceil_ms(stats, 20, peaks) / step - 1) < 1e-12
