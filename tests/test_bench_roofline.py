"""The bench's roofline names the kernel that runs at a size and counts what it executes."""
import pytest

import bench


@pytest.mark.parametrize("n,tensor,kernel,executed_over_flops", [
    (256, True, "k_pass_tc", 3.0), (64, True, "k_pass_tc", 3.0), (96, True, "k_pass_tc", 3.0 * 64 / 48), (32, True, "k_pass_tc", 6.0),
    (100, True, "k_digit_pass<float>", 4.0 * 64 * 64 / (50 * 50)), (250, True, "k_digit_pass<float>", 4.0 * 128 * 128 / (125 * 125)),
    (48, False, "k_half", 1.0), (33, False, "k_half", 1.0)])
def test_pass_work(n, tensor, kernel, executed_over_flops):
    name, flops, executed = bench.pass_work(n, tensor)
    assert name.startswith(kernel)
    h = (n + 1) // 2
    assert flops == 2.0 * n * n * (h * h + h * h)  # multiply-adds of both halves of every row
    assert flops <= 1.1 * float(n) ** 4            # half of a dense pass' 2 n^4
    assert executed == pytest.approx(executed_over_flops * flops)
