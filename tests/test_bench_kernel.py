"""The kernel and FP64-pipe count that bench.py prints belong to the run's size and options."""
import importlib


def test_step_kernel_follows_the_ensemble():
    b = importlib.import_module("bench")
    assert b.step_kernel(4096, 1) == ("k_step<8,1,1>", b.FP64_PIPE_FLOPS)
    assert b.step_kernel(4864, 1)[0] == "k_step<8,1,1>" and b.step_kernel(4865, 1)[0] == "k_step_queue<8,1>"
    assert b.step_kernel(1824, 1) == ("k_step_wide<8,1>", None) and b.step_kernel(1825, 1)[0] == "k_step<8,1,1>"
    assert b.step_kernel(4096, 0) == ("k_step<8,0,1>", None) and b.step_kernel(65536, 2)[1] is None
