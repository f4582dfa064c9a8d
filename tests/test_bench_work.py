"""The benchmark's FP64-pipe work of a slice: what the kernels leave to that pipe, not the method's FMAs."""
from types import SimpleNamespace

import bench


def _wl(n):
    return SimpleNamespace(N=n * n, Lx=n, L=10)


def test_folded_lines():
    assert bench.folded_line(12) == (38, 40) and bench.folded_line(16) == (66, 56)  # as counted beside the transforms
    for n in range(3, 33):
        fma, add = bench.folded_line(n)
        # two halves of about n / 2 values squared, or four of about n / 4
        assert abs(fma - n * n / (4.0 if n % 2 == 0 and n >= 4 else 2.0)) <= n and add <= 4 * n


def test_slices_on_the_tensor_instruction_count_no_fp64_flops():
    assert bench.slice_pipe_flops(_wl(12)) == 0.0 and bench.slice_pipe_flops(_wl(16)) == 0.0
    assert bench.slice_pipe_flops(_wl(12), dense=True) == 2.0 * 144 ** 3
    for n in (6, 8, 18, 24):
        method = 2.0 * float(n * n) ** 2 * 2 * n
        assert 0.2 * method < bench.slice_pipe_flops(_wl(n)) < 0.8 * method
