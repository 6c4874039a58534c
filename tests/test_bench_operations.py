"""The bench's operation count of the Jacobian action against the executed FP64 instructions.

Reference: additions, products and multiply-adds of all threads per element, counted by the profiler's
instruction counters for the face and the volume pass at 16^3. The count leaves out what a compiler adds
or shares (a few per thread and phase); 3 % covers it.
"""
import pytest

import bench


@pytest.mark.parametrize("k,face,vol", [(2, 2700, 1537), (3, 5670, 4373), (4, 9777, 9059)])
def test_count_matches_executed_instructions(k, face, vol):
    f, v = bench.jv_flops(k)
    assert abs(f / 2 / face - 1) < 0.03
    assert abs(v / 2 / vol - 1) < 0.03
