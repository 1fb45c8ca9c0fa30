"""The tests that compare two kernels of one step rely on where the dispatch
changes from one to the other: a limit that moves in the code has to move there
too, or they would compare a kernel with itself."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2311_10827_gb300", "csrc")


def test_one_tile_kernel_limit_is_the_tests():
    import test_gpu_shot_kernel as t
    with open(os.path.join(CSRC, "kernels_d2q9.cu")) as fh:
        text = fh.read()
    assert int(re.search(r"SHOT_MAX_NODES = (\d+);", text).group(1)) == t.MOST
    assert re.search(r"P\.N <= SHOT_MAX_NODES", text)


@pytest.mark.gpu
def test_four_warp_kernel_limit_is_the_tests():
    """One tile per SM; test_gpu_fp64_march repeats its flows past 152 tiles."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    with open(os.path.join(CSRC, "kernels_d2q9.cu")) as fh:
        assert re.search(r"tiles\.x \* \(long long\)tiles\.y <= \(s\.num_sms > 0 \? s\.num_sms : 152\)",
                         fh.read())
    assert torch.cuda.get_device_properties(0).multi_processor_count <= 152
