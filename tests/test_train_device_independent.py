"""One seed gives one network on every device: no device property enters the training kernels' launch
shapes, whose sums would otherwise be added in another order."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1711_10855_gb300", "csrc")


def test_training_launches_depend_on_shapes_only():
    with open(os.path.join(CSRC, "fdas_train.cu")) as f:
        code = re.sub(r"//[^\n]*", "", f.read())
    assert not re.findall(r"sm_count|cudaDeviceGetAttribute|cudaGetDeviceProperties|cudaOccupancy\w+", code)
