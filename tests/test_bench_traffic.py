"""The DRAM traffic that bench.py reports for the projections of a 7B step comes from a committed capture: it has to be of kernels that
read their weights once and nothing for others."""
import bench
from workloads import WORKLOADS


def test_traffic_per_launch_is_that_of_the_weights():
    shape = WORKLOADS["C3"].shape
    weights = 2 * shape.streamed_params / (4 * shape.n_layers + 1)
    # beside the weights: operand images and residual rows (0.3 MB a launch), and the LM head's logits (1 MB of 262)
    assert weights <= bench.gemm_traffic_per_launch(WORKLOADS["C3"]) <= 1.03 * weights
