"""The network's kernels at the edges of their tiles: the forward pass's blocks of 64 samples, the
backward pass's tiles of 32 rows and its steps of 32 samples dealt to two groups, one
sample; through the checks of test_gpu_mlp against the oracle
and their tolerances."""
import pytest

import test_gpu_mlp as net
from test_gpu_mlp import B  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 15, 16, 17, 63, 64, 65, 129])
def test_forward_at_the_edges_of_its_blocks(B, n):  # noqa: F811
    net.test_forward_matches_oracle(B, n)


@pytest.mark.parametrize("n", [1, 31, 32, 33, 63, 64, 65, 97, 2049])
def test_gradient_at_the_edges_of_its_tiles(B, n):  # noqa: F811
    net.test_gradient_matches_oracle(B, n)
