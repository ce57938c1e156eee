"""The adjoint of a single sweep (its own kernel) at the edges of its blocks,
against the FP64 adjoint under the bar of the other sizes."""
import pytest

import test_gpu_adjoint_blocks as blocks
from test_gpu_adjoint_blocks import dev  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(1, 1, 1), (2, 65, 257), (3, 2, 256), (300, 16, 16)])
def test_single_sweep_matches_oracle(dev, shape):  # noqa: F811
    blocks.test_blocks_match_oracle(dev, shape, 1)
