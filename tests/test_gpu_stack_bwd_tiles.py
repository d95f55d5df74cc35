"""The scorer stack's tensor-core backward at the edges of its 96-row tiles, and blocks of several tiles (two buffers of input rows take
turns) with an odd and an even number of them, with and without the gradient of the inputs."""
import pytest

from tests.test_gpu_scores_stack import test_stack_backward as check

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T,in_grad,B,H", [(13, True, 1, 2), (96, True, 1, 2), (97, False, 2, 1), (192, True, 2, 80), (193, False, 2, 80), (385, False, 4, 40)])
def test_tiles(T, in_grad, B, H):
    check("bf16", T, 9, 6, True, in_grad, B, H, 64)
