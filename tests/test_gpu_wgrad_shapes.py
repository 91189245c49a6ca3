"""Weight gradients on the tensor cores over the operand shapes the kernel chooses between:
nine taps per CTA (narrow layers) or one kernel row, MMA rows from the output or the input
channels, column tiles of 16 to 128, channel counts that fill the 128 rows in part.  The checks
are those of test_gpu_learned.py (FP64 oracle with the same bfloat16 weights, 1e-4)."""
import pytest

from tests import test_gpu_learned as learned
from tests.test_gpu_learned import lib  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("widths,N", [((32, 32, 32), 1), ((160, 96, 224), 1), ((128, 256, 192), 2), ((64, 160, 32), 3)])
def test_wgrad_operand_shapes(lib, widths, N):  # noqa: F811
    learned.test_network_forward_and_gradients_match_the_oracle(lib, widths, N)
