"""The down-converter's remainder blocks of 4 and of 8 and 4 taps (filters of 4
and 12 taps per plane, alone and behind a block of 16) against the FP64 oracle."""
import pytest

from tests.test_gpu_ddc_blocks import test_every_block_and_remainder as _check
from tests.test_gpu_narrowband import _cuda  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("D,Th,L", [(32, 2, 64 * 129), (4, 2, 16 * 77), (16, 6, 32 * 131), (2, 10, 16 * 201),
                                    (8, 14, 1 << 14)])
def test_remainders(D, Th, L):
    _check(D, Th, L)
