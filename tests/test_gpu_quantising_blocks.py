"""The quantising gather by one block an SM and by two (quant.cu: two where three rows of A fit in half of the shared memory)."""
import pytest

from test_gpu_quantising_gather import test_codes_and_steps_match_the_definition as check

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,K,k", [
    (296, 4096, 2052), (297, 4096, 4096), (593, 4100, 4097),      # a row a block, two, three; one and two groups of 2048 outputs, a third
    (600, 18416, 2100), (300, 18416, 16384), (40, 18416, 16385),  # the longest rows of two blocks; all eight groups; one output more
    (300, 18417, 16384), (300, 18432, 9000),                      # one block
    (1, 18416, 8193), (900, 9000, 6145),
])
def test_one_and_two_blocks(oracle, M, K, k):
    check(oracle, M, K, k)
