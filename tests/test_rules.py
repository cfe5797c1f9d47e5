"""Launch rules (csrc/rules.h) on the host."""
import pytest

from tests import rules_lib

# words that fit a 284 208 MiB device beside nothing else
MOST_WORDS = 284208 * (1 << 20) // 8


@pytest.mark.parametrize("k", [1, 16, 17, 784, 6272, (1 << 31) + 5, (1 << 34) - 1, 1 << 34, (1 << 34) + 1, 1 << 35,
                               MOST_WORDS])
@pytest.mark.parametrize("tiles", [1, 3, 100, 457, 100000])
def test_ring_parts_cover_every_reduction_that_fits_the_device(k, tiles):
    """Every reduction whose operand fits the device is taken, in launches of at most
    ring_launch_k elements: a launch's parts cover its chunks once, none is empty, and no
    chunk number (the kernel looks three ahead) leaves 32 bits."""
    most, start = rules_lib.ring_launch_k(), 0
    assert most % 16 == 0
    while start < k:
        part = min(k - start, most)
        chunks, per, parts = rules_lib.ring_split(part, tiles)
        assert chunks == -(-part // 16) and chunks + 3 < 1 << 31
        assert (parts - 1) * per < chunks <= parts * per
        assert 1 <= parts <= 65535 and (parts == 1 or per >= 4)
        start += part
