"""Launch rules (csrc/rules.h) on the host."""
import pytest

from tests import rules_lib

# words that fit a 284 208 MiB device beside nothing else
MOST_WORDS = 284208 * (1 << 20) // 8


@pytest.mark.parametrize("k", [1, 16, 17, 784, 6272, (1 << 31) + 5, (1 << 34) - 1, (1 << 34) + 1, 1 << 35, (1 << 35) + 16,
                               MOST_WORDS])
@pytest.mark.parametrize("tiles", [1, 3, 100, 457, 100000])
def test_ring_parts_cover_every_reduction_that_fits_the_device(k, tiles):
    """Every reduction whose operand fits the device is taken; its parts cover the chunks
    once, none is empty, and no chunk number (the kernel looks three ahead) leaves 32 bits."""
    split = rules_lib.ring_split(k, tiles)
    assert split is not None
    chunks, per, parts = split
    assert chunks == -(-k // 16)
    assert (parts - 1) * per < chunks <= parts * per
    assert parts <= 65535 and (parts == 1 or per >= 4)
    assert chunks + 3 < 1 << 32


def test_ring_refuses_what_cannot_exist():
    assert rules_lib.ring_split(0, 1) is None
    assert rules_lib.ring_split(3 << 34, 1) is None
