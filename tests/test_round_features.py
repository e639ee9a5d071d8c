"""The library's bf16 rounding of host features equals the integer rule bit for bit, whatever the pattern."""
import numpy as np

from paper_2304_14698_b200 import xrl_round_features
from paper_2304_14698_b200.binding import to_bf16_bits


def test_rounding_of_every_kind_of_pattern():
    rng = np.random.default_rng(3)
    u = rng.integers(0, 2**32, size=100003, dtype=np.uint64).astype(np.uint32)
    edges = np.array([0, 0x80000000, 0x7F800000, 0xFF800000, 0x7FC00000, 0x7F800001, 0xFFFFFFFF, 0x3F808000, 0x3F818000,
                      0x7F7FFFFF, 1, 0x007FFFFF], np.uint32)
    x = np.concatenate([edges, u]).view(np.float32)
    assert np.array_equal(xrl_round_features(x), to_bf16_bits(x))
    assert np.array_equal(xrl_round_features(x[:24].reshape(3, 8)[:, ::2]), to_bf16_bits(x[:24].reshape(3, 8)[:, ::2]))
    assert xrl_round_features(np.zeros((0, 8), np.float32)).shape == (0, 8)
