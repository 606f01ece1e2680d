"""K2's shared row limit: the rounded-up entry bounds every exact value that
carries its tag (plain Python restatement of the library's bit rule)."""
import numpy as np
import pytest


def tag_ceil(v, mask):
    u = int(np.float32(v).view(np.uint32))
    u = (u & ~mask) if u & 0x80000000 else (u | mask)
    return np.uint32(u & 0xffffffff).view(np.float32)


@pytest.mark.parametrize("tag_bits", [4, 5])
def test_ceiling_is_at_least_the_exact_value(tag_bits):
    rng = np.random.default_rng(tag_bits)
    mask = (1 << tag_bits) - 1
    vals = np.concatenate([rng.normal(size=500) * 10.0 ** rng.uniform(-40, 38, 500), [0.0, -0.0, 1e-45, 3.4e38]])
    for v in vals.astype(np.float32):
        for tag in (0, 1, mask):
            tagged = np.uint32((int(v.view(np.uint32)) & ~mask & 0xffffffff) | tag).view(np.float32)
            assert tag_ceil(tagged, mask) >= v
