"""CPU check of the visited table's tags (visit_tags in csrc/search_impl.cuh): for
the table shapes of the launches, set and tag together tell all ids below 2^b
apart, the set lies in the table and the tag in 15 bits."""
import numpy as np
import pytest


@pytest.mark.parametrize("buckets", [128, 136, 320, 384, 488, 512, 576, 640])
@pytest.mark.parametrize("spare", [1, 8, 12])
def test_set_and_tag_are_the_id(buckets, spare):
    lg = buckets.bit_length() - 1
    b = lg + spare
    shift, tag_shift = 32 - b, 32 - b + lg
    ids = np.arange(1 << b, dtype=np.uint64)
    x = ((ids * 0x9E3779B1) & 0xFFFFFFFF) << shift & 0xFFFFFFFF
    p = x * buckets
    sets, tags = p >> 32, (p & 0xFFFFFFFF) >> tag_shift
    assert sets.max() < buckets and tags.max() < 0x8000
    assert len(np.unique(sets << 16 | tags)) == len(ids)


def test_the_widest_tag_fits_fifteen_bits():
    buckets, lg = 384, 8                     # ids up to 2^23
    last = np.arange((1 << 23) - 4096, 1 << 23, dtype=np.uint64)
    inv = pow(0x9E3779B1, -1, 1 << 23)       # the ids whose hash is the largest
    x = ((last * inv & 0x7FFFFF) * 0x9E3779B1 & 0xFFFFFFFF) << 9 & 0xFFFFFFFF
    p = x * buckets
    assert (p >> 32).max() == buckets - 1 and ((p & 0xFFFFFFFF) >> (9 + lg)).max() < 0x8000
