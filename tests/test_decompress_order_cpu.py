"""What `decompress` says of a stream that holds no image is known from the
stream alone: no GPU is asked for, and a malformed body comes before it."""
import zlib

import numpy as np
import pytest

import bitstream_format as bsf
from paper_2605_09190_gb300 import aqmp, build_lib


@pytest.fixture(scope="module", autouse=True)
def lib():
    build_lib.build()


def stream():
    shapes = [(8, 8), (8, 16)]
    leaves = [{"plane": p, "b": 8, "n_atoms": 1, "atom_off": i} for i, p in enumerate((0, 1, 1))]
    return bsf.write(shapes, leaves, np.zeros(3, int), np.ones(3), 0, 8, 8)


def test_planes_of_different_sizes_are_no_image():
    with pytest.raises(ValueError, match="different sizes"):
        aqmp.decompress(zlib.compress(stream()))


def test_a_malformed_body_is_reported_first():
    with pytest.raises(aqmp.AqmpError) as e:
        aqmp.decompress(zlib.compress(stream()[:-1]))
    assert e.value.code == -1                                  # AQMP_E_ARG
