"""Exactly tied correlations at every side and launch shape: the leader's
words come from one lane's registers after the magnitudes alone have been
reduced, so equal magnitudes in one lane, in lanes of one warp and in several
warps must all be decided from the full values, the lowest index first."""
import numpy as np
import pytest

import oracle
import parity

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lib():
    from paper_2605_09190_gb300 import aqmp, build_lib
    build_lib.build()
    assert torch.cuda.is_available()
    return aqmp


def tied_block(b, shift):
    """128 plus b/4 finest-level 2-D Haar atoms of equal magnitude and either
    sign on disjoint 2x2 supports (pixels 128 +- 10); `shift` moves them over
    the columns, so that they fall on other lanes, groups and warps."""
    H = oracle.haar_1d(b)
    fine = [r for r in range(b) if np.count_nonzero(np.abs(H[r]) > 1e-12) == 2]
    y = np.zeros((b, b))
    for k in range(b // 4):
        p, q = fine[(2 * k) % len(fine)], fine[(2 * k + shift) % len(fine)]
        y += (20.0 if k % 3 else -20.0) * np.outer(H[p], H[q])
    blk = np.rint(128.0 + y)
    assert np.allclose(blk, 128.0 + y)
    return blk.astype(np.uint8)


@pytest.mark.parametrize("alt", [False, True])
@pytest.mark.parametrize("b", [4, 8, 16, 32, 64, 128])
def test_tied_atoms_are_taken_in_index_order(lib, b, alt):
    plane = np.concatenate([tied_block(b, s) for s in (0, 1, b // 8)], axis=1)
    dev = [torch.from_numpy(plane).cuda()]
    code = lib.aqmp_encode_planes(dev, [0.5], min_block=b, max_block=b, autotune=False, alt_threads=alt)
    leaves, atoms, lo = code.copy()
    parity.compare(oracle.encode([plane], [0.5], min_block=b, max_block=b), leaves, atoms, lo, [plane])
    fp32 = lib.aqmp_encode_planes(dev, [0.5], min_block=b, max_block=b, autotune=False, alt_threads=alt,
                                  precision=lib.AQMP_PREC_FP32).copy()
    np.testing.assert_array_equal(fp32[0]["n_atoms"], leaves["n_atoms"])
    np.testing.assert_array_equal(fp32[1]["j"], atoms["j"])
