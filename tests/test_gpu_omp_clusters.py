"""Orthogonal MP at sides 32 and 64 takes one to eight CTAs a leaf, as the
level's leaves leave SMs for: every width of the cluster must make the same
choices, with coefficients equal up to the rounding of FP64 sums in another
order, and the widest must agree with the FP64 oracle."""
import numpy as np
import pytest

import oracle
import parity
from paper_2605_09190_gb300 import synthetic

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lib():
    from paper_2605_09190_gb300 import aqmp, build_lib
    build_lib.build()
    assert torch.cuda.is_available()
    return aqmp


def encode(lib, plane, tol, **kw):
    code = lib.aqmp_encode_planes([torch.from_numpy(plane).cuda()], tol, omp=True, **kw)
    return code.copy()


@pytest.mark.parametrize("b,cap", [(64, (3, 128)), (64, (1, 4)), (32, (3, 64)), (32, (1, 4))])
def test_every_cluster_width_makes_the_same_choices(lib, b, cap):
    # two blocks, one that converges soon and one with more structure; with a
    # quarter of the pixels as budget the support arrays are at their largest
    tol = 4.0
    two = np.concatenate([synthetic.gradient_scene(b, b, seed=2), synthetic.piecewise_scene(b, b, seed=9, patch=b // 2)], 1)
    kw = dict(min_block=b, max_block=b, cap_num=cap[0], cap_den=cap[1])
    leaves, atoms, lo = encode(lib, two, tol, **kw)
    assert leaves["n_atoms"].min() >= 2
    if not (b == 64 and cap == (1, 4)):      # the oracle's re-fit of 1024 atoms takes the better part of an hour
        parity.compare(oracle.encode([two], [tol], algorithm="omp", **kw), leaves, atoms, lo, [two])
    alpha = atoms["alpha"].astype(np.float64) + lo
    for copies in (10, 20, 40, 80):
        gl, ga, glo = encode(lib, np.tile(two, (1, copies)), tol, **kw)
        np.testing.assert_array_equal(gl["n_atoms"], np.tile(leaves["n_atoms"], copies))
        np.testing.assert_array_equal(gl["flags"], np.tile(leaves["flags"], copies))
        np.testing.assert_array_equal(ga["j"], np.tile(atoms["j"], copies))
        got = ga["alpha"].astype(np.float64) + glo
        # a few hundred FP64 operations each, amplified by the support's condition
        assert np.abs(got - np.tile(alpha, copies)).max() <= 1e-9 * np.abs(alpha).max()
