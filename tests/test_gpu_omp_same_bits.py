"""A leaf's OMP coefficients at sides 32 and 64 are sums whose order goes by the
support alone: they have the same bits however many leaves share the call (and
so however many CTAs a leaf gets), and supports of up to 1024 atoms solve their
least-squares problem to FP64 accuracy."""
import numpy as np
import pytest

import oracle
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
    return lib.aqmp_encode_planes([torch.from_numpy(plane).cuda()], tol, omp=True, **kw).copy()


# budgets on both sides of where a product is formed as fewer partial sums (256, 512 atoms), one block of 32, all
@pytest.mark.parametrize("b,k", [(64, 31), (64, 260), (64, 520), (64, 1024), (32, 33), (32, 256)])
def test_bits_do_not_depend_on_the_number_of_leaves(lib, b, k):
    two = np.concatenate([synthetic.noise_plane(b, b, seed=4), synthetic.piecewise_scene(b, b, seed=9, patch=b // 2)], 1)
    kw = dict(min_block=b, max_block=b, cap_num=k, cap_den=b * b)
    leaves, atoms, lo = encode(lib, two, 0.0, **kw)
    assert (leaves["n_atoms"] == k).all()
    for copies in (10, 20, 40, 80):                            # 8, 4, 2 CTAs a leaf and one at side 64
        gl, ga, glo = encode(lib, np.tile(two, (1, copies)), 0.0, **kw)
        np.testing.assert_array_equal(gl["flags"], np.tile(leaves["flags"], copies))
        np.testing.assert_array_equal(ga["j"], np.tile(atoms["j"], copies))
        np.testing.assert_array_equal(ga["alpha"].view(np.uint32), np.tile(atoms["alpha"].view(np.uint32), copies))
        np.testing.assert_array_equal(glo.view(np.uint32), np.tile(lo.view(np.uint32), copies))


@pytest.mark.parametrize("b", [32, 64])
def test_long_supports_solve_the_least_squares_problem(lib, b):
    blk = synthetic.piecewise_scene(b, b, seed=9, patch=b // 2)
    _, atoms, lo = encode(lib, blk, 0.0, min_block=b, max_block=b)
    D = oracle.dictionary(b, 0)[atoms["j"]]
    y = oracle.unravel(blk).astype(np.float64)
    G, x = D @ D.T, np.zeros(len(D), np.longdouble)
    Dl = D.astype(np.longdouble)
    for _ in range(3):                                         # refined with long double residuals
        x = x + np.linalg.solve(G, (Dl @ (y - Dl.T @ x)).astype(np.float64))
    assert len(D) == b * b // 4
    got = atoms["alpha"].astype(np.float64) + lo
    # correlations and Gram entries good to 2^-47, a support's condition (17 and 35), and the 48 bits of the result
    assert np.abs(got - x).max() <= 2.0 ** -47 * np.linalg.cond(G) * np.abs(x).max()
