"""Exactly tied correlations in Orthogonal MP at sides 32 and 64, where the
CTAs of a cluster hold different columns of a leaf's atoms: the tied atoms lie
in several CTAs at every width of the cluster, and are taken in index order."""
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
    """128 plus b/4 finest-level 2-D Haar atoms of equal magnitude and either sign on disjoint 2x2 supports."""
    H = oracle.haar_1d(b)
    y = sum((20.0 if k % 3 else -20.0) * np.outer(H[b // 2 + 2 * k % (b // 2)], H[b // 2 + (2 * k + shift) % (b // 2)])
            for k in range(b // 4))
    blk = np.rint(128.0 + y)
    assert np.allclose(blk, 128.0 + y)
    return blk.astype(np.uint8)


@pytest.mark.parametrize("b", [32, 64])
def test_tied_atoms_of_several_ctas_are_taken_in_index_order(lib, b):
    three = np.concatenate([tied_block(b, s) for s in (0, 1, b // 8)], axis=1)
    kw = dict(min_block=b, max_block=b)
    want = oracle.encode([three], [0.5], algorithm="omp", **kw)
    j = want.atom_j[1:int(want.leaves["n_atoms"][0])].astype(np.int64)
    assert len(j) >= 8
    assert np.all(np.diff(j) > 0) and len(np.unique(j % (b * b) // b // (b // 8))) == 4      # in eighths of the columns
    for copies in (1, 10, 20, 40):                             # 8, 4, 2 CTAs a leaf and one at side 64
        plane = np.tile(three, (1, copies))
        leaves, atoms, lo = lib.aqmp_encode_planes([torch.from_numpy(plane).cuda()], 0.5, omp=True, **kw).copy()
        n = int(want.leaves["n_atoms"].sum())
        assert len(atoms) == copies * n
        for i in range(copies):
            own = leaves[3 * i:3 * i + 3].copy()
            own["x"] -= 3 * b * i
            own["atom_off"] -= n * i
            parity.compare(want, own, atoms[n * i:n * i + n], lo[n * i:n * i + n], [three], df_tol=2.0 ** -30)
