"""The gather reads four pixels at a time where a plane's address and pitch are
multiples of four, and single bytes elsewhere: the code must not depend on
where the plane lies."""
import numpy as np
import pytest

from paper_2605_09190_gb300 import synthetic

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lib():
    from paper_2605_09190_gb300 import aqmp, build_lib
    build_lib.build()
    assert torch.cuda.is_available()
    return aqmp


@pytest.mark.parametrize("max_block,prec", [(4, 0), (8, 0), (16, 0), (32, 0), (64, 0), (64, 4), (128, 0)])
def test_code_does_not_depend_on_the_planes_alignment(lib, max_block, prec):
    h, w = 2 * max_block, 3 * max_block                 # fewer and more leaves than a group of threads takes
    plane = torch.from_numpy(synthetic.piecewise_scene(h, w, seed=4, patch=max(4, max_block // 2))).cuda()
    params = lib.default_params(rmse_tol=6.0, min_block=4, max_block=max_block, precision=prec)
    want = lib.aqmp_encode_planes([plane], None, params).copy()
    for shift, extra in ((1, 0), (2, 2), (0, 3), (4, 4)):
        room = torch.zeros(h * (w + extra) + shift, dtype=torch.uint8, device="cuda")
        view = room[shift:].as_strided((h, w), (w + extra, 1))
        view.copy_(plane)
        got = lib.aqmp_encode_planes([view], None, params).copy()
        # two calls of the form with rescore on one plane differ in the low words
        for a, b in list(zip(want, got))[:2 if prec == 4 else 3]:
            np.testing.assert_array_equal(a, b)


@pytest.mark.parametrize("b", [4, 16, 32, 64, 128])
def test_correlation_does_not_depend_on_the_blocks_alignment(lib, b):
    n = 5
    blocks = torch.from_numpy(np.random.default_rng(b).integers(0, 256, (n, b, b), dtype=np.uint8)).cuda()
    room = torch.zeros(n * b * b + 1, dtype=torch.uint8, device="cuda")
    odd = room[1:].view(n, b, b)
    odd.copy_(blocks)
    assert torch.equal(lib.aqmp_correlate(b, 0, odd), lib.aqmp_correlate(b, 0, blocks))
    if b == 64:                                         # centred on the blocks' means
        for x, y in zip(lib.aqmp_correlate_bf16x2(b, 0, odd), lib.aqmp_correlate_bf16x2(b, 0, blocks)):
            assert torch.equal(x, y)
