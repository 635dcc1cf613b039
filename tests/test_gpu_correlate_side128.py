"""Side 128 on the tensor cores takes one leaf at a time per SM: one leaf, a few,
and more than there are SMs (so that a CTA goes on to another leaf) must give
the integer SIMT kernel's bits, on noise, on flat blocks at both ends of the
range and on halves of opposite value, where the digit sums are largest."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lib():
    from paper_2605_09190_gb300 import aqmp, build_lib
    build_lib.build()
    assert torch.cuda.is_available()
    return aqmp


@pytest.mark.parametrize("dict_id,L", [(0, 1), (1, 3), (0, 7), (1, 350)])
def test_tensor_cores_give_the_simt_bits(lib, dict_id, L):
    b = 128
    x = np.random.default_rng(L).integers(0, 256, size=(L, b, b), dtype=np.uint8)
    if L > 3:
        x[0], x[1] = 0, 255
        x[2] = np.where(np.arange(b)[None, :] < b // 2, 255, 0)
        x[3] = np.where(np.arange(b)[:, None] < b // 2, 0, 255)
    dev = torch.from_numpy(x).cuda()
    got, want = lib.aqmp_correlate(b, dict_id, dev, gemm=0), lib.aqmp_correlate(b, dict_id, dev, gemm=1)
    assert torch.equal(got.view(torch.int32), want.view(torch.int32))
