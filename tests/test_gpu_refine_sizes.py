"""The planes of a refinement step have to have their own size: the synthesis
writes, and the adjoint reads, the whole plane of the code, while the SSIM goes
by the descriptor.  Every image here has room for the largest descriptor."""
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


@pytest.mark.parametrize("dh,dw", [(-16, 0), (0, -16), (1, 0), (0, 1), (16, 16)])
def test_another_size_than_the_planes_is_refused(lib, dh, dw):
    h, w = 32, 48
    code = lib.aqmp_encode_planes([torch.from_numpy(synthetic.gradient_scene(h, w, seed=1)).cuda()], 2.0,
                                  min_block=4, max_block=16)
    _, alpha = lib.aqmp_device_atoms(code)
    pitch = 96
    ref, recon, grad = (torch.zeros((96, pitch), device="cuda") for _ in range(3))
    ssim = torch.zeros(1, dtype=torch.float64, device="cuda")
    work = torch.zeros(1 << 20, dtype=torch.uint8, device="cuda")
    out = torch.zeros_like(alpha)

    def rows(hh, ww):
        return lib.aqmp_refine_planes([(0, hh, ww, ref.data_ptr(), pitch, recon.data_ptr(), pitch, grad.data_ptr(),
                                        pitch)])

    lib.aqmp_refine_forward(code, alpha, rows(h, w), ssim, work)
    lib.aqmp_refine_backward(code, rows(h, w), out)
    for call in (lambda p: lib.aqmp_refine_forward(code, alpha, p, ssim),
                 lambda p: lib.aqmp_refine_forward(code, alpha, p, ssim, work),
                 lambda p: lib.aqmp_refine_backward(code, p, out)):
        with pytest.raises(lib.AqmpError) as e:
            call(rows(h + dh, w + dw))
        assert e.value.code == -1                              # AQMP_E_ARG
    torch.cuda.synchronize()
    assert np.isfinite(float(ssim))
