"""What the refinement's autograd function hands to the library, with stand-ins
for the library's calls: references that can be walked once only, and in the
backward no address but those of the gradient images it keeps."""
import pytest

torch = pytest.importorskip("torch")


@pytest.fixture
def calls(monkeypatch):
    from paper_2605_09190_gb300 import aqmp
    seen = {}
    monkeypatch.setattr(aqmp, "aqmp_refine_planes", lambda rows: list(rows))
    monkeypatch.setattr(aqmp, "aqmp_refine_workspace", lambda planes: 16)

    def forward(code, alpha, planes, ssim, workspace=None, stream=None):
        seen["forward"] = planes
        ssim.copy_(torch.arange(1.0, len(planes) + 1.0))
        return ssim

    def backward(code, planes, grad_alpha, stream=None):
        seen["backward"] = planes
        return grad_alpha.fill_(3.0)

    monkeypatch.setattr(aqmp, "aqmp_refine_forward", forward)
    monkeypatch.setattr(aqmp, "aqmp_refine_backward", backward)
    return seen


@pytest.mark.parametrize("grad", [False, True])
def test_references_may_come_from_a_generator(calls, grad):
    from paper_2605_09190_gb300 import refine
    alpha = torch.zeros(5, requires_grad=grad)
    images = [torch.zeros(16, 24), torch.zeros(32, 16)]
    s = refine.synthesis_ssim(alpha, None, ((p, im) for p, im in enumerate(images)))
    assert float(s) == 1.5
    assert [r[:4] for r in calls["forward"]] == [(p, *im.shape, im.data_ptr()) for p, im in enumerate(images)]
    if grad:
        s.backward()
        assert torch.equal(alpha.grad, torch.full((5,), 1.5))


def test_backward_keeps_no_address_of_the_forward(calls):
    from paper_2605_09190_gb300 import refine
    alpha = torch.zeros(5, requires_grad=True)
    images = [torch.zeros(16, 24), torch.zeros(32, 16)]
    s = refine.synthesis_ssim(alpha, None, list(enumerate(images)))
    kept = s.grad_fn.images                                    # alive until the backward
    s.backward()
    # plane, height, width, reference, pitch, synthesis, pitch, gradient, pitch
    at = kept.data_ptr()
    assert calls["backward"] == [(0, 16, 24, None, 0, None, 0, at, 24), (1, 32, 16, None, 0, None, 0, at + 4 * 16 * 24, 16)]
    assert not hasattr(s.grad_fn, "planes")
