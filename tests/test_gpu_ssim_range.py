"""The SSIM and its gradient for pixels far beyond any image's, as a refinement
that diverges meets them: as accurate as inside, up to where the squares of the
pixels leave FP32; and gradients scaled by factors that FP32 does not hold.
Reference: the same formula in FP64."""
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


def reference(x, y):
    """Mean SSIM and its gradient by y, in FP64."""
    g = torch.exp(-(torch.arange(11, dtype=torch.float64) - 5) ** 2 / (2 * 1.5 ** 2))
    g = g / g.sum()

    def window(v):
        v = sum(g[i] * v[i:v.shape[0] - 10 + i] for i in range(11))
        return sum(g[i] * v[:, i:v.shape[1] - 10 + i] for i in range(11))

    x, y = x.double().cpu(), y.double().cpu().requires_grad_(True)
    c1, c2 = (0.01 * 255) ** 2, (0.03 * 255) ** 2
    mx, my = window(x), window(y)
    xx, yy, xy = window(x * x) - mx * mx, window(y * y) - my * my, window(x * y) - mx * my
    s = ((2 * mx * my + c1) * (2 * xy + c2) / ((mx * mx + my * my + c1) * (xx + yy + c2))).mean()
    s.backward()
    return float(s.detach()), y.grad.numpy()


@pytest.mark.parametrize("peak", [255.0, 1e6, 1e7, 3e7, 1e9, 1e10, 1e12, 1e15])
def test_pixels_beyond_images(lib, peak):
    rng = np.random.default_rng(5)
    x = rng.uniform(0.0, peak, (75, 90)).astype(np.float32)
    y = (x + rng.uniform(-0.3, 0.3, x.shape) * peak).astype(np.float32)
    y[:30] = rng.uniform(0.0, 255.0, (30, 90))            # windows of image values beside them
    x, y = torch.from_numpy(x).cuda(), torch.from_numpy(y).cuda()
    s, grad = torch.zeros((), dtype=torch.float64, device="cuda"), torch.empty_like(y)
    lib.aqmp_ssim(x, y, s, grad)
    want, want_grad = reference(x, y)
    # window sums good to 2^-44 of E[x^2 + y^2], of which the variances here are a tenth or more
    assert abs(float(s) - want) <= 1e-11
    # ... and the sum of three terms, rounded to FP32, each at most 50 times the largest gradient
    err = np.abs(grad.cpu().numpy().astype(np.float64) - want_grad).max()
    assert err <= 2.0 ** -23 * np.abs(want_grad).max()


@pytest.mark.parametrize("scale", [1.0, -3.0, 3e42, 1e-30, -1e-41, 0.0])
def test_scaled_gradients(lib, scale):
    rng = np.random.default_rng(6)
    x = torch.from_numpy(rng.uniform(0.0, 255.0, (64, 64)).astype(np.float32)).cuda()
    y = torch.from_numpy(rng.uniform(0.0, 255.0, (64, 64)).astype(np.float32)).cuda()
    s, grad = torch.zeros((), dtype=torch.float64, device="cuda"), torch.empty_like(y)
    lib.aqmp_ssim(x, y, s, grad, scale)
    want = reference(x, y)[1] * scale
    assert np.abs(want).max() < np.finfo(np.float32).max
    err = np.abs(grad.cpu().numpy().astype(np.float64) - want).max()
    assert err <= 2.0 ** -23 * np.abs(want).max() + 2.0 ** -149      # the last: the spacing of the smallest FP32 numbers
