"""The mean SSIM of images that hardly differ, and of images that do, against
the formula in long double: the windows' errors may not hide 1 - SSIM."""
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


def windows(x, y):
    """The windows' SSIM in long double, and 1 - A2 / B2 and E[x^2 + y^2] / B2 of each."""
    L = np.longdouble
    g = np.exp(-(np.arange(11, dtype=L) - 5) ** 2 / L(4.5))
    g = (g / g.sum()).astype(L)

    def w(v):
        v = sum(g[i] * v[:, i:v.shape[1] - 10 + i] for i in range(11))
        return sum(g[i] * v[i:v.shape[0] - 10 + i] for i in range(11))

    x, y = x.astype(L), y.astype(L)
    c1, c2 = L(0.01 * 255) ** 2, L(0.03 * 255) ** 2
    mx, my, es, exy = w(x), w(y), w(x * x + y * y), w(x * y)
    a2, b2 = 2 * (exy - mx * my) + c2, es - mx * mx - my * my + c2
    return (2 * mx * my + c1) / (mx * mx + my * my + c1) * a2 / b2, np.abs(1 - a2 / b2), es / b2


@pytest.mark.parametrize("scene,noise", [("flat", 0.01), ("flat", 5.0), ("piecewise", 0.3), ("piecewise", 1.0),
                                         ("piecewise", 4.0), ("gradient", 8.0)])
def test_mean_against_long_double(lib, scene, noise):
    h, w = 150, 170
    x = {"flat": lambda: np.full((h, w), 250), "piecewise": lambda: synthetic.piecewise_scene(h, w, seed=3),
         "gradient": lambda: synthetic.gradient_scene(h, w, seed=3)}[scene]().astype(np.float32)
    y = (x + np.random.default_rng(1).normal(0.0, noise, x.shape)).astype(np.float32)
    f, far, amp = windows(x, y)
    s = torch.zeros((), dtype=torch.float64, device="cuda")
    lib.aqmp_ssim(torch.from_numpy(x).cuda(), torch.from_numpy(y).cuda(), s)
    # window sums good to 2^-45; what they leave in B2, times 1 - A2 / B2; the formula's own roundings
    bound = 2.0 ** -45 * float((amp * far).mean()) + 2.0 ** -44
    assert abs(float(np.longdouble(float(s)) - f.mean())) <= bound
