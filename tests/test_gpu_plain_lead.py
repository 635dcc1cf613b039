"""The FP32 form finds a step's leader in one of two ways, by the correlations a
thread holds.  The launch shapes of sides 16 and 32 lie on both sides of that
rule, and both must make the same choices: on noise, and on blocks whose
correlations tie exactly (a flat one, a checkerboard, a single bright pixel)."""
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


@pytest.mark.parametrize("b,dict_id", [(8, 0), (16, 0), (16, 1), (32, 0), (32, 2)])
def test_launch_shapes_agree_in_the_fp32_form(lib, b, dict_id):
    plane = synthetic.noise_plane(4 * b, 8 * b, seed=b + dict_id).copy()
    plane[:b, :b] = 77
    plane[:b, b:2 * b] = 255 * ((np.arange(b)[:, None] + np.arange(b)[None, :]) % 2)
    plane[:b, 2 * b:3 * b] = 0
    plane[b // 2, 2 * b + b // 4] = 255
    params = lib.default_params(rmse_tol=2.0, min_block=b, max_block=b, dict_id=dict_id, precision=1)
    dev = torch.from_numpy(plane).cuda()
    one = lib.aqmp_encode_planes([dev], None, params, autotune=False).copy()
    other = lib.aqmp_encode_planes([dev], None, params, autotune=False, alt_threads=True).copy()
    assert one[0]["n_atoms"].max() == b * b // 4
    for x, y in zip(one, other):
        np.testing.assert_array_equal(x, y)
