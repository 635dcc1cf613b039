"""The plain FP32 form against a restatement on the host, bit for bit: the
largest magnitude, the lowest index among equals, one FMA an element.  Every
side, dictionary and launch shape, on noise and on blocks whose correlations
tie exactly; the restatement starts from the library's own correlations."""
import numpy as np
import pytest

import oracle
from paper_2605_09190_gb300 import synthetic

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
f32 = np.float32


@pytest.fixture(scope="module")
def lib():
    from paper_2605_09190_gb300 import aqmp, build_lib
    build_lib.build()
    assert torch.cuda.is_available()
    return aqmp


def fma(a, b, c):
    """a b + c rounded once: the sum of a 48-bit product and a 24-bit number in long double, then to FP32."""
    return (a.astype(np.longdouble) * b.astype(np.longdouble) + c.astype(np.longdouble)).astype(f32)


def pursuit(c, e0, eps2, k, b, W):
    """c: [families][q][p] FP32.  Returns (j, alpha)."""
    n, c, e, js, alphas = b * b, c.copy(), f32(e0), [], []
    while not e < eps2 and len(js) < k:
        j = int(np.argmax(np.abs(c.reshape(-1))))
        a = c.reshape(-1)[j]
        if a == 0:
            break
        js.append(j)
        alphas.append(a)
        e = fma(-a[None], a[None], np.array([e], f32))[0]
        fam, q, p = j // n, j % n // b, j % b
        if len(c) == 2:
            V = W if fam == 0 else W.T
            u = a * V[p]                                       # by p'
            c[1 - fam] = fma(np.broadcast_to(-u[None, :], (b, b)), np.broadcast_to(V[q][:, None], (b, b)), c[1 - fam])
        c.reshape(-1)[j] = 0
    return js, alphas


@pytest.mark.parametrize("alt", [False, True])
@pytest.mark.parametrize("b,dict_id", [(b, d) for b in (4, 8, 16, 32, 64, 128) for d in (0, 1, 2)])
def test_choices_and_coefficients(lib, b, dict_id, alt):
    plane = synthetic.noise_plane(b, 5 * b, seed=b + dict_id).copy()
    plane[:, :b] = 77
    plane[:, b:2 * b] = 255 * ((np.arange(b)[:, None] + np.arange(b)[None, :]) % 2)
    plane[:, 2 * b:3 * b] = 0
    plane[b // 2, 2 * b + b // 4] = 255
    plane[:, 3 * b:4 * b] = synthetic.piecewise_scene(b, b, seed=2, patch=b // 2)
    tol, k = 2.0, min(b * b // 4, 200)
    params = lib.default_params(rmse_tol=tol, min_block=b, max_block=b, dict_id=dict_id, precision=lib.AQMP_PREC_FP32,
                                cap_num=k, cap_den=b * b)
    leaves, atoms, lo = lib.aqmp_encode_planes([torch.from_numpy(plane).cuda()], None, params, autotune=False,
                                               alt_threads=alt).copy()
    blocks = np.ascontiguousarray(plane.reshape(b, 5, b).transpose(1, 0, 2))
    c = lib.aqmp_correlate(b, dict_id, torch.from_numpy(blocks).cuda()).cpu().numpy()[..., 0]
    W = oracle.dct_1d(b) @ oracle.haar_1d(b).T
    W[np.abs(W) < 2.0 ** -40] = 0.0
    eps2 = f32(f32(tol) * f32(tol)) * f32(b * b)
    assert len(leaves) == 5 and not np.any(lo)
    for i, L in enumerate(leaves):
        e0 = int((blocks[i].astype(np.int64) ** 2).sum())
        js, alphas = pursuit(c[i].reshape(-1, b, b), e0, eps2, k, b, W.astype(f32))
        at = slice(int(L["atom_off"]), int(L["atom_off"]) + int(L["n_atoms"]))
        np.testing.assert_array_equal(atoms["j"][at], js)
        np.testing.assert_array_equal(atoms["alpha"][at].view(np.uint32), np.array(alphas, f32).view(np.uint32))
