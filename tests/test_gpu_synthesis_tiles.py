"""The synthesis, its adjoint and the SSIM pair at the sizes where their tiles
can go wrong: every side alone and all of them mixed, leaves without atoms
and with more than a batch of them, planes in any order, images one window
high or wide and one off every tile edge.  Reference: plain FP64."""
import numpy as np
import pytest

import bitstream_format
import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
U = 2.0 ** -24                                    # unit roundoff of FP32


@pytest.fixture(scope="module")
def lib():
    from paper_2605_09190_gb300 import aqmp, build_lib
    build_lib.build()
    assert torch.cuda.is_available()
    return aqmp


def make_code(lib, shapes, nb, mb, dict_id, seed):
    """Planes whose roots are split at random, step counts 0, 1, 33 and up to the budget."""
    rng = np.random.default_rng(seed)
    leaves, js, alphas = [], [], []

    def visit(p, y, x, b):
        if b > nb and rng.random() < 0.5:
            h = b // 2
            for dy, dx in ((0, 0), (0, h), (h, 0), (h, h)):
                visit(p, y + dy, x + dx, h)
            return
        n = min(int(rng.choice([0, 1, 2, 33, 70])), max(1, b * b // 4))
        leaves.append({"plane": p, "y": y, "x": x, "b": b, "n_atoms": n, "atom_off": len(js)})
        js.extend(rng.integers(0, (2 if dict_id == 0 else 1) * b * b, n).tolist())
        alphas.extend((rng.normal(0, 10, n) * b / (1 + np.arange(n))).tolist())

    for p, (h, w) in enumerate(shapes):
        for y in range(0, h, mb):
            for x in range(0, w, mb):
                visit(p, y, x, mb)
    js, alphas = np.array(js, np.int64), np.array(alphas, np.float32)
    data = bitstream_format.write(shapes, leaves, js, alphas, dict_id, nb, mb)
    return lib.aqmp_code_from_bitstream(data), leaves, js, alphas


def bases(b, dict_id):
    fam = [oracle.dct_1d(b), oracle.haar_1d(b)]
    return fam if dict_id == 0 else [fam[dict_id - 1]]


def synthesis(shapes, leaves, js, a, dict_id):
    """FP64 planes and the sum of the terms' magnitudes per pixel."""
    out, mag = ([np.zeros(s) for s in shapes] for _ in range(2))
    for L in leaves:
        b, p, n = L["b"], L["plane"], L["b"] ** 2
        sl = np.s_[L["y"]:L["y"] + b, L["x"]:L["x"] + b]
        B = bases(b, dict_id)
        for t in range(L["atom_off"], L["atom_off"] + L["n_atoms"]):
            f = int(js[t]) % n
            term = a[t] * np.outer(B[int(js[t]) // n][f % b], B[int(js[t]) // n][f // b])
            out[p][sl] += term
            mag[p][sl] += np.abs(term)
    return out, mag


CASES = [(4, 4, 0), (8, 8, 0), (16, 16, 0), (32, 32, 0), (64, 64, 0), (128, 128, 0), (4, 128, 0), (4, 64, 1), (8, 64, 2)]


@pytest.mark.parametrize("nb,mb,dict_id", CASES)
def test_synthesis_and_adjoint(lib, nb, mb, dict_id):
    shapes = [(mb, 3 * mb), (2 * mb, mb), (mb, mb)]
    code, leaves, js, alphas = make_code(lib, shapes, nb, mb, dict_id, 7 * mb + nb + dict_id)
    want, mag = synthesis(shapes, leaves, js, alphas.astype(np.float64), dict_id)
    # t terms summed in FP32, each a product of four rounded factors
    bound = [(70 + 6) * U * m for m in mag]
    got = []
    for p, s in enumerate(shapes):
        out = torch.full((s[0], s[1] + 5), float("nan"), device="cuda")       # a pitch of its own
        code.decode(p, out[:, :s[1]])
        assert torch.isnan(out[:, s[1]:]).all()
        got.append(out[:, :s[1]].cpu().numpy())
        assert np.all(np.abs(got[p] - want[p]) <= bound[p] + 1e-30), p

    # all planes in one call, in an order that breaks the run of planes
    rng = np.random.default_rng(3)
    order = [2, 0, 1]
    refs = [torch.from_numpy(rng.uniform(0, 255, shapes[p]).astype(np.float32)).cuda() for p in order]
    recon = [torch.empty_like(r) for r in refs]
    grad = [torch.from_numpy(rng.normal(0, 1, shapes[p]).astype(np.float32)).cuda() for p in order]
    alpha = torch.from_numpy(alphas).cuda()
    if min(min(s) for s in shapes) >= 11:
        rows = lib.aqmp_refine_planes([(p, *shapes[p], r.data_ptr(), r.stride(0), y.data_ptr(), y.stride(0),
                                        g.data_ptr(), g.stride(0)) for p, r, y, g in zip(order, refs, recon, grad)])
        ssim = torch.empty(3, dtype=torch.float64, device="cuda")
        lib.aqmp_refine_forward(code, alpha, rows, ssim)
        for p, y, r, s in zip(order, recon, refs, ssim.tolist()):
            np.testing.assert_array_equal(y.cpu().numpy(), got[p])
            assert abs(s - oracle.ssim(y.cpu().numpy(), r.cpu().numpy(), clip=False)) <= 1e-9
        ga = torch.full_like(alpha, float("nan"))
        lib.aqmp_refine_backward(code, rows, ga)
    else:
        ga = torch.full_like(alpha, float("nan"))
        for p, g in zip(order, grad):
            lib.aqmp_synth_backward(code, p, g, ga)
    ga = ga.cpu().numpy()
    G = {p: g.cpu().numpy().astype(np.float64) for p, g in zip(order, grad)}
    for L in leaves:
        b, n = L["b"], L["b"] ** 2
        blk = G[L["plane"]][L["y"]:L["y"] + b, L["x"]:L["x"] + b]
        B = bases(b, dict_id)
        T = [m @ blk @ m.T for m in B]
        # two sums of b products each of rounded factors
        E = [(2 * b + 8) * U * (np.abs(m) @ np.abs(blk) @ np.abs(m).T) for m in B]
        for t in range(L["atom_off"], L["atom_off"] + L["n_atoms"]):
            fam, f = int(js[t]) // n, int(js[t]) % n
            assert abs(ga[t] - T[fam][f % b, f // b]) <= E[fam][f % b, f // b], (L, t)
    # one plane at a time gives the same, and leaves the others alone
    one = torch.full_like(alpha, float("nan"))
    lib.aqmp_synth_backward(code, order[1], grad[1], one)
    one = one.cpu().numpy()
    mine = np.zeros(len(js), bool)
    for L in leaves:
        if L["plane"] == order[1]:
            mine[L["atom_off"]:L["atom_off"] + L["n_atoms"]] = True
    np.testing.assert_array_equal(one[mine], ga[mine])
    assert np.all(np.isnan(one[~mine]))


def ssim64(x, y):
    t = torch.arange(11, dtype=torch.float64) - 5
    g = torch.exp(-t * t / (2 * 1.5 ** 2))
    g = g / g.sum()

    def win(v):
        h, w = v.shape
        v = sum(g[i] * v[i:h - 10 + i] for i in range(11))
        return sum(g[i] * v[:, i:w - 10 + i] for i in range(11))

    c1, c2 = (0.01 * 255) ** 2, (0.03 * 255) ** 2
    mx, my = win(x), win(y)
    xx, yy, xy = win(x * x) - mx * mx, win(y * y) - my * my, win(x * y) - mx * my
    return ((2 * mx * my + c1) * (2 * xy + c2) / ((mx * mx + my * my + c1) * (xx + yy + c2))).mean()


@pytest.mark.parametrize("h,w", [(11, 11), (11, 300), (300, 11), (32, 42), (33, 43), (64, 74), (65, 75), (63, 73),
                                 (54, 32), (55, 33), (512, 520), (1100, 700)])
@pytest.mark.parametrize("kind", ["noise", "flat", "same"])
def test_ssim_and_gradient_at_tile_edges(lib, h, w, kind):
    rng = np.random.default_rng(h * 1000 + w)
    x = rng.uniform(0, 255, (h, w)).astype(np.float32)
    if kind == "flat":
        x[:] = 137.0
    y = x if kind == "same" else (x + rng.normal(0, 9, (h, w))).astype(np.float32)
    pitch = w + 3
    dev = [torch.zeros((h, pitch), device="cuda") for _ in range(3)]
    dev[0][:, :w], dev[1][:, :w] = torch.from_numpy(x), torch.from_numpy(y)
    dev[2].fill_(float("nan"))
    out = torch.empty((), dtype=torch.float64, device="cuda")
    lib.aqmp_ssim(dev[0][:, :w], dev[1][:, :w], out, dev[2][:, :w], 3.0)
    y64 = torch.from_numpy(y.astype(np.float64)).requires_grad_(True)
    s = ssim64(torch.from_numpy(x.astype(np.float64)), y64)
    (3.0 * s).backward()
    g = y64.grad.numpy()
    assert abs(float(out) - float(s.detach())) <= 1e-9
    got = dev[2].cpu().numpy()
    assert np.all(np.isnan(got[:, w:]))
    # FP32 rounding of each value; the double-float sums err by ~2^-40 of the terms
    assert np.all(np.abs(got[:, :w] - g) <= 2 * U * np.abs(g) + 1e-9 * (np.abs(g).max() + 3.0 / ((h - 10) * (w - 10))))
    val = torch.empty((), dtype=torch.float64, device="cuda")
    lib.aqmp_ssim(dev[0][:, :w], dev[1][:, :w], val)
    assert abs(float(val) - float(out)) <= 1e-12


def test_more_planes_than_one_launch_takes(lib):
    from paper_2605_09190_gb300 import refine
    shapes = [(16, 32)] * 35
    code, leaves, js, alphas = make_code(lib, shapes, 8, 16, 0, 5)
    rng = np.random.default_rng(1)
    refs = [(p, torch.from_numpy(rng.uniform(0, 255, s).astype(np.float32)).cuda()) for p, s in enumerate(shapes)]
    alpha = torch.from_numpy(alphas).cuda().requires_grad_(True)
    total = refine.synthesis_ssim(alpha, code, refs)
    total.backward()
    want, grads = 0.0, torch.zeros_like(alpha)
    for p, r in refs:
        a = torch.from_numpy(alphas).cuda().requires_grad_(True)
        s = refine.synthesis_ssim(a, code, [(p, r)])
        s.backward()
        want += float(s.detach()) / len(refs)
        grads += a.grad / len(refs)
    assert abs(float(total.detach()) - want) <= 1e-12
    assert torch.allclose(alpha.grad, grads, rtol=1e-5, atol=float(grads.abs().max()) * 1e-6)
