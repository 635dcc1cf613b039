"""Performance cases: the calls a program makes of this package, over the sizes it makes them at.

Encodes of whole images (the encoder is what the package is for) from one 64x64 block to a batch of 64 colour
images, with Matching Pursuit at every root side and with Orthogonal Matching Pursuit; the initial correlation
on its own; the decoder and the whole of `decompress`; one step of the coefficient refinement, forward and
backward.  Images are the synthetic scenes of `paper_2605_09190_gb300/synthetic.py`, drawn on the GPU from the
case's seed; the decoder's and the refinement's codes are written here as bitstreams, so that what they should
return can be computed without the package.
"""
import math
import struct
import zlib

import numpy as np
import torch

from paper_2605_09190_gb300 import aqmp, refine

DEV = "cuda"
# atoms the encoder emits per pixel, measured on the scenes below (rounded): what an encode has to write
ATOMS = {("gradient", 1.0): 0.2, ("gradient", 2.0): 0.01, ("gradient", 4.0): 0.003, ("gradient", 8.0): 0.001,
         ("piecewise", 1.0): 0.16, ("piecewise", 2.0): 0.1, ("piecewise", 4.0): 0.02, ("piecewise", 8.0): 0.004}


def listed():
    return [
        # one 64x64 grey block: the smallest call there is, bound by launches and latency
        {"name": "encode 64x64", "kind": "encode", "images": 1, "channels": 1, "h": 64, "w": 64, "uneven": 0,
         "scene": "gradient", "tol": 2.0, "sweep": False, "min_block": 4, "max_block": 64, "precision": 0,
         "omp": False, "host": False},
        # one 512x512 grey image at four tolerances in one call (choosing a quality), from host memory, as a
        # program that has just read the file has it
        {"name": "encode 512 sweep", "kind": "encode", "images": 4, "channels": 1, "h": 512, "w": 512, "uneven": 0,
         "scene": "piecewise", "tol": 1.0, "sweep": True, "min_block": 4, "max_block": 64, "precision": 0,
         "omp": False, "host": True},
        # 64 RGB images of uneven sizes in one call, mostly smooth content: the largest batch
        {"name": "encode batch 64 gradient", "kind": "encode", "images": 64, "channels": 3, "h": 1536, "w": 2048,
         "uneven": 1, "scene": "gradient", "tol": 2.0, "sweep": False, "min_block": 4, "max_block": 64,
         "precision": 0, "omp": False, "host": False},
        # a dozen RGB images of uneven sizes, detailed content: most blocks split down the tree
        {"name": "encode batch 12 piecewise", "kind": "encode", "images": 12, "channels": 3, "h": 1536, "w": 2048,
         "uneven": 2, "scene": "piecewise", "tol": 2.0, "sweep": False, "min_block": 4, "max_block": 64,
         "precision": 0, "omp": False, "host": False},
        # one large RGB image with 128x128 roots
        {"name": "encode 4096 root 128", "kind": "encode", "images": 1, "channels": 3, "h": 4096, "w": 4096,
         "uneven": 0, "scene": "gradient", "tol": 2.0, "sweep": False, "min_block": 4, "max_block": 128,
         "precision": 0, "omp": False, "host": False},
        # a photograph-sized RGB image in the plain FP32 form (speed before certified decisions)
        {"name": "encode 1088x1920 fp32", "kind": "encode", "images": 1, "channels": 3, "h": 1088, "w": 1920,
         "uneven": 0, "scene": "piecewise", "tol": 4.0, "sweep": False, "min_block": 4, "max_block": 64,
         "precision": 1, "omp": False, "host": False},
        # Orthogonal Matching Pursuit, the solver the paper's authors ran: small roots over a whole image, and
        # the default roots on a small one
        {"name": "encode 512 omp root 16", "kind": "encode", "images": 4, "channels": 1, "h": 512, "w": 512,
         "uneven": 0, "scene": "piecewise", "tol": 1.0, "sweep": True, "min_block": 4, "max_block": 16,
         "precision": 0, "omp": True, "host": False},
        {"name": "encode 256 omp root 64", "kind": "encode", "images": 1, "channels": 1, "h": 256, "w": 256,
         "uneven": 0, "scene": "piecewise", "tol": 8.0, "sweep": False, "min_block": 4, "max_block": 64,
         "precision": 0, "omp": True, "host": False},
        # the initial correlation by itself, for a program with a solver of its own
        {"name": "correlate 64", "kind": "correlate", "b": 64, "blocks": 4096, "dict": 0},
        # decoding a large RGB image into device memory
        {"name": "decode 1536x2048", "kind": "decode", "channels": 3, "h": 1536, "w": 2048, "min_block": 4,
         "max_block": 64, "codec": False},
        # a small compressed YCbCr file to an image: inflate, parse, upload, decode, colour conversion
        {"name": "decompress 512x768", "kind": "decode", "channels": 3, "h": 512, "w": 768, "min_block": 4,
         "max_block": 64, "codec": True},
        # one refinement step of 16 planes: SSIM of the synthesis and its gradient by the coefficients
        {"name": "refine 16x512", "kind": "refine", "channels": 16, "h": 512, "w": 512, "min_block": 8,
         "max_block": 32},
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _size(rng, side, lo, hi):
    """A side length in [lo, hi], a multiple of the root side `side`."""
    return max(side, int(_log(rng, lo, hi)) // side * side)


def draw(rng):
    what = rng.choice(["encode"] * 9 + ["omp"] * 2 + ["correlate"] * 2 + ["decode"] * 2 + ["codec"] + ["refine"] * 2)
    if what == "encode":
        root = rng.choice([16, 32, 64, 64, 64, 64, 128])
        channels = rng.choice([1, 3, 3])
        h, w = _size(rng, root, 64, 2048), _size(rng, root, 64, 2048)
        most = (8 << 20) if root == 128 else (48 << 20)               # pixels of all planes
        images = max(1, min(64, int(_log(rng, 1, 64)), most // (h * w * channels)))
        return {"kind": "encode", "images": images, "channels": channels, "h": h, "w": w,
                "uneven": rng.randrange(1, 1000) if images > 2 else 0, "scene": rng.choice(["gradient", "piecewise"]),
                "tol": rng.choice([1.0, 2.0, 2.0, 4.0, 8.0]), "sweep": False, "min_block": rng.choice([4, 4, 4, 8]),
                "max_block": root, "precision": rng.choice([0, 0, 0, 0, 1, 2, 4]), "omp": False,
                "host": rng.random() < 0.2}
    if what == "omp":
        root = rng.choice([8, 16, 16, 32, 64])
        most = {8: 1024, 16: 1024, 32: 384, 64: 192}[root]
        return {"kind": "encode", "images": 1, "channels": rng.choice([1, 3]) if root < 32 else 1,
                "h": _size(rng, root, 64, most), "w": _size(rng, root, 64, most), "uneven": 0,
                "scene": rng.choice(["gradient", "piecewise"]), "tol": rng.choice([4.0, 8.0]), "sweep": False,
                "min_block": 4, "max_block": root, "precision": 0, "omp": True, "host": False}
    if what == "correlate":
        b = rng.choice([4, 8, 16, 32, 64, 128])
        return {"kind": "correlate", "b": b, "blocks": max(1, int(_log(rng, 1 << 14, 1 << 24)) // (b * b)),
                "dict": rng.choice([0, 0, 0, 1, 2])}
    if what in ("decode", "codec"):
        root = rng.choice([16, 32, 64, 64, 64, 128])
        return {"kind": "decode", "channels": rng.choice([1, 3]) if what == "decode" else 3,
                "h": _size(rng, root, 64, 2048 if what == "decode" else 768),
                "w": _size(rng, root, 64, 2048 if what == "decode" else 768), "min_block": rng.choice([4, 8]),
                "max_block": root, "codec": what == "codec"}
    root = rng.choice([16, 32, 32, 64])
    h, w = _size(rng, root, 64, 1024), _size(rng, root, 64, 1024)
    return {"kind": "refine", "channels": max(1, min(16, int(_log(rng, 1, 16)), (4 << 20) // (h * w))), "h": h,
            "w": w, "min_block": rng.choice([4, 8]), "max_block": root}


# ------------------------------------------------------------------ inputs

def _sizes(case):
    """(h, w) of every image: the case's own, or uneven ones up to it, in multiples of the root side."""
    if not case["uneven"]:
        return [(case["h"], case["w"])] * case["images"]
    rng = np.random.default_rng(case["uneven"])
    side, h, w = case["max_block"], case["h"], case["w"]
    return [(side * int(rng.integers(max(1, h // 6 // side), h // side + 1)),
             side * int(rng.integers(max(1, w // 8 // side), w // side + 1))) for _ in range(case["images"])]


def _gradient(h, w, rng, gen):
    yy = torch.arange(h, device=DEV, dtype=torch.float32)[:, None]
    xx = torch.arange(w, device=DEV, dtype=torch.float32)[None]
    img = 40.0 + 60.0 * (xx / w + yy / h)
    img = img + 60.0 * (xx >= rng.uniform(0.25 * w, 0.75 * w)) - 60.0 * (yy >= rng.uniform(0.25 * h, 0.75 * h))
    rad = 12.0 * min(h, w) / 64.0
    img = img + 80.0 * ((yy - rng.uniform(0, h)) ** 2 + (xx - rng.uniform(0, w)) ** 2 <= rad * rad)
    return img + 2.0 * torch.randn((h, w), generator=gen, device=DEV)


def _piecewise(h, w, rng, gen):
    yy = torch.arange(h, device=DEV, dtype=torch.float32)[:, None]
    xx = torch.arange(w, device=DEV, dtype=torch.float32)[None]
    best = img = None
    for _ in range(8):                                                # Voronoi regions, a plane each
        sy, sx = rng.uniform(0, h), rng.uniform(0, w)
        d2 = (yy - sy) ** 2 + (xx - sx) ** 2
        plane = rng.uniform(50, 200) + rng.uniform(-0.15, 0.15) * (yy - sy) + rng.uniform(-0.15, 0.15) * (xx - sx)
        img = plane if best is None else torch.where(d2 < best, plane, img)
        best = d2 if best is None else torch.minimum(best, d2)
    for _ in range(20):                                               # straight step edges
        py, px, th = rng.uniform(0, h), rng.uniform(0, w), rng.uniform(0, math.pi)
        hgt = rng.uniform(20.0, 60.0) * rng.choice([-1.0, 1.0])
        img = img + hgt * ((yy - py) * math.cos(th) - (xx - px) * math.sin(th) >= 0)
    ph, pw = min(128, h), min(128, w)                                 # a texture patch
    ty, tx = int(rng.integers(0, h - ph + 1)), int(rng.integers(0, w - pw + 1))
    tex = torch.zeros((ph, pw), device=DEV)
    for _ in range(16):
        fr, an, phs = rng.uniform(0.02, 0.25), rng.uniform(0, 2 * math.pi), rng.uniform(0, 2 * math.pi)
        tex += torch.cos(2 * math.pi * fr * (math.cos(an) * xx[:, :pw] + math.sin(an) * yy[:ph]) + phs)
    img[ty:ty + ph, tx:tx + pw] += tex * (20.0 / math.sqrt(8.0))
    return img + 3.0 * torch.randn((h, w), generator=gen, device=DEV)


def _scene(scene, h, w, rng, gen):
    img = (_gradient if scene == "gradient" else _piecewise)(h, w, rng, gen)
    return img.round().clamp(0, 255)


def _gen(seed):
    return np.random.default_rng(seed), torch.Generator(device=DEV).manual_seed(int(seed) % (1 << 62))


def _code_arrays(case, seed):
    """A code as an encoder leaves it: per plane the quadtree's leaves in canonical order (row, column, side,
    step count) and all atoms (index, coefficient), step counts and magnitudes like those of real pursuits.
    The tree belongs to the case (so that results of one case have one shape), the atoms to the seed."""
    rng = np.random.default_rng(case["h"] * 65536 + case["w"])
    nb, mb = case["min_block"], case["max_block"]
    levels = int(math.log2(mb // nb))
    ry, rx = case["h"] // mb, case["w"] // mb
    planes = []
    for _ in range(case["channels"]):
        root = np.arange(ry * rx)
        y, x, z = root // rx * mb, root % rx * mb, root << (2 * levels)   # z: position in depth-first order
        got = []
        for lev in range(levels + 1):
            b = mb >> lev
            split = (rng.random(len(y)) < (0.75, 0.65, 0.45, 0.35, 0.3)[min(lev, 4)]) & (lev < levels)
            keep = ~split
            got.append(np.stack([z[keep], y[keep], x[keep], np.full(keep.sum(), b)], 1))
            y, x, z = y[split], x[split], z[split]
            q, h = 1 << (2 * (levels - lev - 1)) if lev < levels else 0, b // 2
            z = (z[:, None] + q * np.arange(4)).ravel()
            y, x = (y[:, None] + h * np.array([0, 0, 1, 1])).ravel(), (x[:, None] + h * np.array([0, 1, 0, 1])).ravel()
        leaves = np.concatenate(got)
        leaves = leaves[np.argsort(leaves[:, 0])][:, 1:]
        k = np.maximum(1, leaves[:, 2] ** 2 // 4)
        planes.append((leaves, np.maximum(1, (k * rng.random(len(k)) ** 3).astype(np.int64))))
    rng = np.random.default_rng(seed)
    sides = np.concatenate([p[0][:, 2] for p in planes])
    steps = np.concatenate([p[1] for p in planes])
    at = np.repeat(np.arange(len(steps)), steps)                       # the atoms' leaves
    t = np.arange(len(at)) - np.repeat(np.cumsum(steps) - steps, steps)
    b = sides[at]
    p, q = ((b * rng.random(len(at)) ** 1.5).astype(np.int64) for _ in range(2))   # low frequencies more often
    j = np.where(t == 0, 0, rng.integers(0, 2, len(at)) * b * b + q * b + p)
    alpha = np.where(t == 0, b * rng.uniform(60, 190, len(at)), b * rng.normal(0, 12, len(at)) / (1 + t))
    return planes, at, sides, j, alpha.astype(np.float32)


def _bitstream(case, planes, j, alpha, color):
    top = int(math.log2(case["max_block"]))
    out = [struct.pack("<4sBBBBHHI", b"AQMP", 1, color, 0, 0, case["min_block"], case["max_block"], len(planes))]
    out += [struct.pack("<IIII", case["h"], case["w"], len(n), int(n.sum())) for _, n in planes]
    off = 0
    for leaves, n in planes:
        out.append((top - np.log2(leaves[:, 2]).astype(np.int64)).astype(np.uint8).tobytes())
        v = n.copy()
        part = np.stack([v & 127, v >> 7 & 127, v >> 14], 1)            # LEB128, at most three bytes
        more = np.stack([v >= 1 << 7, v >= 1 << 14, np.zeros(len(v), bool)], 1)
        keep = np.concatenate([np.ones((len(v), 1), bool), more[:, :2]], 1)
        out.append((part | more << 7).astype(np.uint8)[keep].tobytes())
        m = int(n.sum())
        out += [j[off:off + m].astype("<u2").tobytes(), alpha[off:off + m].astype("<f4").tobytes()]
        off += m
    return b"".join(out)


def _refs(case, seed):
    rng, gen = _gen(seed)
    return [_scene("piecewise", case["h"], case["w"], rng, gen) for _ in range(case["channels"])]


def _records(case, n_leaves=0, n_atoms=0):
    """Page-locked arrays that a program keeps to read results into, with room for more than is expected (zeros
    past the result): leaves, atoms (index, coefficient bits), low words."""
    px = sum(h * w for h, w in _sizes(case)) * (1 if case["sweep"] else case["channels"])
    worst = px // case["min_block"] ** 2
    tols = [2.0 ** i for i in range(case["images"])] if case["sweep"] else [case["tol"]]
    expect = int(px * max(ATOMS[case["scene"], t] for t in tols))
    if px <= (2 << 20) or case["precision"] == 2:
        expect = px
    n_leaves = max(n_leaves, min(worst, (1 << 18) + expect // 2))
    n_atoms = max(n_atoms, min(px // 4 + worst, (1 << 16) + 3 * expect))
    return [torch.zeros(s, dtype=torch.int32, pin_memory=True)
            for s in ((n_leaves, aqmp.LEAF_DTYPE.itemsize // 4), (n_atoms, 2), (n_atoms,))]


def prepare(case, seed):
    kind = case["kind"]
    if kind == "encode":
        rng, gen = _gen(seed)
        images = []
        for h, w in _sizes(case):
            planes = [_scene(case["scene"], h, w, rng, gen).to(torch.uint8) for _ in range(case["channels"])]
            images.append(torch.stack(planes))
        if case["sweep"]:                                             # one image, a plane per tolerance
            images = images[:1]
        if case["host"]:
            images = [im.cpu().numpy() for im in images]
        params = aqmp.default_params(rmse_tol=case["tol"], min_block=case["min_block"], max_block=case["max_block"],
                                     precision=case["precision"])
        return {"case": case, "images": images, "params": params, "records": _records(case)}
    if kind == "correlate":
        rng, gen = _gen(seed)
        b, n = case["b"], case["blocks"]
        wide = min(n, max(1, 2048 // b))                               # blocks of a piecewise scene, in raster order
        img = _scene("piecewise", -(-n // wide) * b, wide * b, rng, gen).to(torch.uint8)
        blocks = img.reshape(-1, b, wide, b).transpose(1, 2).reshape(-1, b, b)[:n].contiguous()
        return {"case": case, "blocks": blocks}
    planes, _, _, j, alpha = _code_arrays(case, seed)
    data = _bitstream(case, planes, j, alpha, 2 if case.get("codec") else 0)
    if kind == "decode" and case["codec"]:
        return {"case": case, "blob": zlib.compress(data, 6)}
    code = aqmp.aqmp_code_from_bitstream(data)
    if kind == "decode":
        return {"case": case, "code": code, "out": torch.empty((case["channels"], case["h"], case["w"]), device=DEV)}
    return {"case": case, "code": code, "alpha": torch.from_numpy(alpha).to(DEV),
            "refs": list(enumerate(_refs(case, seed)))}


# ------------------------------------------------------------------ one pass

def run(state):
    case = state["case"]
    if case["kind"] == "encode":
        images, params = state["images"], state["params"]
        if case["sweep"]:
            code = aqmp.aqmp_encode_planes([images[0][0]] * case["images"], [2.0 ** i for i in range(case["images"])],
                                           params, omp=case["omp"])
        elif len(images) > 1 and not case["host"]:
            code = aqmp.aqmp_encode_batch(images, params)
        else:
            code = aqmp.aqmp_encode_planes([p for im in images for p in im], None, params, omp=case["omp"])
        stats = code.stats()
        if stats["n_leaves"] > len(state["records"][0]) or stats["n_atoms"] > len(state["records"][1]):
            state["records"] = _records(case, stats["n_leaves"], stats["n_atoms"])
        leaves, atoms, lo = state["records"]
        rc = aqmp.load_library().aqmp_code_copy(code.handle, leaves.data_ptr(), atoms.data_ptr(), lo.data_ptr())
        code.free()
        if rc != aqmp.AQMP_OK:
            raise RuntimeError("aqmp_code_copy: %d" % rc)
        return {"leaves": leaves, "j": atoms[:, 0], "alpha": atoms.view(torch.float32)[:, 1],
                "alpha_lo": lo.view(torch.float32)}
    if case["kind"] == "correlate":
        c = aqmp.aqmp_correlate(case["b"], case["dict"], state["blocks"])
        return {"hi": c[..., 0], "lo": c[..., 1]}
    if case["kind"] == "decode":
        if case["codec"]:
            return aqmp.decompress(state["blob"])
        for c in range(case["channels"]):
            state["code"].decode(c, state["out"][c])
        return state["out"]
    alpha = state["alpha"].detach().requires_grad_(True)
    s = refine.synthesis_ssim(alpha, state["code"], state["refs"])
    (-s).backward()
    return {"ssim": s.detach(), "grad": alpha.grad}


def work(case):
    if case["kind"] == "correlate":
        b, n, fam = case["b"], case["blocks"], 2 if case["dict"] == 0 else 1
        return {"bytes": n * b * b * (1 + 8 * fam), "flops": 4.0 * fam * n * b ** 3}
    px = float(case["channels"] * case["h"] * case["w"])
    if case["kind"] == "encode":
        px = sum(float(h * w) for h, w in _sizes(case)) * case["channels"]
        tols = [2.0 ** i for i in range(case["images"])] if case["sweep"] else [case["tol"]]
        atoms = sum(ATOMS[case["scene"], t] for t in tols) / len(tols) * px
        # pixels in, atoms (and low words) out; the separable products at the roots, and for each emitted atom
        # one update of the other family's correlations at the smallest side it may come from
        read = px / (len(tols) if case["sweep"] else 1)
        return {"bytes": read + 12 * atoms,
                "flops": 8.0 * px * case["max_block"] + 2.0 * atoms * case["min_block"] ** 2}
    atoms = 0.06 * px                                                  # _code_arrays' mean
    if case["kind"] == "decode":
        return {"bytes": 8 * atoms + (1 if case["codec"] else 4) * px, "flops": 4.0 * px * case["min_block"]}
    # the synthesis, the window sums (five fields forward, three back, 11 + 11 taps), the adjoint's products
    return {"bytes": 4 * px + 12 * atoms, "flops": px * (2.0 * 22 * 8 + 8.0 * case["min_block"])}


# ------------------------------------------------------------------ in 64 bits

def _bases(b):
    k, m = torch.arange(b, dtype=torch.float64)[:, None], torch.arange(b, dtype=torch.float64)[None]
    dct = math.sqrt(2.0 / b) * torch.cos(math.pi * (2 * m + 1) * k / (2 * b))
    dct[0] = math.sqrt(1.0 / b)
    haar = torch.zeros((b, b), dtype=torch.float64)
    haar[0] = math.sqrt(1.0 / b)
    for r in range(1, b):
        s = 1 << (r.bit_length() - 1)
        n, t = b // s, r - s
        haar[r, t * n:t * n + n // 2] = math.sqrt(s / b)
        haar[r, t * n + n // 2:(t + 1) * n] = -math.sqrt(s / b)
    return [dct.to(DEV), haar.to(DEV)]


def _synthesis(case, seed):
    """A function of the coefficients (FP64, on the GPU): the planes they stand for."""
    planes, at, sides, j, alpha = _code_arrays(case, seed)
    first = np.concatenate([[0], np.cumsum([len(p[1]) for p in planes])])
    where = np.concatenate([np.concatenate([np.full((len(p[0]), 1), i), p[0][:, :2]], 1)
                            for i, p in enumerate(planes)])
    jt, plan = torch.from_numpy(j).to(DEV), []
    assert first[-1] == len(sides)
    for b in np.unique(sides):
        b = int(b)
        ids = np.flatnonzero(sides == b)
        slot = np.full(len(sides), -1)
        slot[ids] = np.arange(len(ids))
        pick = np.flatnonzero(slot[at] >= 0)
        grid = torch.arange(b, device=DEV)
        pyx = torch.from_numpy(where[ids]).to(DEV)
        index = ((pyx[:, 0, None, None] * case["h"] + pyx[:, 1, None, None] + grid[:, None]) * case["w"]
                 + pyx[:, 2, None, None] + grid)
        pick_t = torch.from_numpy(pick).to(DEV)
        plan.append((b, len(ids), pick_t, torch.from_numpy(slot[at[pick]]).to(DEV) * 2 * b * b + jt[pick_t], index))

    def synth(a):
        out = torch.zeros(case["channels"] * case["h"] * case["w"], dtype=torch.float64, device=DEV)
        for b, n, pick_t, to, index in plan:
            x = torch.zeros(n * 2 * b * b, dtype=torch.float64, device=DEV).index_add(0, to, a[pick_t])
            x = x.reshape(n, 2, b, b)                                  # [leaf][family][q][p]
            y = sum(m.T @ x[:, f].transpose(1, 2) @ m for f, m in enumerate(_bases(b)))   # rows by p, columns by q
            out = out.index_put((index.reshape(-1),), y.reshape(-1))
        return out.reshape(case["channels"], case["h"], case["w"])

    return synth, torch.from_numpy(alpha.astype(np.float64)).to(DEV)


def _mean_ssim(x, y):
    g = torch.exp(-(torch.arange(11, dtype=torch.float64, device=DEV) - 5) ** 2 / (2 * 1.5 ** 2))
    g = g / g.sum()

    def window(v):
        h, w = v.shape
        v = sum(g[i] * v[i:h - 10 + i] for i in range(11))
        return sum(g[i] * v[:, i:w - 10 + i] for i in range(11))

    c1, c2 = (0.01 * 255) ** 2, (0.03 * 255) ** 2
    mx, my = window(x), window(y)
    xx, yy, xy = window(x * x) - mx * mx, window(y * y) - my * my, window(x * y) - mx * my
    return ((2 * mx * my + c1) * (2 * xy + c2) / ((mx * mx + my * my + c1) * (xx + yy + c2))).mean()


def exact(case, seed):
    if case["kind"] == "correlate":
        b = case["b"]
        y = prepare(case, seed)["blocks"].double()
        fam = [m for f, m in enumerate(_bases(b)) if case["dict"] in (0, f + 1)]
        # c[q b + p] = sum_i,m B[p][i] y[i][m] B[q][m]
        c = torch.stack([(m @ y @ m.T).transpose(1, 2).reshape(len(y), b * b) for m in fam], 1)
        return {"hi": c.reshape(len(y), -1), "lo": None}
    if case["kind"] == "decode":
        if case["codec"]:
            return None                                                # bytes
        synth, a = _synthesis(case, seed)
        return synth(a)
    if case["kind"] == "refine":
        synth, a = _synthesis(case, seed)
        a.requires_grad_(True)
        y = synth(a)
        s = torch.stack([_mean_ssim(x.double(), y[c]) for c, x in enumerate(_refs(case, seed))]).mean()
        (-s).backward()
        return {"ssim": s.detach(), "grad": a.grad}
    return None                                                        # a pursuit: decisions, not a formula
