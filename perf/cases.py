"""Performance cases of the framework: the calls its users make, over the sizes they make them at.

``listed()`` names twelve cases, ``draw(rng)`` gives more of the same ranges.  A case is a dict of
plain values; ``prepare`` builds the inputs and handles a user's program holds before the call,
``run`` is one pass through the public entry points, ``work`` counts the bytes and operations the
pass cannot do without, and ``exact`` evaluates the same outputs in float64 with plain torch.

Inputs follow the recipe of the synthetic workloads: atoms uniform in a ball, images composed from
a true orientation, defocus, B-factor, displacement, scale and offset with white noise at SNR 0.1,
grids of uniform orientations x evenly spaced defocus values x {0, 50} A^2.
"""
import math

import numpy as np
import torch

import paper_1609_06634_gb300 as bioem

SIGMA_A = 1.5
SNR = 0.1
FOV_A = 140.8          # field of view of the 64 .. 192 px images
QBINS, DBINS = 4608, 4  # the proposal network's coarse orientation cells and defocus bins
CHANNELS, DOWN, MAX_BATCH = 32, 2, 256
STRIDES = (1, 2, 1, 2, 1, 2)
MAX_SHIFT = {32: 4, 64: 8, 96: 12, 128: 16, 192: 24}


def listed():
    return [
        # the smallest call: 16 images of 32 px against 6912 parameter sets, every output asked for
        {"name": "score_all_32px", "kind": "score", "npix": 32, "n_atoms": 500, "n_img": 16, "nq": 1152, "n_defocus": 3,
         "n_b": 2, "shift": 4, "mode": "fp32", "out": "all"},
        # small images, narrow window, the default arithmetic
        {"name": "score_64px_s4", "kind": "score", "npix": 64, "n_atoms": 5000, "n_img": 64, "nq": 1152, "n_defocus": 3,
         "n_b": 2, "shift": 4, "mode": "fp32", "out": "logP"},
        # odd counts at a size that is no power of two, per-pair outputs
        {"name": "pairs_96px_s12_ragged", "kind": "score", "npix": 96, "n_atoms": 1777, "n_img": 37, "nq": 331,
         "n_defocus": 3, "n_b": 1, "shift": 12, "mode": "fp32", "out": "pairs"},
        # centred particles: 128 px, narrow window, the default arithmetic and the tensor-core form
        {"name": "score_128px_s4", "kind": "score", "npix": 128, "n_atoms": 5000, "n_img": 64, "nq": 1152, "n_defocus": 3,
         "n_b": 2, "shift": 4, "mode": "fp32", "out": "logP"},
        {"name": "score_128px_s4_bf16x2", "kind": "score", "npix": 128, "n_atoms": 5000, "n_img": 64, "nq": 1152,
         "n_defocus": 3, "n_b": 2, "shift": 4, "mode": "bf16x2", "out": "logP"},
        # the throughput workload's scoring (fewer images and orientations, the same work per pair)
        {"name": "score_128px_s16_large", "kind": "score", "npix": 128, "n_atoms": 5000, "n_img": 512, "nq": 1152,
         "n_defocus": 4, "n_b": 2, "shift": 16, "mode": "fp32", "out": "logP"},
        # a new model for images at hand: prepare, project and score in one step
        {"name": "step_128px_new_model", "kind": "step", "npix": 128, "n_atoms": 5000, "n_img": 64, "nq": 576,
         "n_defocus": 4, "n_b": 2, "shift": 16},
        # synthetic maps, as training images are composed from
        {"name": "maps_128px", "kind": "maps", "npix": 128, "n_atoms": 5000, "n": 1024},
        # several models against stacks of four image sizes, one graph replay
        {"name": "batch_4x4", "kind": "batch", "n_models": 4, "n64": 32, "n96": 32, "n128": 32, "n192": 16, "nq": 576,
         "n_defocus": 2, "n_b": 2},
        # one wave of a re-ranking: project a few cells, score every image's own list, sum per bin
        {"name": "rerank_wave_128px", "kind": "gathered", "npix": 128, "n_atoms": 5000, "n_img": 1024, "cells": 16,
         "kids": 8, "fraction": 0.22, "shift": 16},
        # the proposal network: a training batch's loss and gradients, and the long proposals of a
        # re-ranking (the short ones, k = 32, are among the drawn cases)
        {"name": "network_gradients_b256", "kind": "gradients", "batch": 256},
        {"name": "propose_4096_bins", "kind": "propose", "n": 256, "k": 4096},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    largest = _pair_flops(128, 16) * 512 * 9216
    kind = rng.choice(["score", "score", "score", "score", "step", "maps", "batch", "gathered", "gradients", "propose"])
    npix = rng.choice([32, 64, 96, 128, 128, 192])
    atoms = _log_int(rng, 500, 5000) if npix > 32 else 500   # a 32 px box holds a small model
    if kind in ("score", "step"):
        shift = rng.choice([MAX_SHIFT[npix], rng.randint(0, MAX_SHIFT[npix]), min(4, MAX_SHIFT[npix])])
        n_defocus, n_b = rng.randint(1, 4), rng.randint(1, 2)
        n_img = _log_int(rng, 1, 512)
        nq = _log_int(rng, 36, 1152)
        while _pair_flops(npix, shift) * n_img * nq * n_defocus * n_b > 0.9 * largest:
            n_img = max(1, n_img // 2)
        c = {"kind": kind, "npix": npix, "n_atoms": atoms, "n_img": n_img, "nq": nq, "n_defocus": n_defocus, "n_b": n_b,
             "shift": shift}
        if kind == "score":
            narrow = shift <= 4 and rng.random() < 0.25
            c["mode"] = rng.choice(["bf16x2", "fp16x2", "bf16x2_real"]) if narrow else "fp32"
            c["out"] = rng.choice(["logP", "logP", "all", "pairs"])
        return c
    if kind == "maps":
        return {"kind": "maps", "npix": npix, "n_atoms": 2 * atoms, "n": _log_int(rng, 16, 1024)}
    if kind == "batch":
        return {"kind": "batch", "n_models": rng.randint(2, 6), "n64": rng.randint(1, 48), "n96": rng.randint(1, 48),
                "n128": rng.randint(1, 48), "n192": rng.randint(1, 24), "nq": _log_int(rng, 72, 576),
                "n_defocus": rng.randint(1, 2), "n_b": 2}
    if kind == "gathered":
        npix = rng.choice([64, 128, 128])
        return {"kind": "gathered", "npix": npix, "n_atoms": atoms, "n_img": _log_int(rng, 64, 2000),
                "cells": rng.choice([16, 32, 64]), "kids": rng.choice([1, 8]), "fraction": rng.uniform(0.05, 0.45),
                "shift": MAX_SHIFT[npix]}
    if kind == "gradients":
        return {"kind": "gradients", "batch": rng.randint(16, 255)}
    k = rng.choice([32, _log_int(rng, 1, 8192), _log_int(rng, 256, 8192)])
    return {"kind": "propose", "n": _log_int(rng, 16, 1024 if k <= 256 else 256), "k": k}


# ---------------------------------------------------------------------------------------- inputs
def _dev():
    return torch.device("cuda", 0)


def _rng(case, seed):
    return np.random.Generator(np.random.PCG64(np.random.SeedSequence(int(seed), spawn_key=(1609, len(case)))))


def _pixel(npix):
    return 2.0 if npix == 32 else FOV_A / npix


def _atoms(rng, n):
    g = rng.standard_normal((n, 3))
    g /= np.linalg.norm(g, axis=1, keepdims=True)
    radius = min(40.0 * (n / 500.0) ** (1.0 / 3.0), 80.0) if n <= 5000 else 80.0 * (n / 5000.0) ** (1.0 / 3.0)
    out = np.empty((n, 4), dtype=np.float32)
    out[:, :3] = g * (radius * rng.random(n) ** (1.0 / 3.0))[:, None]
    out[:, 3] = 1.0
    return torch.from_numpy(out).to(_dev())


def _quats(rng, n):
    q = rng.standard_normal((n, 4))
    return torch.from_numpy((q / np.linalg.norm(q, axis=1, keepdims=True)).astype(np.float32)).to(_dev())


def _ctf_rows(n_defocus, n_b):
    dv = np.linspace(0.5e4, 2.5e4, n_defocus) if n_defocus > 1 else np.array([1.5e4])
    return [(float(d), 0.1, b, 300.0) for d in dv for b in (0.0, 50.0)[:n_b]]


def _random_ctfs(rng, n):
    return [(float(d), 0.1, float(b), 300.0) for d, b in zip(rng.uniform(0.5e4, 2.5e4, n), rng.uniform(0.0, 50.0, n))]


def _project64(atoms, quats, npix, pixel):
    """Float64 projections [n, N, N] of Gaussian atoms integrated over pixels (rows y, columns x)."""
    a, q = atoms.double(), quats.double()
    q = q / q.norm(dim=1, keepdim=True)
    w, x, y, z = q.unbind(1)
    rx = torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y)], 1)
    ry = torch.stack([2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x)], 1)
    edge = (torch.arange(npix + 1, device=a.device, dtype=torch.float64) - npix / 2 - 0.5) * pixel
    out = torch.empty((len(q), npix, npix), dtype=torch.float64, device=a.device)
    step = max(1, 40_000_000 // (len(a) * (npix + 1)))
    for i in range(0, len(q), step):
        ex = torch.erf((edge - (rx[i:i + step] @ a[:, :3].T)[..., None]) / (SIGMA_A * math.sqrt(2.0)))
        ey = torch.erf((edge - (ry[i:i + step] @ a[:, :3].T)[..., None]) / (SIGMA_A * math.sqrt(2.0)))
        gx = 0.5 * (ex[..., 1:] - ex[..., :-1])
        gy = 0.5 * (ey[..., 1:] - ey[..., :-1]) * a[:, 3, None]
        out[i:i + step] = torch.matmul(gy.transpose(1, 2), gx)
    return out


def _ctf64(row, npix, pixel):
    """CTF x envelope on the half spectrum [N, N/2 + 1] of one (defocus, contrast, B, voltage) row."""
    d, amp, b, kv = row
    v = kv * 1.0e3
    lam = 12.2643 / math.sqrt(v * (1.0 + 0.97845e-6 * v))
    fy = torch.fft.fftfreq(npix, pixel, dtype=torch.float64, device=_dev())[:, None]
    fx = torch.fft.rfftfreq(npix, pixel, dtype=torch.float64, device=_dev())[None, :]
    k2 = fx * fx + fy * fy
    phase = math.pi * lam * d * k2
    return (-amp * torch.cos(phase) - math.sqrt(1.0 - amp * amp) * torch.sin(phase)) * torch.exp(-0.25 * b * k2)


def _images(rng, atoms, n, npix, pixel, shift):
    """[n, N, N] float32 images of the model at random orientations, displacements and PSFs, with noise."""
    img = torch.empty((n, npix, npix), dtype=torch.float32, device=_dev())
    quats, ctfs = _quats(rng, n), _random_ctfs(rng, n)
    dy, dx = rng.integers(-shift, shift + 1, n), rng.integers(-shift, shift + 1, n)
    norm, offset = rng.uniform(0.5, 2.0, n), rng.uniform(-1.0, 1.0, n)
    gen = torch.Generator(device=_dev())
    gen.manual_seed(int(rng.integers(1 << 62)))
    for i0 in range(0, n, 256):
        p = _project64(atoms, quats[i0:i0 + 256], npix, pixel)
        t = torch.stack([_ctf64(c, npix, pixel) for c in ctfs[i0:i0 + 256]])
        p = torch.fft.irfft2(torch.fft.rfft2(p) * t, s=(npix, npix))
        for i in range(len(p)):
            j = i0 + i
            img[j] = (float(norm[j]) * torch.roll(p[i], (-int(dy[j]), -int(dx[j])), (0, 1)) - float(offset[j])).float()
    lam = (img.double().var(dim=(1, 2), unbiased=False) / SNR).sqrt().float()
    return img + lam[:, None, None] * torch.randn(img.shape, generator=gen, device=_dev())


def _weights(rng):
    """Flat float32 parameters: uniform weights of variance 2 / fan-in (heads: 1 / fan-in), zero biases."""
    gen = torch.Generator(device=_dev())
    gen.manual_seed(int(rng.integers(1 << 62)))
    convs, feat = _net_sizes()
    parts = []
    for n_in, n_out, gain in [(9 * ci, co, 6.0) for ci, co, _ in convs] + [(feat, QBINS, 3.0), (feat, DBINS, 3.0)]:
        u = torch.rand(n_in * n_out, generator=gen, device=_dev())
        parts += [(2.0 * u - 1.0) * math.sqrt(gain / n_in), torch.zeros(n_out, device=_dev())]
    return torch.cat(parts)


_CTX = []


def _context():
    # a program keeps one context for all its calls
    if not _CTX:
        _CTX.append(bioem.Context(0))
    return _CTX[0]


def _lists(rng, case):
    """Per-image lists (CSR) of the wave's parameter sets: every image keeps a share of the wave's
    (cell, defocus) bins; a bin is its cell's child orientations x both B-factors."""
    n, cells, kids = case["n_img"], case["cells"], case["kids"]
    total = n * cells * 4
    kept = np.sort(rng.permutation(total)[:max(1, int(case["fraction"] * total))])
    img, b = kept // (cells * 4), kept % (cells * 4)
    head = (b // 4) * (kids * 8) + (b % 4) * 2
    tail = (np.arange(kids)[:, None] * 8 + np.arange(2)[None, :]).reshape(-1)
    off = np.zeros(n + 1, dtype=np.int64)
    np.cumsum(np.bincount(img, minlength=n) * (kids * 2), out=off[1:])
    return off.astype(np.int32), (head[:, None] + tail[None, :]).reshape(-1).astype(np.int32)


def _inputs(case, seed):
    """The pass's inputs as a dict of device tensors and host values."""
    rng = _rng(case, seed)
    kind = case["kind"]
    if kind == "batch":
        n_atoms = [int(round(math.exp(rng.uniform(math.log(500), math.log(20000))))) for _ in range(case["n_models"])]
        models = [_atoms(rng, n) for n in n_atoms]
        stacks = []
        for npix in (64, 96, 128, 192):
            n, pixel = case["n%d" % npix], _pixel(npix)
            which = rng.integers(0, len(models), n)
            imgs = torch.cat([_images(rng, models[m], int((which == m).sum()), npix, pixel, npix // 8)
                              for m in range(len(models)) if (which == m).any()])
            stacks.append({"npix": npix, "pixel": pixel, "images": imgs, "quats": _quats(rng, case["nq"])})
        return {"models": models, "stacks": stacks, "ctfs": _ctf_rows(case["n_defocus"], case["n_b"])}
    if kind in ("gradients", "propose"):
        n = case["batch"] if kind == "gradients" else case["n"]
        imgs = _images(rng, _atoms(rng, 2000), n, 128, 1.1, 16)
        yq = torch.from_numpy(rng.integers(0, QBINS, n).astype(np.int32)).to(_dev())
        yd = torch.from_numpy(rng.integers(0, DBINS, n).astype(np.int32)).to(_dev())
        return {"images": imgs, "yq": yq, "yd": yd, "theta": _weights(rng)}
    npix, pixel = case["npix"], _pixel(case["npix"])
    atoms = _atoms(rng, case["n_atoms"])
    if kind == "maps":
        return {"atoms": atoms, "quats": _quats(rng, case["n"]), "ctfs": _random_ctfs(rng, case["n"]), "pixel": pixel}
    d = {"atoms": atoms, "pixel": pixel, "images": _images(rng, atoms, case["n_img"], npix, pixel, case["shift"])}
    if kind == "gathered":
        off, idx = _lists(rng, case)
        d.update(quats=_quats(rng, case["cells"] * case["kids"]), ctfs=_ctf_rows(4, 2),
                 off=torch.from_numpy(off).to(_dev()), idx=torch.from_numpy(idx).to(_dev()),
                 most=max(1, int(np.diff(off).max())))
    else:
        d.update(quats=_quats(rng, case["nq"]), ctfs=_ctf_rows(case["n_defocus"], case["n_b"]))
    return d


# ---------------------------------------------------------------------------------------- passes
def prepare(case, seed):
    ctx = _context()
    s = {"case": case, "ctx": ctx, "in": _inputs(case, seed)}
    d, kind = s["in"], case["kind"]
    if kind == "score":
        s["images"] = bioem.prepare_images(ctx, d["images"], d["pixel"])
        s["projset"] = bioem.project_model(ctx, d["atoms"], SIGMA_A, d["quats"], d["ctfs"], case["npix"], d["pixel"])
    elif kind == "gathered":
        s["images"] = bioem.prepare_images(ctx, d["images"], d["pixel"])
    elif kind == "batch":
        s["stacks"] = [bioem.prepare_images(ctx, st["images"], st["pixel"]) for st in d["stacks"]]
        s["projsets"] = [[bioem.project_model(ctx, a, SIGMA_A, st["quats"], d["ctfs"], st["npix"], st["pixel"])
                          for st in d["stacks"]] for a in d["models"]]
        s["batch"] = bioem.Batch(ctx, s["stacks"], s["projsets"], [st["npix"] // 8 for st in d["stacks"]])
    elif kind in ("gradients", "propose"):
        s["net"] = bioem.CNN(ctx, 128, DOWN, CHANNELS, QBINS, DBINS, MAX_BATCH)
        s["net"].set_params(d["theta"])
    return s


def run(state):
    case, ctx, d = state["case"], state["ctx"], state["in"]
    kind = case["kind"]
    if kind == "score":
        im, ps, shift = state["images"], state["projset"], case["shift"]
        ctx.set_precision(case["mode"])
        if case["out"] == "all":
            out = bioem.score_all(ctx, im, ps, shift, per_orient=True, best=True)
        elif case["out"] == "pairs":
            out = bioem.score_pairs(ctx, im, ps, shift)
        else:
            out = bioem.score(ctx, im, ps, shift)
        ctx.set_precision("fp32")
        return out
    if kind == "step":
        im = bioem.prepare_images(ctx, d["images"], d["pixel"])
        ps = bioem.project_model(ctx, d["atoms"], SIGMA_A, d["quats"], d["ctfs"], case["npix"], d["pixel"])
        out = bioem.score_all(ctx, im, ps, case["shift"], best=True)
        ps.close()
        im.close()
        return out
    if kind == "maps":
        return bioem.synthetic_maps(ctx, d["atoms"], SIGMA_A, d["quats"], d["ctfs"], case["npix"], d["pixel"])
    if kind == "batch":
        return state["batch"].run()
    if kind == "gathered":
        ps = bioem.project_model(ctx, d["atoms"], SIGMA_A, d["quats"], d["ctfs"], case["npix"], d["pixel"])
        v = bioem.score_gathered_pairs(ctx, state["images"], ps, case["shift"], d["off"], d["idx"], d["most"])
        g = bioem.group_logsumexp(ctx, v, case["kids"] * 2)
        ps.close()
        return {"pairs": v, "bins": g}
    if kind == "gradients":
        grads, loss = state["net"].gradients(d["images"], d["yq"], d["yd"])
        return {"grads": grads, "loss": loss}
    bins, scores = state["net"].propose(d["images"], case["k"])
    return {"bins": bins, "scores": scores}


# ---------------------------------------------------------------------------------------- work
def _pair_flops(npix, shift):
    """One image against one parameter set: the Fourier product, then a real inverse transform of the
    whole map or the wanted displacements alone, whichever is less, and the closed form."""
    half, n, S = npix * (npix // 2 + 1), npix * npix, (2 * shift + 1) ** 2
    return min(6 * half + 2.5 * n * math.log2(n), 4 * half * S) + 4 * S


def _spec_bytes(npix):
    return npix * (npix // 2 + 1) * 8


def _project_flops(npix, atoms, nq):
    # both axes' pixel integrals where they are not zero (about +-7 sigma) and their outer products
    reach = min(npix, int(14 * SIGMA_A / _pixel(npix)) + 2)
    return nq * atoms * (2.0 * reach * reach + 40.0 * reach) + nq * 2.5 * npix * npix * math.log2(npix * npix)


def _net_sizes():
    s, cin, convs = 128 // DOWN, 1, []
    for st in STRIDES:
        s //= st
        convs.append((cin, CHANNELS, s))
        cin = CHANNELS
    return convs, CHANNELS * s * s


def _net_params():
    convs, feat = _net_sizes()
    return sum(ci * co * 9 + co for ci, co, _ in convs) + (QBINS + DBINS) * (feat + 1)


def work(case):
    kind = case["kind"]
    if kind == "batch":
        b = f = 0.0
        n_ps = case["nq"] * case["n_defocus"] * case["n_b"]
        for npix in (64, 96, 128, 192):
            n = case["n%d" % npix]
            b += _spec_bytes(npix) * (n + case["n_models"] * n_ps) + 4 * n * case["n_models"]
            f += _pair_flops(npix, npix // 8) * n * n_ps * case["n_models"]
        return {"bytes": b, "flops": f}
    if kind in ("gradients", "propose"):
        n = case["batch"] if kind == "gradients" else case["n"]
        convs, feat = _net_sizes()
        fwd = n * (sum(2.0 * 9 * ci * co * s * s for ci, co, s in convs) + 2.0 * (QBINS + DBINS) * feat)
        b = n * 128 * 128 * 4 + _net_params() * 2
        if kind == "gradients":
            return {"bytes": b + _net_params() * 4, "flops": 3 * fwd}
        return {"bytes": b + n * case["k"] * 8, "flops": fwd + 2.0 * n * QBINS * DBINS}
    npix = case["npix"]
    if kind == "maps":
        n = case["n"]
        return {"bytes": n * npix * npix * 4.0,
                "flops": _project_flops(npix, case["n_atoms"], n) + n * 2.5 * npix * npix * math.log2(npix * npix)}
    n_img, shift = case["n_img"], case["shift"]
    if kind == "gathered":
        n_ps = case["cells"] * case["kids"] * 8
        pairs = n_img * case["cells"] * 4 * case["fraction"] * case["kids"] * 2
        return {"bytes": _spec_bytes(npix) * n_img + pairs * 12 + case["n_atoms"] * 16,
                "flops": pairs * _pair_flops(npix, shift) + _project_flops(npix, case["n_atoms"], n_ps // 8)}
    n_ps = case["nq"] * case["n_defocus"] * case["n_b"]
    f = n_img * n_ps * _pair_flops(npix, shift)
    if kind == "step":
        f += _project_flops(npix, case["n_atoms"], case["nq"]) + n_img * 2.5 * npix * npix * math.log2(npix * npix)
        return {"bytes": n_img * (npix * npix * 4.0 + 32) + case["nq"] * 16 + case["n_atoms"] * 16, "flops": f}
    b = _spec_bytes(npix) * (n_img + n_ps) + 8.0 * n_img
    if case["out"] == "all":
        b += n_img * (24 + 8 * case["nq"])
    elif case["out"] == "pairs":
        b += 16.0 * n_img * n_ps
    return {"bytes": b, "flops": f}


# ---------------------------------------------------------------------------------------- float64
def _unit64(spec, npix):
    """(unit-norm spectra with the mean removed, n x the sum of squared deviations) of [n, N, N/2 + 1]."""
    spec = spec.clone()
    spec[:, 0, 0] = 0.0
    w = torch.full((npix // 2 + 1,), 2.0, dtype=torch.float64, device=spec.device)
    w[0] = w[-1] = 1.0
    e = (spec.abs().square() * w).sum((1, 2))   # = n sum x^2 - (sum x)^2 by Parseval
    return spec / e.sqrt()[:, None, None], e


def _projset64(atoms, quats, ctfs, npix, pixel):
    """(unit-norm projection spectra [n_ps, N, N/2 + 1], -1/2 ln B) of the whole grid."""
    t = torch.stack([_ctf64(c, npix, pixel) for c in ctfs])
    specs, kb = [], []
    for i in range(0, len(quats), 64):
        f = torch.fft.rfft2(_project64(atoms, quats[i:i + 64], npix, pixel))
        u, e = _unit64((f[:, None] * t[None]).reshape(-1, npix, npix // 2 + 1), npix)
        specs.append(u)
        kb.append(-0.5 * e.log())
    return torch.cat(specs), torch.cat(kb)


def _imageset64(images, npix):
    n = npix * npix
    u, a = _unit64(torch.fft.rfft2(images.double()), npix)
    c = (-math.log(2.0) + (1.0 - n / 2.0) * math.log(2.0 * math.pi) + math.lgamma((n - 3) / 2.0)
         + (n - 3) / 2.0 * math.log(2.0 * n))
    return u, 0.5 * (3.0 - n) * a.log() + c


def _pairs64(img, proj, npix, shift):
    """ln(1 - rho^2) of one image spectrum against proj [p, N, N/2 + 1] at every displacement: [p, S]."""
    rows = [d % npix for d in range(-shift, shift + 1)]
    out = []
    step = max(1, 60_000_000 // (npix * npix))
    for i in range(0, len(proj), step):
        col = torch.fft.ifft(img.conj() * proj[i:i + step], dim=1)[:, rows]
        rho = torch.fft.irfft(col, n=npix, dim=2)[:, :, rows] * (npix * npix)
        out.append(torch.log1p(-rho.square()).flatten(1))
    return torch.cat(out)


def _score64(images, spec, kb, npix, shift, nctf, want):
    n, S, n_ps = npix * npix, (2 * shift + 1) ** 2, len(spec)
    u, ka = _imageset64(images, npix)
    logp, orient, best, pmax, plse = [], [], [], [], []
    for w in range(len(images)):
        ll = ka[w] + kb[:, None] + 0.5 * (3.0 - n) * _pairs64(u[w], spec, npix, shift)
        logp.append(torch.logsumexp(ll.flatten(), 0) - math.log(n_ps * S))
        if want == "all":
            orient.append(torch.logsumexp(ll.reshape(n_ps // nctf, -1), 1) - math.log(nctf * S))
        if want in ("all", "best"):
            best.append(ll.max())
        if want == "pairs":
            pmax.append(ll.max(1).values)
            plse.append(torch.logsumexp(ll, 1))
    if want == "pairs":
        return torch.stack(pmax), torch.stack(plse)
    if want == "logP":
        return torch.stack(logp)
    out = {"logP": torch.stack(logp), "best_logL": torch.stack(best)}
    out.update({k: None for k in ("best_q", "best_ctf", "best_dx", "best_dy")})
    if want == "all":
        out["logP_orient"] = torch.stack(orient)
    return out


def _net64(theta, images):
    """Float64 logits of the network whose float16 weights are theta's, and the tensors they came from."""
    x = torch.nn.functional.avg_pool2d(images.double()[:, None], DOWN)
    x = (x - x.mean((1, 2, 3), keepdim=True)) / x.var((1, 2, 3), unbiased=False, keepdim=True).sqrt()
    convs, feat = _net_sizes()
    at = 0

    def take(*shape):
        nonlocal at
        n = math.prod(shape)
        at += n
        return theta[at - n:at].reshape(shape)

    for (ci, co, _), st in zip(convs, STRIDES):
        x = torch.relu(torch.nn.functional.conv2d(x, take(co, ci, 3, 3), take(co), stride=st, padding=1))
    x = x.flatten(1)
    lq = x @ take(QBINS, feat).T + take(QBINS)
    return lq, x @ take(DBINS, feat).T + take(DBINS)


def exact(case, seed):
    kind = case["kind"]
    d = _inputs(case, seed)
    if kind in ("gradients", "propose"):
        theta = d["theta"].half().double().requires_grad_(kind == "gradients")
        if kind == "gradients":
            lq, ld = _net64(theta, d["images"])
            loss = torch.nn.functional.cross_entropy(lq, d["yq"].long(), reduction="none") + \
                torch.nn.functional.cross_entropy(ld, d["yd"].long(), reduction="none")
            loss.mean().backward()
            return {"grads": theta.grad, "loss": loss.detach()}
        lq, ld = _net64(theta, d["images"])
        joint = (torch.log_softmax(lq, 1)[:, :, None] + torch.log_softmax(ld, 1)[:, None, :]).flatten(1)
        return {"bins": None, "scores": torch.sort(joint, dim=1, descending=True).values[:, :case["k"]].contiguous()}
    if kind == "batch":
        rows = []
        for a in d["models"]:
            cols = []
            for st in d["stacks"]:
                spec, kb = _projset64(a, st["quats"], d["ctfs"], st["npix"], st["pixel"])
                cols.append(_score64(st["images"], spec, kb, st["npix"], st["npix"] // 8, len(d["ctfs"]), "logP"))
            rows.append(torch.cat(cols))
        return torch.stack(rows)
    npix = case["npix"]
    if kind == "maps":
        f = torch.fft.rfft2(_project64(d["atoms"], d["quats"], npix, d["pixel"]))
        return torch.fft.irfft2(f * torch.stack([_ctf64(c, npix, d["pixel"]) for c in d["ctfs"]]), s=(npix, npix))
    spec, kb = _projset64(d["atoms"], d["quats"], d["ctfs"], npix, d["pixel"])
    if kind == "gathered":
        n, off = npix * npix, d["off"].tolist()
        u, ka = _imageset64(d["images"], npix)
        v = []
        for w in range(len(d["images"])):
            idx = d["idx"][off[w]:off[w + 1]].long()
            if len(idx):
                ll = 0.5 * (3.0 - n) * _pairs64(u[w], spec[idx], npix, case["shift"])
                v.append(ka[w] + kb[idx] + torch.logsumexp(ll, 1))
        v = torch.cat(v)
        return {"pairs": v, "bins": torch.logsumexp(v.reshape(-1, case["kids"] * 2), 1)}
    want = case["out"] if kind == "score" else "best"
    return _score64(d["images"], spec, kb, npix, case["shift"], len(d["ctfs"]), want)
