"""The calls that a user of this library makes, over the sizes that it is used at.

A case is one of five calls of the public binding (`paper_1411_6206_gb300.lps`):

- "dc"      one data-consistency update X = Z - E^H(E Z - d) with its residual: step (4) of every
            iteration, and the call of a caller that runs its own outer loop;
- "encode"  the acquisition operator both ways, E x and E^H d: simulating samples from an image
            and the zero-filled start of a reconstruction;
- "svt"     the two contractions of the singular-value step, the Casorati Gram and the
            reprojection, for a caller that thresholds the singular values itself;
- "frame"   one time instance as a session runs it: the frame's new mask and samples, then the
            reconstruction;
- "batch"   one frame step of several independent problems of uneven size.

Sizes are those of the benchmark workloads (32x32x8 with one coil, the 128x128x16 cardiac
sequence with 8 coils, the 192x192x32 precision study with 12 coils, the uneven mix) and, for
drawn cases, anything between: in-plane multiples of 8, any slice count up to 32, 1 to 16 coils,
undersampling 2 to 12, 3D and per-slice encode, float32 and binary16 maps and samples, float32,
TF32 and BF16 contractions. Frames run few iterations here: every iteration costs the same, and
after many the float32 rounding of the first has travelled through all that follow.
"""
import math

import numpy as np
import torch

from paper_1411_6206_gb300 import lps
from paper_1411_6206_gb300 import phantom
from paper_1411_6206_gb300 import phantom_gpu

NOISE = 1e-3
PRECISIONS = {"fp32": lps.FP32, "tf32": lps.TF32_REFINE, "bf16": lps.BF16_REFINE}


def _case(name, kind, nx, ny, nz, ncoil, accel, fft_z=1, half=0, precision="fp32", iters=0, prior=0):
    return {"name": name, "kind": kind, "nx": nx, "ny": ny, "nz": nz, "ncoil": ncoil, "accel": accel,
            "fft_z": fft_z, "half": half, "precision": precision, "iters": iters, "prior": prior}


def listed():
    return [
        # the smallest workload of the benchmark (one coil, a quarter of the lines): latency
        _case("dc_small", "dc", 32, 32, 8, 1, 4.0),
        # the cardiac sequence's update, in float32 and with binary16 maps and samples
        _case("dc_cardiac", "dc", 128, 128, 16, 8, 8.0),
        _case("dc_cardiac_half", "dc", 128, 128, 16, 8, 8.0, half=2),
        # the precision study's update: the largest plane that the library takes
        _case("dc_large", "dc", 192, 192, 32, 12, 10.0),
        # a volume as a scanner gives it: ragged in-plane size, odd slice count
        _case("dc_ragged", "dc", 120, 104, 15, 6, 5.0),
        # a large member of the uneven mix, both directions of the acquisition operator
        _case("encode_mix", "encode", 160, 160, 24, 14, 6.0),
        # the singular-value contractions of the precision study, on FMA and on the tensor cores
        _case("svt_fp32", "svt", 192, 192, 32, 1, 10.0),
        _case("svt_bf16", "svt", 192, 192, 32, 1, 10.0, precision="bf16"),
        # whole frames: the smallest workload's first frame, a later frame of the cardiac sequence
        # (prior support and singular values from the frame before), and the precision study's first
        _case("frame_small", "frame", 32, 32, 8, 1, 4.0, iters=10),
        _case("frame_cardiac", "frame", 128, 128, 16, 8, 8.0, iters=5, prior=1),
        _case("frame_large_bf16", "frame", 192, 192, 32, 12, 10.0, precision="bf16", iters=5),
        # one frame step of a batch of uneven problems (sizes of the batched study)
        {"name": "batch_mix", "kind": "batch", "members": 8, "mix": 3, "iters": 10},
    ]


LARGEST = 192 * 192 * 32 * 12   # voxels times coils of the largest workload


def draw(rng):
    kind = rng.choice(["dc", "dc", "encode", "svt", "frame", "frame", "batch"])
    while kind == "batch":
        c = {"kind": "batch", "members": rng.randint(2, 8), "mix": rng.randint(10, 9999), "iters": rng.randint(3, 10)}
        if work(c)["flops"] <= work(listed()[-1])["flops"]:
            return c

    def size(lo, hi, step):
        return step * round(math.exp(rng.uniform(math.log(lo), math.log(hi))) / step)

    while True:
        nx, ny = size(32, 192, 8), size(32, 192, 8)
        if rng.random() < 0.5:
            ny = nx
        nz = rng.choice([8, 16, 32, rng.randint(3, 32), rng.randint(8, 31)])
        ncoil = rng.randint(1, 16)
        # a runtime-sized plane may cost several times what a benchmark plane of its size does
        if nx * ny * nz * ncoil <= LARGEST // 4:
            break
    precision = rng.choice(["fp32", "fp32", "tf32", "bf16"]) if kind in ("svt", "frame") else "fp32"
    # a few coils carry a few times fewer lines than the volume has
    accel = round(rng.uniform(2.0, min(12.0, 3.0 + ncoil)), 1)
    prior = rng.randint(0, 1) if kind == "frame" else 0
    c = _case("", kind, nx, ny, nz, ncoil, accel, fft_z=rng.choice([1, 1, 0]),
              half=rng.choice([0, 0, 1, 2]) if kind == "dc" else 0, precision=precision,
              iters=rng.randint(2, 3 if prior else 10) if kind == "frame" else 0, prior=prior)
    del c["name"]
    return c


def members(case):
    """The problems of a batch: sizes of the uneven mix."""
    rng = np.random.default_rng(case["mix"])
    out = []
    for _ in range(case["members"]):
        n = int(rng.choice(np.arange(64, 161, 16)))
        out.append(_case("", "frame", n, n, int(rng.choice([8, 10, 12, 14, 16, 20, 24, 28, 32])),
                         int(rng.integers(4, 17)), float(rng.integers(4, 13)), iters=case["iters"]))
    return out


# ---- inputs ---------------------------------------------------------------------------------

def _axes(case):
    return (-3, -2, -1) if case["fft_z"] else (-2, -1)


def _image(case, seed, t):
    w = phantom.Workload("case", case["nx"], case["ny"], case["nz"], case["ncoil"], 20, 1, 4.0, seed)
    return phantom_gpu.HeartFrames(w).frame(t)


def _mask(case, seed):
    ny, nz = case["ny"], case["nz"]
    return phantom.vd_mask(ny, nz, max(4, round(ny * nz / case["accel"])), min(4, nz), seed, case["fft_z"])


def _lines(mask):
    kz, ky = np.nonzero(mask)
    return torch.from_numpy(kz).cuda(), torch.from_numpy(ky).cuda()


def _encode(x, coils, mask, case):
    kz, ky = _lines(mask)
    k = torch.fft.fftn(coils * x, dim=_axes(case), norm="ortho")
    return k[:, kz, :, ky].permute(1, 0, 2).contiguous()   # [line][coil][kx] -> [coil][line][kx]


def _problem(case, seed):
    """Coil maps, mask, samples and the image behind them, all in float32."""
    coils = phantom_gpu.coil_maps(case["nx"], case["ny"], case["nz"], case["ncoil"], seed + 1)
    mask = _mask(case, seed + 2)
    x = _image(case, seed + 3, 1 + seed % 8)
    d = _encode(x, coils, mask, case)
    d = d + phantom_gpu.noise(d.shape[0], d.shape[1], d.shape[2], NOISE, seed + 4)
    return coils, mask, x, d.contiguous()


def _gaussian(shape, sigma, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.complex(torch.randn(shape, generator=g, device="cuda"),
                         torch.randn(shape, generator=g, device="cuda")) * sigma


def _svt_inputs(case, seed):
    """X, a sparse S and the thresholding matrix W = V diag(max(s - lambda, 0) / s) V^H."""
    shape = (case["nz"], case["nx"], case["ny"])
    X = _image(case, seed + 3, 1 + seed % 8) + _gaussian(shape, 0.02, seed + 5)
    g = torch.Generator(device="cuda").manual_seed(seed + 6)
    S = _gaussian(shape, 0.2, seed + 7) * (torch.rand(shape, generator=g, device="cuda") < 0.05)
    M = (X - S).to(torch.complex128).reshape(case["nz"], -1)
    lam, V = np.linalg.eigh((M.conj() @ M.T).cpu().numpy())
    s = np.sqrt(np.maximum(lam, 0.0))
    W = (V * (np.maximum(s - 0.01 * s.max(), 0.0) / np.maximum(s, 1e-30))) @ V.conj().T
    return X.contiguous(), S.contiguous(), torch.from_numpy(W.astype(np.complex64)).cuda()


def _prior(case, seed):
    """Support and singular values of the frame before: its image's wavelet support, and the
    thresholded singular values at the scale that undersampled lines leave them."""
    x = _image(case, seed + 3, seed % 8).to(torch.complex128)
    c = _haar(x)
    keep = c.abs() > 0.005 * c.abs().max()
    coils = phantom_gpu.coil_maps(case["nx"], case["ny"], case["nz"], case["ncoil"], seed + 1).to(torch.complex128)
    mask = _mask(case, seed + 50)
    M = _adjoint(_encode(x, coils, mask, case), coils, mask, case).reshape(case["nz"], -1)
    lam = np.linalg.eigvalsh((M.conj() @ M.T).cpu().numpy())[::-1]
    s = np.sqrt(np.maximum(lam, 0.0))
    return keep, np.maximum(s - 0.01 * s[0], 0.0)


def _support_words(keep):
    return np.packbits(keep.cpu().numpy().reshape(-1), bitorder="little").view(np.uint32)


def prepare(case, seed):
    if case["kind"] == "batch":
        probs = members(case)
        made = [_problem(c, seed + 100 * i) for i, c in enumerate(probs)]
        batch = lps.Batch([lps.params_init(nx=c["nx"], ny=c["ny"], nz=c["nz"], ncoil=c["ncoil"], max_iters=c["iters"])
                           for c in probs])
        for m, (coils, _, _, _) in zip(batch.members, made):
            m.set_coils(coils)
        return {"kind": "batch", "batch": batch, "masks": [p[1] for p in made], "d": [p[3] for p in made],
                "out": [torch.empty_like(p[2]) for p in made]}
    options = dict(fft_z=case["fft_z"], precision=PRECISIONS[case["precision"]], max_iters=max(1, case["iters"]),
                   coil_format=lps.COILS_FP16 if case["half"] >= 1 else lps.COILS_FP32,
                   data_format=lps.DATA_FP16 if case["half"] >= 2 else lps.DATA_FP32,
                   eig_precision=lps.EIG_FP32 if case["precision"] == "fp32" else lps.EIG_FP64)
    plan = lps.Plan(case["nx"], case["ny"], case["nz"], case["ncoil"], **options)
    state = {"kind": case["kind"], "plan": plan}
    shape = (case["nz"], case["nx"], case["ny"])
    new = lambda *s: torch.empty(s, dtype=torch.complex64, device="cuda")  # noqa: E731
    if case["kind"] == "svt":
        X, S, W = _svt_inputs(case, seed)
        return {**state, "X": X, "S": S, "W": W, "G": new(case["nz"], case["nz"]), "L": new(*shape)}
    coils, mask, x, d = _problem(case, seed)
    plan.set_coils(coils)
    plan.set_mask(mask)
    if case["kind"] == "dc":
        plan.set_data(d)
        return {**state, "Z": (x + _gaussian(shape, 0.05, seed + 8)).contiguous(), "X": new(*shape)}
    if case["kind"] == "encode":
        return {**state, "x": x, "d": d, "k": new(*d.shape), "image": new(*shape)}
    if case["prior"]:
        keep, sigma = _prior(case, seed)
        plan.set_prior(torch.from_numpy(_support_words(keep).view(np.int32)).cuda(), torch.from_numpy(sigma).cuda())
    return {**state, "mask": mask, "d": d, "recon": new(*shape)}


def run(state):
    kind = state["kind"]
    if kind == "batch":
        batch = state["batch"]
        for m, mask, d in zip(batch.members, state["masks"], state["d"]):
            m.set_mask(mask)
            m.set_data(d)
        batch.reconstruct()
        return [m.recon(out) for m, out in zip(batch.members, state["out"])]
    plan = state["plan"]
    if kind == "dc":
        resid = lps.data_consistency(plan.handle, state["Z"], state["X"])
        return {"X": state["X"], "resid": np.float32(resid)}   # a sum of float32 residuals
    if kind == "encode":
        lps.forward(plan.handle, state["x"], state["k"])
        lps.adjoint(plan.handle, state["d"], state["image"])
        return {"k": state["k"], "image": state["image"]}
    if kind == "svt":
        lps.casorati_gram(plan.handle, state["X"], state["S"], state["G"])
        lps.lowrank_reproject(plan.handle, state["X"], state["S"], state["W"], state["L"])
        return {"G": state["G"], "L": state["L"]}
    plan.set_mask(state["mask"])
    plan.set_data(state["d"])
    plan.reconstruct_frame(recon=state["recon"], stats=False)
    return state["recon"]


# ---- what a pass cannot do without ----------------------------------------------------------

def work(case):
    if case["kind"] == "batch":
        each = [work(c) for c in members(case)]
        return {"bytes": sum(w["bytes"] for w in each), "flops": sum(w["flops"] for w in each)}
    nx, ny, nz, nc = case["nx"], case["ny"], case["nz"], case["ncoil"]
    N = nx * ny * nz
    samples = nc * int(_mask(case, 1).sum()) * nx
    coil = nc * N * (4 if case["half"] else 8)
    held = samples * (4 if case["half"] == 2 else 8)
    # one coil's transform over (y, z) or y: 5 n log2 n; the coil product and sum
    fft = nc * 5.0 * N * math.log2(ny * nz if case["fft_z"] else ny)
    update = {"bytes": 16 * N + coil + held, "flops": 2 * fft + 14.0 * nc * N}
    readout = {"bytes": 16 * samples, "flops": 5.0 * samples * math.log2(nx)}
    svt = {"bytes": 24 * N, "flops": 4.0 * nz * N + 8.0 * nz * N}
    if case["kind"] == "dc":
        return update
    if case["kind"] == "encode":
        # two calls, each reading the maps: E x (image in, samples out) and E^H d (the reverse)
        return {"bytes": 2 * (8 * N + coil + 8 * samples), "flops": 2 * (fft + readout["flops"] + 7.0 * nc * N)}
    if case["kind"] == "svt":
        # two calls, each reading X and S
        return {"bytes": 40 * N, "flops": svt["flops"]}
    # each input once (maps, samples, the kx transform's both sides) and the image; the iterations'
    # own arrays need not leave the chip
    k = case["iters"]
    return {"bytes": coil + readout["bytes"] + 8 * N,
            "flops": k * (update["flops"] + svt["flops"] + 40.0 * N) + readout["flops"] + fft}


# ---- the same in 64 bits --------------------------------------------------------------------

def _haar(x):
    """Orthonormal 2D Haar pyramid (3 levels) of every 8 x 8 tile: [z][tx][ty][8][8]."""
    nz, nx, ny = x.shape
    b = x.reshape(nz, nx // 8, 8, ny // 8, 8).permute(0, 1, 3, 2, 4).contiguous()
    for h in (8, 4, 2):
        a = b[..., :h, :h].clone()
        lo, hi = (a[..., :, 0::2] + a[..., :, 1::2]) / math.sqrt(2), (a[..., :, 0::2] - a[..., :, 1::2]) / math.sqrt(2)
        a = torch.cat([lo, hi], -1)
        lo, hi = (a[..., 0::2, :] + a[..., 1::2, :]) / math.sqrt(2), (a[..., 0::2, :] - a[..., 1::2, :]) / math.sqrt(2)
        b[..., :h, :h] = torch.cat([lo, hi], -2)
    return b


def _unhaar(b):
    b = b.clone()
    for h in (2, 4, 8):
        a = b[..., :h, :h].clone()
        lo, hi = a[..., : h // 2, :], a[..., h // 2:, :]
        a = torch.stack([(lo + hi), (lo - hi)], -2).reshape(*b.shape[:-2], h, h) / math.sqrt(2)
        lo, hi = a[..., :, : h // 2], a[..., :, h // 2:]
        b[..., :h, :h] = torch.stack([(lo + hi), (lo - hi)], -1).reshape(*b.shape[:-2], h, h) / math.sqrt(2)
    nz, tx, ty = b.shape[:3]
    return b.permute(0, 1, 3, 2, 4).reshape(nz, tx * 8, ty * 8).contiguous()


def _half(a):
    return torch.view_as_complex(torch.view_as_real(a.to(torch.complex64)).half().double())


def _adjoint(d, coils, mask, case):
    kz, ky = _lines(mask)
    x = torch.zeros(coils.shape[1:], dtype=torch.complex128, device="cuda")
    for c in range(coils.shape[0]):
        k = torch.zeros(coils.shape[1:], dtype=torch.complex128, device="cuda")
        k[kz, :, ky] = d[c]
        x += coils[c].conj() * torch.fft.ifftn(k, dim=_axes(case), norm="ortho")
    return x


def _exact_frame(case, seed):
    coils, mask, _, d = _problem(case, seed)
    coils, d = coils.to(torch.complex128), d.to(torch.complex128)
    nz = case["nz"]
    X = _adjoint(d, coils, mask, case)
    S, L = torch.zeros_like(X), X.clone()
    svals = lambda M: np.linalg.eigh((M.conj() @ M.T).cpu().numpy())  # noqa: E731
    lamL = 0.01 * math.sqrt(max(svals(X.reshape(nz, -1))[0].max(), 0.0))
    lamS = 0.005 * _haar(X).abs().max()
    keep, sigma = _prior(case, seed) if case["prior"] else (None, None)
    for _ in range(case["iters"]):
        M = (X - S).reshape(nz, -1)
        lam, V = svals(M)
        lam, V = lam[::-1], V[:, ::-1]
        s = np.sqrt(np.maximum(lam, 0.0))
        s2 = np.maximum(s - lamL, 0.0)
        if sigma is not None:
            s2 = s2 - 0.5 * (s2 - sigma)
        s2 = np.where(s <= 1e-3 * s[0], 0.0, s2)
        # M here is [column][voxel]; its Gram conj(M) M^T = G, L = M^T W
        W = (V * (s2 / np.maximum(s, 1e-300))) @ V.conj().T
        c = _haar(X - L)
        a = c.abs()
        c2 = c * torch.where(a > lamS, (a - lamS) / a.clamp_min(1e-300), torch.zeros_like(a))
        c2 = torch.where(keep, c, c2) if keep is not None else c2
        L = (torch.from_numpy(np.ascontiguousarray(W.T)).cuda() @ M).reshape(X.shape)
        S = _unhaar(c2)
        Z = L + S
        X = Z - _adjoint(_encode(Z, coils, mask, case) - d, coils, mask, case)
    return L + S


def exact(case, seed):
    if case["kind"] == "batch":
        return [_exact_frame(c, seed + 100 * i) for i, c in enumerate(members(case))]
    if case["kind"] == "frame":
        return _exact_frame(case, seed)
    if case["kind"] == "svt":
        X, S, W = (t.to(torch.complex128) for t in _svt_inputs(case, seed))
        M = (X - S).reshape(case["nz"], -1)
        return {"G": M.conj() @ M.T, "L": (W.T @ M).reshape(X.shape)}
    coils, mask, x, d = _problem(case, seed)
    c64, d64 = coils.to(torch.complex128), d.to(torch.complex128)
    if case["kind"] == "encode":
        return {"k": _encode(x.to(torch.complex128), c64, mask, case), "image": _adjoint(d64, c64, mask, case)}
    if case["half"] >= 1:
        c64 = _half(coils)
    if case["half"] >= 2:   # the samples are held, rounded, in the space (x, line)
        d64 = torch.fft.fft(_half(torch.fft.ifft(d64, norm="ortho")), norm="ortho")
    Z = (x + _gaussian(x.shape, 0.05, seed + 8)).contiguous().to(torch.complex128)
    R = _encode(Z, c64, mask, case) - d64
    return {"X": Z - _adjoint(R, c64, mask, case), "resid": float(R.abs().square().sum())}
