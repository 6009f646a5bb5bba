"""Factored-row data-consistency kernel (csrc/k_dc_rows.cuh): step (4), E and E^H against the oracle
at the edges of its range (smallest and largest rows and slice counts, odd and prime factors, one
coil, as many CTAs a plane as coils, samples staged and not), its agreement with the runtime-sized
kernel, and the order of the iteration form's reads (a plan's first frame equals its later ones)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import lps_oracle as O
from tests.gpu_cases import c64, make_case, rel, up

pytestmark = pytest.mark.gpu

OP_TOL = 1e-5          # the operators' bound (float32 transforms give about 1e-7 log2 n)


@pytest.fixture(scope="module")
def L():
    from paper_1411_6206_gb300 import lps
    if not torch.cuda.is_available():
        pytest.fail("CUDA device required for -m gpu tests")
    lps.load()
    return lps


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def plan_for(L, case, nz, nx, ny, nc, **kw):
    pl = L.Plan(nx, ny, nz, nc, **kw)
    pl.set_coils(dev(case["coils"]))
    assert pl.set_mask(dev(case["mask"])) == case["nlines"]
    pl.set_data(dev(case["d"]))
    return pl


SHAPES = [
    # nz, nx, ny, ncoil, fft_z, dense mask
    (1, 8, 8, 1, 1, True), (3, 8, 24, 2, 1, False), (32, 8, 16, 2, 1, False), (5, 16, 40, 7, 1, False),
    (7, 8, 56, 2, 0, False), (9, 8, 72, 1, 1, True), (15, 24, 104, 6, 1, False), (17, 8, 120, 2, 1, False),
    (31, 8, 136, 3, 1, True), (13, 16, 152, 5, 1, False), (11, 8, 168, 2, 0, False), (23, 8, 184, 9, 1, False),
    (19, 8, 200, 2, 1, True), (4, 8, 208, 3, 1, False), (6, 8, 216, 1, 1, False), (14, 16, 256, 4, 1, False),
    (8, 40, 32, 1, 1, False), (10, 8, 64, 16, 1, False), (32, 8, 192, 3, 1, True), (32, 16, 192, 4, 0, False),
    (16, 8, 128, 2, 1, True), (28, 8, 144, 5, 1, True),
]


@pytest.mark.parametrize("nz,nx,ny,nc,fz,full", SHAPES)
def test_operators(L, nz, nx, ny, nc, fz, full):
    case = make_case(nz, nx, ny, nc, seed=nz * 7 + ny, fft_z=fz, full=full)
    pl = plan_for(L, case, nz, nx, ny, nc, fft_z=fz)
    if (nz, ny) == (16, 128):
        L.apply_tune(pl.handle, 0, (), (), lrs_tiles=1)      # its default is the register-transform kernel
    rng = np.random.default_rng(5)
    Z = c64(rng.standard_normal((nz, nx, ny)) + 1j * rng.standard_normal((nz, nx, ny)))
    X = torch.empty((nz, nx, ny), dtype=torch.complex64, device="cuda")
    r2 = L.data_consistency(pl.handle, dev(Z), X)
    coils, d = up(case["coils"]), up(case["d"])
    R = O.E(up(Z), coils, case["mask"], fz) - d
    assert rel(X.cpu().numpy(), up(Z) - O.EH(R, coils, case["mask"], fz)) < OP_TOL
    assert abs(r2 - np.vdot(R, R).real) < 1e-5 * np.vdot(R, R).real
    inplace = dev(Z)
    L.data_consistency(pl.handle, inplace, inplace)
    assert torch.equal(inplace, X)
    k = torch.empty((nc, case["nlines"], nx), dtype=torch.complex64, device="cuda")
    L.forward(pl.handle, dev(Z), k)
    assert rel(k.cpu().numpy(), R + d) < OP_TOL
    L.adjoint(pl.handle, dev(case["d"]), X)
    assert rel(X.cpu().numpy(), O.EH(d, coils, case["mask"], fz)) < OP_TOL
    pl.close()


@pytest.mark.parametrize("nz,nx,ny,nc,fmt", [(15, 16, 104, 3, 0), (15, 16, 104, 3, 1), (20, 8, 96, 5, 0), (20, 8, 96, 5, 1)])
def test_half_maps_and_samples_read_the_rounded_values(L, nz, nx, ny, nc, fmt):
    """Binary16 maps that are half-representable give the bits of the float32 format; binary16 samples
    the update of the rounded samples."""
    case = make_case(nz, nx, ny, nc, seed=3 + ny)
    r16 = lambda a: c64(a.real.astype(np.float16).astype(np.float32) + 1j * a.imag.astype(np.float16).astype(np.float32))  # noqa: E731
    case["coils"] = r16(case["coils"])
    rng = np.random.default_rng(4)
    Z = dev(c64(rng.standard_normal((nz, nx, ny)) + 1j * rng.standard_normal((nz, nx, ny))))
    out = []
    for kw in ({}, dict(coil_format=L.COILS_FP16) if fmt == 0 else dict(data_format=L.DATA_FP16)):
        pl = plan_for(L, case, nz, nx, ny, nc, **kw)
        X = torch.empty_like(Z)
        L.data_consistency(pl.handle, Z, X)
        out.append(X.cpu().numpy())
        pl.close()
    if fmt == 0:
        assert np.array_equal(out[0], out[1])
    else:
        h = np.fft.ifft(up(case["d"]), axis=-1, norm="ortho")
        d = np.fft.fft(up(r16(h)), axis=-1, norm="ortho")
        coils = up(case["coils"])
        z = up(Z.cpu().numpy())
        ref = z - O.EH(O.E(z, coils, case["mask"]) - d, coils, case["mask"])
        assert rel(out[1], ref) < 2e-5        # a sample within rounding of a binary16 tie may go the other way


def radix_plan(n):
    out = []
    for r in (16, 8, 4, 2, 3, 5, 7):
        while n % r == 0:
            out.append(r)
            n //= r
    return tuple(out)


@pytest.mark.parametrize("half", ["", "coil_format", "data_format"])
@pytest.mark.parametrize("nz,nx,ny,nc,fz", [(2, 8, 16, 2, 1), (5, 16, 40, 7, 0), (9, 8, 72, 1, 1), (15, 24, 120, 6, 1),
                                            (14, 16, 160, 5, 0), (20, 8, 96, 4, 1), (21, 8, 168, 3, 1), (24, 8, 240, 2, 1),
                                            (32, 16, 192, 4, 1)])
def test_equals_the_runtime_sized_kernel(L, nz, nx, ny, nc, fz, half):
    """Step (4), E and E^H of the default path against the runtime-sized kernel on the same plan (so on
    the same rounded maps or samples): two float32 evaluations of one sum, within the operators' bound."""
    case = make_case(nz, nx, ny, nc, seed=ny + nz, fft_z=fz, frac=0.4)
    pl = plan_for(L, case, nz, nx, ny, nc, fft_z=fz, **({half: 1} if half else {}))
    rng = np.random.default_rng(6)
    Z = dev(c64(rng.standard_normal((nz, nx, ny)) + 1j * rng.standard_normal((nz, nx, ny))))
    outs = []
    for generic in (False, True):
        if generic:
            L.apply_tune(pl.handle, 2, radix_plan(ny), radix_plan(nz), lrs_tiles=1)
        X, A = torch.empty_like(Z), torch.empty_like(Z)
        k = torch.empty((nc, case["nlines"], nx), dtype=torch.complex64, device="cuda")
        r2 = L.data_consistency(pl.handle, Z, X)
        L.forward(pl.handle, Z, k)
        L.adjoint(pl.handle, dev(case["d"]), A)
        outs.append((X.cpu().numpy(), k.cpu().numpy(), A.cpu().numpy(), r2))
    for got, want in zip(outs[0][:3], outs[1][:3]):
        assert rel(got, up(want)) < OP_TOL
    assert abs(outs[0][3] - outs[1][3]) < 1e-5 * outs[1][3]
    pl.close()


@pytest.mark.parametrize("nz,nx,ny,nc", [(5, 64, 48, 3), (7, 72, 40, 6), (10, 64, 80, 4), (15, 64, 104, 5), (32, 16, 192, 2),
                                         (16, 128, 128, 8)])
def test_first_frame_equals_later_frames(L, nz, nx, ny, nc):
    """The iteration form reads S_k only once the sparse step beside the eigen kernel has written it: a
    plan's first frame, whose S buffers hold nothing yet, has the bits of its second."""
    case = make_case(nz, nx, ny, nc, seed=21, frac=0.3)
    pl = plan_for(L, case, nz, nx, ny, nc, max_iters=5)
    recs = []
    for _ in range(3):
        pl.set_data(dev(case["d"]))
        r = torch.empty((nz, nx, ny), dtype=torch.complex64, device="cuda")
        pl.reconstruct_frame(recon=r)
        recs.append(r.cpu().numpy())
    assert np.array_equal(recs[0], recs[1]) and np.array_equal(recs[0], recs[2])
    pl.close()
