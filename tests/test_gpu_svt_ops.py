"""Stand-alone Gram and reprojection (csrc/k_svt.cu, csrc/k_tc.cu) against the oracle's plain definitions:
column counts at the edges of the tiles, images whose voxels do not fill the last tile, no S, images
that start on an odd complex value, and 3D frames (columns of several slices)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import lps_oracle as O
from tests.gpu_cases import c64, rel, up

pytestmark = pytest.mark.gpu

# float32: sums of at most 256 terms a thread, then of the partials (measured 2e-7 to 7e-7). Split
# operands: 3 u^2 of the split and the float32 sums, relative to the trace / the factors' norms, twice over.
TOL = {"fp32": 2e-6, "tf32": 4e-6, "bf16": 5e-5}


@pytest.fixture(scope="module")
def L():
    from paper_1411_6206_gb300 import lps
    if not torch.cuda.is_available():
        pytest.fail("CUDA device required for -m gpu tests")
    lps.load()
    return lps


def odd(a):
    """The array on the device, 8 bytes past a 16-byte boundary."""
    b = torch.empty(a.size + 1, dtype=torch.complex64, device="cuda")
    v = b[1:].view(a.shape)
    v.copy_(torch.from_numpy(a))
    assert v.data_ptr() % 16 == 8 and v.is_contiguous()
    return v


@pytest.mark.parametrize("mode", ["fp32", "tf32", "bf16"])
@pytest.mark.parametrize("nz,nx,ny,with_s,shifted,cs", [
    (1, 8, 8, True, False, 1), (3, 8, 24, False, False, 1), (4, 16, 40, True, True, 1), (5, 24, 40, True, False, 1),
    (8, 32, 32, True, False, 1), (9, 8, 72, True, True, 1), (16, 40, 48, False, True, 1), (17, 24, 104, True, False, 1),
    (25, 16, 136, True, False, 1), (31, 8, 56, True, True, 1), (32, 72, 64, True, False, 1), (24, 16, 16, True, False, 4)])
def test_gram_and_reprojection(L, mode, nz, nx, ny, with_s, shifted, cs):
    kw = {}
    if cs > 1:
        if mode != "fp32":
            pytest.skip("3D frames run the float32 path")
        kw = dict(layout=L.LAYOUT_FRAMES, frame_slices=cs)
    prec = {"fp32": L.FP32, "tf32": L.TF32_REFINE, "bf16": L.BF16_REFINE}[mode]
    pl = L.Plan(nx, ny, nz, 1, precision=prec, max_iters=1, **kw)
    rng = np.random.default_rng(nz * 100 + ny)
    X = c64(rng.standard_normal((nz, nx, ny)) + 1j * rng.standard_normal((nz, nx, ny)))
    S = c64(0.3 * (rng.standard_normal((nz, nx, ny)) + 1j * rng.standard_normal((nz, nx, ny)))) if with_s else None
    n = nz // cs
    W = c64(rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n)))
    put = odd if shifted else (lambda a: torch.from_numpy(a).cuda())
    dX, dS, dW = put(X), (put(S) if with_s else None), torch.from_numpy(W).cuda()
    G = torch.empty((n, n), dtype=torch.complex64, device="cuda")
    Lo = torch.empty((nz, nx, ny), dtype=torch.complex64, device="cuda")
    L.casorati_gram(pl.handle, dX, dS, G)
    L.lowrank_reproject(pl.handle, dX, dS, dW, Lo)
    ref = O.casorati_gram(up(X), up(S) if with_s else None, cs)
    g = G.cpu().numpy()
    assert np.array_equal(g, g.conj().T)
    assert np.linalg.norm(g - ref) < TOL[mode] * np.trace(ref).real
    assert rel(Lo.cpu().numpy(), O.reproject(up(X), up(S) if with_s else None, W, cs)) < TOL[mode] * 4
    pl.close()
