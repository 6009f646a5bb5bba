"""Readout transform of planes without a factored-row form (3D frames, and rows of 232 points): the lines are
in the user's order and no table of raster numbers is read. E and E^H against the oracle over its row
lengths (in the register table and outside it) and line counts that are no multiple of a CTA's 16."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import lps_oracle as O
from tests.gpu_cases import c64, make_case, rel, up

pytestmark = pytest.mark.gpu

OP_TOL = 1e-5          # the operators' bound (float32 transforms give about 1e-7 log2 n)


@pytest.mark.parametrize("nx", [8, 56, 104, 160, 184, 200, 232, 256])
@pytest.mark.parametrize("nz,ny,nc,fs,frac", [(4, 16, 2, 2, 0.35), (8, 32, 1, 4, 0.2), (2, 232, 2, 1, 0.1)])
def test_both_directions(nx, nz, ny, nc, fs, frac):
    from paper_1411_6206_gb300 import lps as L
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()   # noqa: E731
    rng = np.random.default_rng(nx + ny)
    coils = make_case(nz, nx, ny, nc, seed=nx + nz, centre=1)["coils"]
    mask = (rng.random((nz, ny)) < frac).astype(np.uint8)
    mask[:, 0] = 1
    kw = dict(layout=L.LAYOUT_FRAMES, frame_slices=fs) if fs > 1 else {}
    pl = L.Plan(nx, ny, nz, nc, **kw)
    pl.set_coils(dev(coils))
    m = pl.set_mask(dev(mask))
    zb = fs if fs > 1 else nz
    Z, d = (c64(rng.standard_normal(s) + 1j * rng.standard_normal(s)) for s in ((nz, nx, ny), (nc, m, nx)))
    k = torch.empty((nc, m, nx), dtype=torch.complex64, device="cuda")
    L.forward(pl.handle, dev(Z), k)
    assert rel(k.cpu().numpy(), O.E(up(Z), up(coils), mask, 1, zb)) < OP_TOL
    X = torch.empty((nz, nx, ny), dtype=torch.complex64, device="cuda")
    L.adjoint(pl.handle, dev(d), X)
    assert rel(X.cpu().numpy(), O.EH(up(d), up(coils), mask, 1, zb)) < OP_TOL
    pl.close()
