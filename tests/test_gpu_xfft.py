"""Readout transform in two register passes (csrc/xfft_rows.cuh): E and E^H against the oracle over its row
lengths (smallest, largest, odd and prime factors, a length outside its table), line counts that are
no multiple of a CTA's 16, one and several coils, lines in task order and in the user's."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import lps_oracle as O
from tests.gpu_cases import c64, make_case, rel, up

pytestmark = pytest.mark.gpu

OP_TOL = 1e-5          # the operators' bound (float32 transforms give about 1e-7 log2 n)


@pytest.mark.parametrize("nx", [8, 16, 24, 48, 56, 96, 104, 128, 152, 160, 176, 184, 200, 208, 216, 224, 232, 240, 256])
@pytest.mark.parametrize("nz,ny,nc,frac", [(3, 16, 2, 0.35), (8, 32, 1, 0.2), (1, 8, 3, 0.125)])
def test_both_directions(nx, nz, ny, nc, frac):
    from paper_1411_6206_gb300 import lps as L
    case = make_case(nz, nx, ny, nc, seed=nx + nz, frac=frac, centre=1)
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()   # noqa: E731
    pl = L.Plan(nx, ny, nz, nc)
    pl.set_coils(dev(case["coils"]))
    m = pl.set_mask(dev(case["mask"]))
    rng = np.random.default_rng(nx)
    Z = c64(rng.standard_normal((nz, nx, ny)) + 1j * rng.standard_normal((nz, nx, ny)))
    coils = up(case["coils"])
    k = torch.empty((nc, m, nx), dtype=torch.complex64, device="cuda")
    L.forward(pl.handle, dev(Z), k)
    assert rel(k.cpu().numpy(), O.E(up(Z), coils, case["mask"])) < OP_TOL
    X = torch.empty((nz, nx, ny), dtype=torch.complex64, device="cuda")
    L.adjoint(pl.handle, dev(case["d"]), X)
    assert rel(X.cpu().numpy(), O.EH(up(case["d"]), coils, case["mask"])) < OP_TOL
    pl.close()
