"""An operator call that directly follows lps_set_coils with LPS_COILS_FP16: the kernel that rounds the
maps has not been waited for by the host, and the call has the bits of one made after a synchronisation."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from tests.gpu_cases import c64, make_case

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nz,nx,ny,nc", [(16, 128, 128, 8), (16, 16, 128, 3), (8, 32, 32, 1), (8, 64, 32, 6), (15, 16, 104, 5)])
def test_call_after_set_coils(nz, nx, ny, nc):
    from paper_1411_6206_gb300 import lps as L
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()   # noqa: E731
    case = make_case(nz, nx, ny, nc, seed=nx + ny)
    rng = np.random.default_rng(8)
    cplx = lambda *s: dev(c64(rng.standard_normal(s) + 1j * rng.standard_normal(s)))   # noqa: E731
    Z, d = cplx(nz, nx, ny), dev(case["d"])
    maps = [dev(case["coils"]), cplx(nc, nz, nx, ny)]
    pl = L.Plan(nx, ny, nz, nc, coil_format=L.COILS_FP16)
    pl.set_coils(maps[1])
    m = pl.set_mask(case["mask"])
    pl.set_data(d)
    out = {}
    for late in (True, False):
        for rep in range(4):
            for i in (0, 1):
                X, k, A = torch.empty_like(Z), torch.empty((nc, m, nx), dtype=Z.dtype, device="cuda"), torch.empty_like(Z)
                for call in (lambda: L.data_consistency(pl.handle, Z, X), lambda: L.forward(pl.handle, Z, k),
                             lambda: L.adjoint(pl.handle, d, A)):
                    pl.set_coils(maps[1 - i])
                    torch.cuda.synchronize()
                    pl.set_coils(maps[i])
                    if late:
                        torch.cuda.synchronize()
                    call()
                got = [t.cpu() for t in (X, k, A)]
                want = out.setdefault(i, got)
                assert all(torch.equal(a, b) for a, b in zip(got, want))
    assert not torch.equal(out[0][0], out[1][0])
    pl.close()
