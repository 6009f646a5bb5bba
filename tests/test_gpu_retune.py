"""Launch shapes changed between two runs of iterations (lps_apply_tune, lps_autotune): the variants leave
different numbers of Gram and statistic partials, and the run goes on from the same state whichever
was in force before. Against an uninterrupted run of the default shapes."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import lps_oracle as O
from tests.gpu_cases import make_case

pytestmark = pytest.mark.gpu

E2E_TOL = 1e-3        # the bound of a run of iterations (two float32 evaluations of one recursion)
STAT_TOL = 1e-3       # a record's float32 sums, of iterates within that bound


def run(L, case, nz, nx, ny, nc, steps, **kw):
    """Iterations in runs of steps[i][0], steps[i][1] (dc_variant, lrs_tiles) or "auto" installed before each."""
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()   # noqa: E731
    pl = L.Plan(nx, ny, nz, nc, max_iters=16, **kw)
    pl.set_coils(dev(case["coils"]))
    pl.set_mask(case["mask"])
    pl.set_data(dev(case["d"]))
    for n, tune in steps:
        if tune == "auto":
            pl.autotune()
        elif tune:
            rad = lambda v: {8: (8,), 16: (16,), 32: (8, 4), 128: (16, 8)}[v] if tune[0] in (1, 2) else ()   # noqa: E731
            L.apply_tune(pl.handle, tune[0], rad(ny), rad(nz), lrs_tiles=tune[1])
        st = pl.iterate(n)
    out = [torch.empty((nz, nx, ny), dtype=torch.complex64, device="cuda") for _ in range(3)]
    L.get_state(pl.handle, *out)
    hist = pl.history()
    pl.close()
    return [t.cpu().numpy() for t in out], hist, st


@pytest.mark.parametrize("nz,nx,ny,nc,steps", [
    (16, 32, 128, 3, [(3, (3, 1)), (3, (0, 1)), (3, (3, 2))]),          # nx / 4, nx, nx / 4 partials
    (16, 32, 128, 6, [(3, (0, 2)), (3, (4, 1)), (3, (2, 1))]),
    (16, 128, 128, 2, [(3, (2, 2)), (3, (3, 1)), (3, (0, 2))]),         # nx partials by a cluster of the eigen kernel
    (8, 32, 32, 2, [(3, (0, 4)), (3, (2, 1)), (3, (0, 3))]),
    (16, 32, 128, 3, [(3, (0, 1)), (3, "auto"), (3, None)]),
    (8, 32, 32, 1, [(3, (2, 4)), (3, "auto"), (3, None)]),
])
def test_retuned_run_goes_on_from_its_state(nz, nx, ny, nc, steps):
    from paper_1411_6206_gb300 import lps as L
    L.load()
    case = make_case(nz, nx, ny, nc, seed=31 + nc)
    ref, href, sref = run(L, case, nz, nx, ny, nc, [(n, None) for n, _ in steps])
    L.autotune_clear_cache()
    got, hist, st = run(L, case, nz, nx, ny, nc, steps)
    for a, b in zip(got, ref):
        assert O.nrmse(a, b.astype(np.complex128)) < E2E_TOL
    assert len(hist) == len(href) == 9
    for h, r in zip(hist, href):
        for key in ("resid_norm2", "nuclear", "l1_off_support"):
            assert abs(h[key] - r[key]) <= STAT_TOL * abs(r[key]), key
        assert h["rank"] == r["rank"]
    assert abs(st.support_count - sref.support_count) <= 0.005 * sref.support_count


@pytest.mark.parametrize("tune", [(0, 1), "auto"])
def test_statistics_after_a_retune(tune):
    """A run of no iterations after the change reports the state's statistics as they were."""
    from paper_1411_6206_gb300 import lps as L
    L.load()
    nz, nx, ny, nc = 16, 32, 128, 3
    case = make_case(nz, nx, ny, nc, seed=5)
    L.autotune_clear_cache()
    _, href, sref = run(L, case, nz, nx, ny, nc, [(4, (3, 2))])
    _, hist, st = run(L, case, nz, nx, ny, nc, [(4, (3, 2)), (0, tune)])
    assert st.support_count == sref.support_count and st.iters == sref.iters == 4
    for h, r in zip(hist, href):
        assert abs(h["l1_off_support"] - r["l1_off_support"]) <= 1e-5 * r["l1_off_support"]
        assert h["resid_norm2"] == r["resid_norm2"]
