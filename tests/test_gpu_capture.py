"""Operator calls captured by the user in a CUDA graph and replayed after lps_set_mask and lps_set_data: the
tables of a mask keep their places, so a replay works on the lines that are in force, not on those of the
capture. Fewer and more lines than at the capture (within the capacity of the first mask), planes with and
without a factored-row form, whole and binary16 samples."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from tests.gpu_cases import c64, make_case

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nz,nx,ny,nc,kw", [
    (8, 32, 32, 1, {}), (16, 16, 128, 3, {}), (15, 16, 104, 5, {}), (15, 16, 104, 2, {"data_format": 1}),
    (32, 16, 192, 2, {}), (3, 232, 16, 2, {}),
    (8, 16, 32, 2, {"layout": 1, "frame_slices": 4}),      # 3D frames: lines in the user's order
])
def test_replay_follows_the_mask(nz, nx, ny, nc, kw):
    from paper_1411_6206_gb300 import lps as L
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()   # noqa: E731
    rng = np.random.default_rng(nz + ny)
    cplx = lambda *s: dev(c64(rng.standard_normal(s) + 1j * rng.standard_normal(s)))   # noqa: E731
    masks = [(rng.random((nz, ny)) < f).astype(np.uint8) for f in (0.9, 0.3, 0.08, 0.5)]
    for m in masks:
        m[:, 1] = 1
    coils = dev(make_case(nz, nx, ny, nc, seed=3)["coils"])
    Z, samples = cplx(nz, nx, ny), cplx(nc, int(masks[0].sum()), nx)
    st = torch.cuda.Stream()
    with torch.cuda.stream(st):
        pl = L.Plan(nx, ny, nz, nc, stream=st, **kw)
        pl.set_coils(coils)
        k, A, X = torch.empty_like(samples), torch.empty_like(Z), torch.empty_like(Z)

        def calls(m):
            """E, E^H and step (4) of the plan's mask; the buffers hold as many lines as the first one has."""
            L._check(L.load().lps_forward(pl.handle, L.ptr(Z), L.ptr(k)), "forward")
            L._check(L.load().lps_adjoint(pl.handle, L.ptr(samples), L.ptr(A)), "adjoint")
            L._check(L.load().lps_data_consistency(pl.handle, L.ptr(Z), L.ptr(X), None), "data_consistency")

        def install(mask):
            m = pl.set_mask(mask)
            pl.set_data(samples)
            return m

        install(masks[0])
        m = install(masks[1])
        st.synchronize()
        calls(m)
        st.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=st, capture_error_mode="relaxed"):
            calls(m)
        for mask in masks[1:] + masks[:1]:
            m = install(mask)
            got, want = [], []
            for out, run in ((want, lambda: calls(m)), (got, graph.replay)):
                for t in (k, A, X):
                    t.fill_(7.0)
                run()
                st.synchronize()
                out.extend(t.cpu() for t in (k, A, X))
            assert all(torch.equal(a, b) for a, b in zip(got, want)), int(m)
        del graph
        pl.close()
