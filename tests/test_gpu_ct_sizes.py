"""The time/frequency transforms at every count of points class (register blocks of
4 to 32 points), odd and even lengths and unaligned slices, and the chi0 chain's
fused column pass at the same counts."""
import numpy as np
import pytest

from paper_1607_02859_gb300 import gw, inputs

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    c = gw.Context(0)
    yield c
    c.close()


@pytest.mark.parametrize("prec", ["fp64", "fp32", "f16x3"])
@pytest.mark.parametrize("n", [1, 2, 3, 4, 5, 8, 9, 12, 13, 16, 17, 20, 21, 24, 25, 31, 32])
def test_transform_of_n_points(ctx, n, prec):
    rng = np.random.default_rng(n)
    dt = gw.cdtype(prec)
    M = rng.uniform(-100, 100, (n, n))
    for elems in (1, 2, 3, 127, 1000, 4097):
        x = torch.from_numpy(rng.standard_normal((n, elems)) + 1j * rng.standard_normal((n, elems))).to("cuda", dtype=dt)
        ref = M @ x.cpu().numpy().astype(np.complex128)
        for kind, f in ((gw.CT, 1), (gw.ST, 1j), (gw.IST, -1j)):
            out = torch.full_like(x, float("nan"))
            gw.tau_to_omega(ctx, kind, M, x, out, prec)
            # n sums of products: u n in the working precision, weights carried as pairs
            tol = (1e-15 if prec == "fp64" else 1.2e-7) * max(4.0, np.sqrt(n) * 2) * np.linalg.norm(M) * np.linalg.norm(x.cpu())
            assert np.linalg.norm(out.cpu().numpy() - f * ref) <= tol
        if elems > 3:                        # slices that start 8 bytes past a 16-byte boundary
            xo = torch.empty(n * elems + 1, dtype=dt, device="cuda")[1:].reshape(n, elems).copy_(x)
            oo = torch.empty(n * elems + 1, dtype=dt, device="cuda")[1:].reshape(n, elems)
            gw.tau_to_omega(ctx, gw.CT, M, xo, oo, prec)
            gw.tau_to_omega(ctx, gw.CT, M, x, out, prec)
            assert torch.equal(oo, out)


@pytest.mark.parametrize("n_grid,n_chi", [((6, 6, 6), 101), ((12, 12, 12), 260)])
@pytest.mark.parametrize("n", [1, 2, 3, 5, 9, 13, 17, 22, 32])
def test_chi0_with_n_times(ctx, n, n_grid, n_chi):
    p = inputs.tiny(seed=13, n=n_grid, n_tau=n, n_chi=n_chi)
    grid = gw.make_grid(p.n, p.lattice)
    idx = gw.g_set(grid, n_chi)[1]
    C = np.random.default_rng(n).uniform(-1, 1, (n, n))
    got = {}
    for prec in ("fp64", "fp32", "f16x3"):
        psi = torch.from_numpy(p.psi).to("cuda", dtype=gw.cdtype(prec))
        out = torch.full((n, n_chi, n_chi), float("nan"), dtype=gw.cdtype(prec), device="cuda")
        gw.chi0_omega(ctx, grid, psi, p.eps, p.n_occ, p.mu, p.tau, C, idx, prec, out)
        got[prec] = out.cpu().numpy()
    ref = got["fp64"]
    assert np.isfinite(ref).all()
    assert np.linalg.norm(got["fp32"] - ref) < 1e-6 * np.linalg.norm(ref)
    assert np.linalg.norm(got["f16x3"] - ref) < 5e-6 * np.linalg.norm(ref)
